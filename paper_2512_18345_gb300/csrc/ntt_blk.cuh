// The block pass of a transform (the last eight stages, on contiguous 256-element
// blocks; ntt.cuh describes the split), with each half-warp on its own.
//
// A block's 256 elements are one half-warp's 16 x 16 register values, so every exchange
// stays inside a warp: no CTA barrier anywhere, and the warps of an SM drift apart, which
// overlaps one's loads with another's butterflies.
//
// What bounds it: at N = 2^16 the pass moves 2 W of data and W x 2 of twiddles per limb, and
// the load/store unit was 79 % busy with half-used sectors (a thread's 16 results and its lo
// twiddles are 64 and 120 contiguous bytes, so 16-byte accesses of a warp were 64 bytes
// apart).  Here
//   * the lo round's 15 twiddles come from a table in thread order (lo_fwd / lo_inv: eight
//     16-byte loads, each 512 contiguous bytes per warp);
//   * results leave, and the inverse's inputs and the combine's operand arrive, as 16-byte
//     accesses in memory order (256 contiguous bytes per half-warp), turned through the
//     half-warp's shared-memory block;
//   * a rotation's input block is one contiguous source block (sigma maps aligned 256-blocks
//     onto 256-blocks): it is staged in memory order and permuted on its way out of shared
//     memory, instead of 4-byte global gathers 64 bytes apart.
// Measured on one GB300 (8 rotations at N = 2^16, L = 24, K = 8, two lanes, traced per
// launch), against the CTA-wide form: ModUp forward 74.7 -> 59.3 us, combine 60.1 -> 50.9 us,
// inverse 20.4 -> 18.7 us, with gather 27.6 -> 27.0 us; the graph step 554 -> 521 us, the
// level-24 dense transform 1335 -> 1277 us.
#pragma once
#include "ntt.cuh"

namespace fhe {

// word of element k of block c: rows of 16, the 16-byte chunks of a row xor-swizzled so that
// scalar accesses along a row and 16-byte accesses down the rows are free of bank conflicts
__device__ __forceinline__ uint32_t nb_blk_addr(int c, int k) {
  const int r = k >> 4;
  return (uint32_t)(c * 272 + r * 16 + ((((k >> 2) & 3) ^ ((r >> 1) & 3)) << 2) + (k & 3));
}

// The lo round's twiddles of thread `tid` of tile `tile`: entry (1 << m) - 1 + j for register
// bit 3 - m and butterfly group j = e >> (bit + 1) (entry 15 is padding).
template <int LOGN>
__device__ __forceinline__ void load_lo_twiddles(const uint4 *lo, int prime, int tile, int tid, uint2 (&tl)[16]) {
  const uint4 *p = lo + ((size_t)prime << (LOGN - 1)) + tile * (kTile / 2) + tid;
#pragma unroll
  for (int v = 0; v < 8; v++) {
    const uint4 w = __ldg(p + v * kNttThreads);
    tl[2 * v] = make_uint2(w.x, w.y);
    tl[2 * v + 1] = make_uint2(w.z, w.w);
  }
}

// Fill that table from the bit-reversed one: one thread per 16-byte entry.
__global__ void k_lo_table(const uint2 *tw, uint4 *lo, int logn, int nprimes) {
  const size_t per = (size_t)1 << (logn - 1), i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= per * nprimes) return;
  const size_t prime = i >> (logn - 1);
  const int w = (int)(i & (per - 1)), tile = w / (kTile / 2), v = (w / kNttThreads) & 7, tid = w % kNttThreads;
  const int blk = tile * 16 + (tid >> 4), tau = tid & 15;
  uint2 o[2];
  for (int h = 0; h < 2; h++) {
    const int entry = 2 * v + h;
    const int m = 31 - __clz(entry + 1), j = entry + 1 - (1 << m);
    o[h] = entry == 15 ? make_uint2(0, 0)
                       : tw[(prime << logn) + ((size_t)1 << (logn - 4 + m)) + ((size_t)blk << (4 + m)) + (tau << m) + j];
  }
  lo[i] = make_uint4(o[0].x, o[0].y, o[1].x, o[1].y);
}

// one radix-16 round (4 butterfly stages on the 16 register values); tw(m, j) is the
// twiddle of register bit 3 - m for butterfly group j
template <bool FWD, class TW>
__device__ __forceinline__ void nb_round(uint32_t (&x)[16], TW tw, uint32_t q) {
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int bit = FWD ? 3 - i : i;
    const int m = 3 - bit;
#pragma unroll
    for (int e = 0; e < 16; e++) {
      if (e & (1 << bit)) continue;
      const int e2 = e | (1 << bit);
      const uint2 w = tw(m, e >> (bit + 1));
      if (FWD) {
        const uint32_t t = red2(shoup_lazy(x[e2], w.x, w.y, q), q);
        const uint32_t u = red2(x[e], q);
        x[e] = u + t;
        x[e2] = u - t + q;
      } else {
        const uint32_t u = red2(x[e], q), v = red2(x[e2], q);
        x[e] = u + v;
        x[e2] = shoup_lazy(u - v + q, w.x, w.y, q);
      }
    }
  }
}

// The hi round of block c with its twiddles in heap order at hw (entry 2^m + j): a stage's are
// consecutive from an even entry, fetched in 16-byte pairs.
template <bool FWD>
__device__ __forceinline__ void nb_round_hi(uint32_t (&x)[16], const uint2 *hw, uint32_t q) {
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int bit = FWD ? 3 - i : i, m = 3 - bit;
    uint2 ws[8];
    if (m == 0) {
      ws[0] = hw[1];
    } else {
#pragma unroll
      for (int k2 = 0; k2 < (1 << m) / 2; k2++) {
        const uint4 w = *reinterpret_cast<const uint4 *>(hw + (1 << m) + 2 * k2);
        ws[2 * k2] = make_uint2(w.x, w.y);
        ws[2 * k2 + 1] = make_uint2(w.z, w.w);
      }
    }
#pragma unroll
    for (int e = 0; e < 16; e++) {
      if (e & (1 << bit)) continue;
      const int e2 = e | (1 << bit);
      const uint2 w = ws[e >> (bit + 1)];
      if (FWD) {
        const uint32_t t = red2(shoup_lazy(x[e2], w.x, w.y, q), q);
        const uint32_t u = red2(x[e], q);
        x[e] = u + t;
        x[e2] = u - t + q;
      } else {
        const uint32_t u = red2(x[e], q), v = red2(x[e2], q);
        x[e] = u + v;
        x[e2] = shoup_lazy(u - v + q, w.x, w.y, q);
      }
    }
  }
}

// ---- the pass in pieces (thread (c, tau) of a 16-block tile; sm: the tile's 16 x 272 words)

// this thread's entry tau of block blk's hi-round twiddles, psi^brv(2^(S0 + m) + (blk << m) + j)
// at 2^m + j (entry 0 unused)
template <int LOGN, bool FWD>
__device__ __forceinline__ uint2 blk_hi_twiddle(const NttTables &tb, int prime, int blk, int tau) {
  if (!tau) return make_uint2(0, 0);
  const int m = 31 - __clz(tau);
  return __ldg((FWD ? tb.tw_fwd : tb.tw_inv) + ((size_t)prime << LOGN) + (((1 << (LOGN - 8)) + blk) << m) + tau - (1 << m));
}
// a thread's i-th 16-byte chunk in memory order: element 64 i + 4 tau of block c
__device__ __forceinline__ uint32_t *blk_lin(uint32_t *sm, int c, int tau, int i) {
  return sm + nb_blk_addr(c, 64 * i + 4 * tau);
}
// forward: x in hi layout (element 16 e + tau) -> lazy results in sm
__device__ __forceinline__ void blk_forward(uint32_t (&x)[16], uint32_t *sm, int c, int tau, const uint2 *hw,
                                            const uint2 (&tl)[16], uint32_t q) {
  nb_round_hi<true>(x, hw, q);
#pragma unroll
  for (int e = 0; e < 16; e++) sm[nb_blk_addr(c, (e << 4) | tau)] = x[e];
  __syncwarp();
#pragma unroll
  for (int m = 0; m < 4; m++) ld4(sm + nb_blk_addr(c, (tau << 4) | (4 * m)), x + 4 * m);
  nb_round<true>(x, [&](int m, int j) { return tl[(1 << m) - 1 + j]; }, q);
#pragma unroll
  for (int m = 0; m < 4; m++) st4(sm + nb_blk_addr(c, (tau << 4) | (4 * m)), x + 4 * m);
  __syncwarp();
}
// write the results in sm to the limb in memory order
template <int EPI, bool DEP>
__device__ __forceinline__ void blk_store(const SegList &sl, const Limb &lb, int blk, uint32_t *sm, int c, int tau,
                                          uint2 scale, uint32_t q) {
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int j = blk * 256 + 64 * i + 4 * tau;
    uint32_t o[4], a[4];
    if (EPI == EPI_COMBINE || EPI == EPI_RESCALE) ld_in4<DEP>(lb.src2 + j, a);
    if (EPI == EPI_SUM) {
      const size_t off = (size_t)(lb.src2 - sl.ks[0].u) + j;
      a[0] = a[1] = a[2] = a[3] = 0;
      for (int k = 0; k < sl.sum_n; k++) {
        uint32_t w[4];
        ld_in4<DEP>(sl.ks[k].u + off, w);
#pragma unroll
        for (int e = 0; e < 4; e++) a[e] = add_mod(a[e], w[e], q);
      }
    }
    ld4(blk_lin(sm, c, tau, i), o);
#pragma unroll
    for (int e = 0; e < 4; e++) {
      o[e] = red2(o[e], q);
      // COMBINE: a = inner product u (with P times the pass-through term folded in)
      if (EPI == EPI_COMBINE || EPI == EPI_RESCALE || EPI == EPI_SUM) o[e] = shoup(a[e] + q - o[e], scale.x, scale.y, q);
    }
    if (EPI == EPI_SUM) {
      uint32_t w[4];
      ld_in4<DEP>(lb.T + j, w);
#pragma unroll
      for (int e = 0; e < 4; e++) o[e] = add_mod(o[e], w[e], q);
    }
    st4(lb.dst + j, o);
  }
}
// the inverse's input: block blk (PRO_GATHER: read through sigma_galois) into lo layout
// (element 16 tau + e); `staged` runs once the loads are on their way
template <int LOGN, int PRO, bool DEP, class F>
__device__ __forceinline__ void blk_load(uint32_t (&x)[16], const Limb &lb, const PrimeC &P, int blk, uint32_t *sm, int c,
                                         int tau, F staged) {
  constexpr int S0 = LOGN - 8;
  constexpr bool GATHER = PRO == PRO_GATHER || PRO == PRO_MUL;
  const uint32_t *src = lb.src;
  const uint32_t galois = lb.galois;
  uint32_t kadd = 0;
  if (GATHER) {
    // index blk 256 + k has brv = brv8(k) 2^S0 + brv(blk); times g plus g >> 1, its low S0
    // bits give the source block and the rest brv8 of the source element: brv8(k) g + kadd
    const uint32_t r = (__brev((uint32_t)blk) >> (32 - S0)) * galois + (galois >> 1);
    kadd = r >> S0;
    src += (__brev(r << (32 - S0)) << 8);
  } else {
    src += blk * 256;
  }
  uint32_t w[16];
#pragma unroll
  for (int i = 0; i < 4; i++) ld_in4<DEP>(src + 64 * i + 4 * tau, w + 4 * i);
  if (PRO == PRO_MUL && lb.src2) {  // (uniform per limb; such a limb has galois 1)
#pragma unroll
    for (int i = 0; i < 4; i++) {
      uint32_t w2[4];
      ld_in4<DEP>(lb.src2 + blk * 256 + 64 * i + 4 * tau, w2);
#pragma unroll
      for (int e = 0; e < 4; e++) w[4 * i + e] = mul_mod(w[4 * i + e], w2[e], P);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; i++) st4(blk_lin(sm, c, tau, i), w + 4 * i);
  staged();
  __syncwarp();
  if (PRO == PRO_GATHER || (PRO == PRO_MUL && galois != 1u)) {
    const uint32_t base = (__brev((uint32_t)tau) >> 28) * galois + kadd;
#pragma unroll
    for (int e = 0; e < 16; e++) {
      const uint32_t be = ((e & 1) << 3) | ((e & 2) << 1) | ((e & 4) >> 1) | ((e & 8) >> 3);  // brv4(e)
      x[e] = sm[nb_blk_addr(c, (int)(__brev(base + be * 16u * galois) >> 24))];
    }
    __syncwarp();  // every lane's reads come before the rows are rewritten
  } else {
#pragma unroll
    for (int m = 0; m < 4; m++) ld4(sm + nb_blk_addr(c, (tau << 4) | (4 * m)), x + 4 * m);
  }
}
// inverse: x in lo layout -> x in hi layout
__device__ __forceinline__ void blk_inverse(uint32_t (&x)[16], uint32_t *sm, int c, int tau, const uint2 *hw,
                                            const uint2 (&tl)[16], uint32_t q) {
  nb_round<false>(x, [&](int m, int j) { return tl[(1 << m) - 1 + j]; }, q);
#pragma unroll
  for (int m = 0; m < 4; m++) st4(sm + nb_blk_addr(c, (tau << 4) | (4 * m)), x + 4 * m);
  __syncwarp();
#pragma unroll
  for (int e = 0; e < 16; e++) x[e] = sm[nb_blk_addr(c, (e << 4) | tau)];
  nb_round_hi<false>(x, hw, q);
}

// Forward: PRO_PLAIN with EPI_PLAIN, EPI_COMBINE, EPI_RESCALE or EPI_SUM; inverse: PRO_PLAIN,
// PRO_GATHER or PRO_MUL with EPI_LAZY.  Residency: 48 registers (16 values, 30 of twiddles), 40
// warps per SM (32 and 48, and loading the lo twiddles after the hi round: within 1 % or slower).
// Four blocks (two warps) per CTA: with no CTA barrier the size only sets how finely the launch
// fills the SMs; against 256 and 128 threads the 64-item mixed plan takes 2444 us instead of 2465
// and 2449, one rotation 99.4 instead of 100.4 and 99.7.
constexpr int kBlkThreads = 64, kBlkBlocks = kBlkThreads / 16;
template <int LOGN, bool FWD, int PRO, int EPI, bool DEP>
__global__ void __launch_bounds__(kBlkThreads, ((DEP && FWD) || PRO == PRO_MUL ? 4 : 5) * (256 / kBlkThreads)) k_ntt_blk(const __grid_constant__ SegList sl, const NttTables tb) {
  constexpr int TILES = (1 << LOGN) / (256 * kBlkBlocks);
  __shared__ __align__(16) uint32_t sm[kBlkBlocks * 272];
  __shared__ __align__(16) uint2 hws[kBlkBlocks * 16];
  const int tid = threadIdx.x, c = tid >> 4, tau = tid & 15;
  const int v = blockIdx.x / TILES, tile = blockIdx.x % TILES;
  const Limb lb = limb_at<EPI == EPI_COMBINE || EPI == EPI_SUM>(sl, v, tb.ninv, LOGN);
  const PrimeC P = tb.pc[lb.prime];
  const uint32_t q = P.q;
  const int blk = tile * kBlkBlocks + c;
  uint2 *hw = hws + c * 16;
  const uint2 h1 = blk_hi_twiddle<LOGN, FWD>(tb, lb.prime, blk, tau);
  uint2 tl[16];
  load_lo_twiddles<LOGN>(FWD ? tb.lo_fwd : tb.lo_inv, lb.prime, blk >> 4, (blk & 15) * 16 + tau, tl);
  uint32_t x[16];
  if (DEP) dep_wait();
  if (FWD) {
    const uint32_t *src = lb.src + blk * 256 + tau;
#pragma unroll
    for (int e = 0; e < 16; e++) x[e] = ld_in<DEP>(src + e * 16);
    hw[tau] = h1;  // (stored after the loads are on their way, so that their latencies overlap)
    __syncwarp();  // the hi-round twiddles
    blk_forward(x, sm, c, tau, hw, tl, q);
    uint2 scale = make_uint2(0, 0);
    if (EPI != EPI_PLAIN) scale = __ldg(lb.scale);
    blk_store<EPI, DEP>(sl, lb, blk, sm, c, tau, scale, q);
  } else {
    blk_load<LOGN, PRO, DEP>(x, lb, P, blk, sm, c, tau, [&] { hw[tau] = h1; });
    blk_inverse(x, sm, c, tau, hw, tl, q);
    uint32_t *dst = lb.dst + blk * 256 + tau;
#pragma unroll
    for (int e = 0; e < 16; e++) dst[e * 16] = x[e];
  }
}

}  // namespace fhe
