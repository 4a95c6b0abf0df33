// The column pass of a transform (the first logN - 8 stages, on strided sub-transforms;
// ntt.cuh describes the split) with warp-private twiddles.
//
// A tile is 16 columns of 2^(logN - 8) rows; thread (c, tau) holds 16 rows of column c, and at
// N = 2^16 the two radix-16 rounds exchange across the CTA's warps through shared memory.
// That exchange is the only CTA barrier: the twiddles a warp needs (15 of the hi round, the
// same for every thread; 15 of the lo round for each of its two tau) are staged by the warp
// for itself, so a warp starts as soon as its own loads land instead of meeting the other
// seven first.  What bounds it: the integer pipes (fmaheavy and ALU near 65 % busy, the rest
// load latency and the exchange).  Measured on one GB300, against staging the twiddles for the
// CTA behind a barrier of its own: the 8-rotation graph step (N = 2^16, L = 24, K = 8)
// 519 -> 507 us, the level-24 dense transform 1275 -> 1254 us.
#pragma once
#include "ntt_blk.cuh"

namespace fhe {

// residency asked of the register allocator: 40 and 32..36 registers; eight CTAs (32 registers)
// on both sides cost 0.5 % of the graph step below
template <bool FWD>
constexpr int ntt_col_ctas() { return FWD ? 6 : 7; }

// Forward: PRO_PLAIN, PRO_REDUCE or PRO_SUM with EPI_LAZY; inverse: PRO_PLAIN with EPI_SCALE.
template <int LOGN, bool FWD, int PRO, int EPI, bool DEP>
__global__ void __launch_bounds__(kNttThreads, ntt_col_ctas<FWD>())
    k_ntt_col(const __grid_constant__ SegList sl, const NttTables tb) {
  using G = NttGeom<LOGN, true>;
  constexpr int R = G::R;  // 8 at N = 2^16 (two rounds), 4 at N = 2^12 (one)
  static_assert(R == 8 || R == 4, "column pass: 8 or 4 stages");
  constexpr int kLo = 18;  // entries between a warp's two lo-round tables (no bank conflict)
  __shared__ uint32_t sm[R == 8 ? G::SMEM : 1];
  __shared__ __align__(16) uint2 tws[8][16 + (R == 8 ? 2 * kLo : 0)];
  const int tid = threadIdx.x, lane = tid & 31;
  const int c = R == 4 ? tid : tid & 15, tau = R == 4 ? 0 : tid >> 4;
  const int v = blockIdx.x / G::TILES, tile = blockIdx.x % G::TILES;
  const Limb lb = limb_at<false>(sl, v, tb.ninv, LOGN);
  const PrimeC P = tb.pc[lb.prime];
  const uint32_t q = P.q;
  const uint2 *tw = (FWD ? tb.tw_fwd : tb.tw_inv) + ((size_t)lb.prime << LOGN);
  uint2 *hw = tws[tid >> 5];
  uint2 h1 = make_uint2(0, 0), h2 = make_uint2(0, 0);
  if (lane < 16) h1 = __ldg(tw + lane);  // hi round: entry 2^m + j is index 2^m + j
  if (R == 8 && (lane & 15)) {           // lo round: entry 2^m + j is index (16 + tau) 2^m + j
    const int h = lane & 15, m = 31 - __clz(h);
    h2 = __ldg(tw + ((16 + tau) << m) + h - (1 << m));
  }
  const uint2 *lw = hw + 16 + (tau & 1) * kLo;
  if (DEP) dep_wait();
  uint32_t x[16];
#pragma unroll
  for (int e = 0; e < 16; e++) x[e] = ld_in<DEP>(lb.src + G::gidx(tile, c, kmap<R>(FWD, e, tau)));
  if (PRO == PRO_SUM) {  // the other items' values (each lazy, in [0, 2q))
    const size_t off = (size_t)(lb.src - sl.ks[0].r);
#pragma unroll
    for (int e = 0; e < 16; e++) x[e] = red2(x[e], q);
    for (int i = 1; i < sl.sum_n; i++) {
      const uint32_t *p = sl.ks[i].r + off;
      uint32_t w[16];
#pragma unroll
      for (int e = 0; e < 16; e++) w[e] = ld_in<DEP>(p + G::gidx(tile, c, kmap<R>(FWD, e, tau)));
#pragma unroll
      for (int e = 0; e < 16; e++) x[e] = add_mod(x[e], red2(w[e], q), q);
    }
  }
  // (stored after the loads are on their way, so that their latencies overlap)
  if (lane < 16) hw[lane] = h1;
  if (R == 8) hw[16 + (lane >> 4) * kLo + (lane & 15)] = h2;
  if (PRO == PRO_REDUCE)
#pragma unroll
    for (int e = 0; e < 16; e++) x[e] = reduce_u64(x[e], P);  // a value of another prime, reduced exactly mod q
  __syncwarp();
  if (R == 4) {
    nb_round_hi<FWD>(x, hw, q);
  } else {
    nb_round_hi<FWD>(x, FWD ? hw : lw, q);
#pragma unroll
    for (int e = 0; e < 16; e++) sm[G::addr(c, kmap<R>(FWD, e, tau))] = x[e];
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 16; e++) x[e] = sm[G::addr(c, kmap<R>(!FWD, e, tau))];
    nb_round_hi<FWD>(x, FWD ? lw : hw, q);
  }
  uint2 scale = make_uint2(0, 0);
  if (EPI == EPI_SCALE) scale = __ldg(lb.scale);
#pragma unroll
  for (int e = 0; e < 16; e++)
    lb.dst[G::gidx(tile, c, kmap<R>(R == 8 && !FWD, e, tau))] =
        EPI == EPI_SCALE ? shoup(x[e], scale.x, scale.y, q) : x[e];
}

}  // namespace fhe
