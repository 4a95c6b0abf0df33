// The stages of a key switch on the small ring (N = 2^12), one limb per CTA.
//
// A 4096-coefficient limb is one CTA's 256 x 16 register values, so a whole transform runs in
// one launch (round 0 across the CTA: the column pass; rounds 1 and 2 inside half-warps: the
// block pass of ntt_blk.cuh), and what stands before and after it rides along:
//   k_small_ntt   forward, from coefficients, from another prime's limb (rescale), or from the
//                 base conversion of up to 16 limbs formed in the prologue; ending plain, in the
//                 ModDown combine or in the rescale;
//   k_small_intt  inverse (with the rotation's gather, or of HMult's d2 = a1 b1) and output scale;
//   k_small_ip    the key inner product of one extended limb and half; a special limb of a key
//                 switch goes on to its inverse transform in the same CTA.
// A key switch is then four launches (inverse, convert + forward, inner product + inverse,
// convert + forward + combine) instead of eleven, and a rescale two instead of four.  What
// bounds it: launches and the latency of a handful of CTAs, not bandwidth (a limb is 16 KB);
// the conversion runs on CUDA cores whatever fhe_ctx_set_bconv says (same bits).  Measured on
// one GB300, against the two-pass stages as dependent launches: HMult + rescale at L = 4, K = 2
// 75 -> 52 us, one double-hoisted CoeffToSlot level at L = 8, K = 2 124 -> 93 us.  The on-the-fly
// twiddle mode and the plain pipeline keep the two-pass stages.
#pragma once
#include "ntt_col.cuh"

namespace fhe {

constexpr int kSmallLogN = 12;

// round 0 of the CTA: element 256 e + tid; tables staged per warp (entry 2^m + j, no CTA barrier)
struct SmallShared {
  __align__(16) uint32_t sm[16 * 272];
  __align__(16) uint2 hws[16 * 16];  // round 1, per block
  __align__(16) uint2 h0[8][16];     // round 0, per warp
};

// inverse from lo layout to the scaled coefficients, written as element 256 e + tid
__device__ __forceinline__ void small_inverse(uint32_t (&x)[16], SmallShared &s, const uint2 (&tl)[16], uint2 scale,
                                              uint32_t q, uint32_t *dst) {
  const int tid = threadIdx.x, c = tid >> 4, tau = tid & 15;
  blk_inverse(x, s.sm, c, tau, s.hws + c * 16, tl, q);
#pragma unroll
  for (int e = 0; e < 16; e++) s.sm[nb_blk_addr(c, (e << 4) | tau)] = x[e];
  __syncthreads();
#pragma unroll
  for (int e = 0; e < 16; e++) x[e] = s.sm[nb_blk_addr(e, tid)];
  nb_round_hi<false>(x, s.h0[tid >> 5], q);
#pragma unroll
  for (int e = 0; e < 16; e++) dst[e * 256 + tid] = shoup(x[e], scale.x, scale.y, q);
}

template <int PRO, bool DEP>
__global__ void __launch_bounds__(kNttThreads, PRO == PRO_MUL ? 3 : 4) k_small_intt(const __grid_constant__ SegList sl, const NttTables tb) {
  __shared__ SmallShared s;
  const int tid = threadIdx.x, c = tid >> 4, tau = tid & 15;
  const Limb lb = limb_at<false>(sl, blockIdx.x, tb.ninv, kSmallLogN);
  const PrimeC P = tb.pc[lb.prime];
  const uint32_t q = P.q;
  const uint2 h1 = blk_hi_twiddle<kSmallLogN, false>(tb, lb.prime, c, tau);
  const uint2 h0 = __ldg(tb.tw_inv + ((size_t)lb.prime << kSmallLogN) + tau);
  const uint2 scale = __ldg(lb.scale);
  uint2 tl[16];
  load_lo_twiddles<kSmallLogN>(tb.lo_inv, lb.prime, 0, tid, tl);
  if (DEP) dep_wait();
  uint32_t x[16];
  blk_load<kSmallLogN, PRO, DEP>(x, lb, P, c, s.sm, c, tau, [&] {
    s.hws[tid] = h1;
    if ((tid & 31) < 16) s.h0[tid >> 5][tau] = h0;
  });
  small_inverse(x, s, tl, scale, q, lb.dst);
}

template <int PRO, int EPI, bool DEP>
__global__ void __launch_bounds__(kNttThreads, PRO == PRO_BCONV ? 2 : 4)
    k_small_ntt(const __grid_constant__ SegList sl, const NttTables tb) {
  __shared__ SmallShared s;
  const int tid = threadIdx.x, c = tid >> 4, tau = tid & 15;
  const Limb lb = limb_at<EPI == EPI_COMBINE>(sl, blockIdx.x, tb.ninv, kSmallLogN);
  const PrimeC P = tb.pc[lb.prime];
  const uint32_t q = P.q;
  s.hws[tid] = blk_hi_twiddle<kSmallLogN, true>(tb, lb.prime, c, tau);
  if ((tid & 31) < 16) s.h0[tid >> 5][tau] = __ldg(tb.tw_fwd + ((size_t)lb.prime << kSmallLogN) + tau);
  uint2 scale = make_uint2(0, 0);
  if (EPI == EPI_COMBINE || EPI == EPI_RESCALE) scale = __ldg(lb.scale);
  __syncwarp();
  if (DEP) dep_wait();
  uint32_t x[16];
  if (PRO == PRO_BCONV) {
    // sum_j y_j T_j: three products below 2^62 between folds (fold34 leaves less than
    // 2^61 + 2^34), one reduction at the end
    uint64_t acc[16] = {};
    for (int j = 0; j < lb.n_in; j++) {
      const uint32_t t = __ldg(lb.T + j);
      const uint32_t *y = lb.src + ((size_t)j << kSmallLogN) + tid;
#pragma unroll
      for (int e = 0; e < 16; e++) acc[e] += (uint64_t)ld_in<DEP>(y + e * 256) * t;
      if (j % 3 == 2)
#pragma unroll
        for (int e = 0; e < 16; e++) acc[e] = fold34(acc[e], P.r34);
    }
#pragma unroll
    for (int e = 0; e < 16; e++) x[e] = reduce_u64(acc[e], P);
  } else {
#pragma unroll
    for (int e = 0; e < 16; e++) x[e] = ld_in<DEP>(lb.src + e * 256 + tid);
    if (PRO == PRO_REDUCE)
#pragma unroll
      for (int e = 0; e < 16; e++) x[e] = reduce_u64(x[e], P);
  }
  nb_round_hi<true>(x, s.h0[tid >> 5], q);
#pragma unroll
  for (int e = 0; e < 16; e++) s.sm[nb_blk_addr(e, tid)] = x[e];
  uint2 tl[16];
  load_lo_twiddles<kSmallLogN>(tb.lo_fwd, lb.prime, 0, tid, tl);
  __syncthreads();
#pragma unroll
  for (int e = 0; e < 16; e++) x[e] = s.sm[nb_blk_addr(c, (e << 4) | tau)];
  blk_forward(x, s.sm, c, tau, s.hws + c * 16, tl, q);
  blk_store<EPI, DEP>(sl, lb, c, s.sm, c, tau, scale, q);
}

// One CTA per extended limb and half: u_c = sum_j ModUp_j key_j[c] (+ P addp_c on the q-limbs),
// at 16 coefficients per thread in memory order.  seg.c = 1: a special limb of a key switch,
// whose inverse transform follows (seg.dst = UC, halves K limbs apart, seg.scale its output
// scale); else u is written (halves n_ext limbs apart).
template <bool MUL, bool DEP>
__global__ void __launch_bounds__(kNttThreads, 2) k_small_ip(const __grid_constant__ SegList sl, const NttTables tb) {
  constexpr int N = 1 << kSmallLogN;
  __shared__ SmallShared s;
  const int tid = threadIdx.x, c = tid >> 4, tau = tid & 15, cc = blockIdx.x & 1;
  int within;
  const Seg &sg = seg_at(sl, seg_find(sl, blockIdx.x >> 1, within));
  const KsArgs &ks = item_ks(sl, sg);
  const int t = sg.t0 + within, row = sg.key_row0 + within, prime = sg.prime + within;
  const bool invert = sg.c != 0;
  const PrimeC P = tb.pc[prime];
  const uint32_t q = P.q;
  if (invert) {
    s.hws[tid] = blk_hi_twiddle<kSmallLogN, false>(tb, prime, c, tau);
    if ((tid & 31) < 16) s.h0[tid >> 5][tau] = __ldg(tb.tw_inv + ((size_t)prime << kSmallLogN) + tau);
  }
  auto at = [&](int i) { return c * 256 + 64 * i + 4 * tau; };  // this thread's chunks
  // four words at chunk i of a limb read through sigma_g
  auto load = [&](const uint32_t *p, uint32_t g, int i, uint32_t *w) {
    if (g == 1u) {
      ld_in4<DEP>(p + at(i), w);
    } else {
#pragma unroll
      for (int e = 0; e < 4; e++) w[e] = ld_in<DEP>(p + galois_src((uint32_t)(at(i) + e), g, kSmallLogN));
    }
  };
  if (DEP) dep_wait();
  uint64_t acc[16] = {};
  const size_t half = (size_t)(ks.L + ks.K) * N;
  for (int jd = 0; jd < ks.beta; jd++) {
    const bool own = t < ks.level && t >= jd * ks.alpha && t < (jd + 1) * ks.alpha;
    const uint32_t *ep = own ? ks.own + (size_t)t * N : ks.ext + ((size_t)jd * ks.n_ext + t) * N;
    const uint32_t *kp = ks.key + (2 * jd + cc) * half + (size_t)row * N;
#pragma unroll
    for (int i = 0; i < 4; i++) {
      uint32_t ev[4];
      if (MUL && own && ks.mul_a) {  // HMult's d2 = a1 b1
        uint32_t w[4];
        ld_in4<DEP>(ks.mul_a + (size_t)(ks.level + t) * N + at(i), ev);
        ld_in4<DEP>(ks.mul_b + (size_t)(ks.level + t) * N + at(i), w);
#pragma unroll
        for (int e = 0; e < 4; e++) ev[e] = mul_mod(ev[e], w[e], P);
      } else {
        load(ep, own ? ks.galois_own : ks.galois_ext, i, ev);
      }
      const uint4 kv = __ldg(reinterpret_cast<const uint4 *>(kp + at(i)));
      acc[4 * i] += (uint64_t)ev[0] * kv.x;
      acc[4 * i + 1] += (uint64_t)ev[1] * kv.y;
      acc[4 * i + 2] += (uint64_t)ev[2] * kv.z;
      acc[4 * i + 3] += (uint64_t)ev[3] * kv.w;
    }
  }
  uint32_t x[16];
#pragma unroll
  for (int e = 0; e < 16; e++) x[e] = reduce_u64(acc[e], P);
  if (ks.addp && t < ks.level && (cc == 0 || ks.add_c1)) {
    const uint2 pm = ks.pmod[t];
    const uint32_t *ap = ks.addp + ((size_t)cc * ks.level + t) * N;
#pragma unroll
    for (int i = 0; i < 4; i++) {
      uint32_t w[4];
      load(ap, ks.galois_add, i, w);
#pragma unroll
      for (int e = 0; e < 4; e++) x[4 * i + e] = add_mod(x[4 * i + e], shoup(w[e], pm.x, pm.y, q), q);
    }
  }
  if (MUL && ks.mul_a && t < ks.level) {  // HMult's d0 = a0 b0, d1 = a0 b1 + a1 b0
    const uint2 pm = ks.pmod[t];
    const size_t p0 = (size_t)t * N, p1 = (size_t)(ks.level + t) * N;
#pragma unroll
    for (int i = 0; i < 4; i++) {
      uint32_t a0[4], b0[4], a1[4], b1[4];
      ld_in4<DEP>(ks.mul_a + p0 + at(i), a0);
      ld_in4<DEP>(ks.mul_b + (cc ? p1 : p0) + at(i), b0);  // a0 b0, or a0 b1 ...
      if (cc) {
        ld_in4<DEP>(ks.mul_a + p1 + at(i), a1);
        ld_in4<DEP>(ks.mul_b + p0 + at(i), b1);  // ... + a1 b0
      }
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const uint64_t d = (uint64_t)a0[e] * b0[e] + (cc ? (uint64_t)a1[e] * b1[e] : 0);  // < 2^63
        x[4 * i + e] = add_mod(x[4 * i + e], shoup(reduce_u64(d, P), pm.x, pm.y, q), q);
      }
    }
  }
  uint32_t *dst = sg.dst + ((size_t)cc * (invert ? ks.K : ks.n_ext) + within) * N;
  if (!invert) {
#pragma unroll
    for (int i = 0; i < 4; i++) st4(dst + at(i), x + 4 * i);
    return;
  }
  uint2 tl[16];
  load_lo_twiddles<kSmallLogN>(tb.lo_inv, prime, 0, tid, tl);
#pragma unroll
  for (int i = 0; i < 4; i++) st4(blk_lin(s.sm, c, tau, i), x + 4 * i);
  __syncwarp();
#pragma unroll
  for (int m = 0; m < 4; m++) ld4(s.sm + nb_blk_addr(c, (tau << 4) | (4 * m)), x + 4 * m);
  small_inverse(x, s, tl, __ldg(sg.scale + within), q, dst);
}

}  // namespace fhe
