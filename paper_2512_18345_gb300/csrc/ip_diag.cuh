// A double-hoisted transform's baby rotations and diagonals in one pass (k_baby_diag), and its giant
// steps' key switches and sum in another (k_giant_ip).
//
// k_baby_diag: for one unit of an extended limb, every baby step's inner product
// u_b = sum_j sigma_b(ModUp_j) key_b,j (+ P sigma_b(c0) on the q-limbs) is formed in registers
// and multiplied at once by the diagonals of up to kBdGiant giant steps, so the baby rotations
// (two extended polynomials each) are neither written nor read back.
//
// Bound by the keys and the diagonals, both read once, from HBM.  A CoeffToSlot level at N = 2^16,
// L = 48, alpha = K = 12 (15 rotating baby and 4 giant steps, 63 diagonals): 3.0 GB in 510 us (5.9
// TB/s), where the two kernels moved 3.9 GB in 661 us; the level 1256 -> 1105 us, one at N = 2^12,
// L = 8 65 -> 58 us.  Work split: as in the hoisted
// inner product (ip_hoisted.cuh), every warp is its own pipeline over 128-coefficient units
// with a ring of D stages filled by 16-byte cp.async pieces; a stage is one baby step of one
// unit.  Neighbouring warps take neighbouring units, so that the digits in use at any time are
// a few limbs', which stay in L2 while every baby step reads them through its automorphism.
//
// Stage layout (rows of 128 words, per warp): beta digit rows, the pass-through row, 2 beta key
// rows, kBdGiant diagonal rows.  A baby step without rotation is P ct: row 0 holds c1, the
// pass-through row c0, and there is no key.
#pragma once
#include "ip_hoisted.cuh"

namespace fhe {

constexpr int kBdMaxBaby = 32, kBdGiant = 4;
// 12 warps: three per scheduler, each with two stages of 17 rows of 512 bytes (13 warps, which the
// shared memory still holds, took a CoeffToSlot level 1108 -> 1155 us, 8 warps with three stages 1286)
constexpr int kBdMaxWarps = 12;
constexpr int kBdStages = 2;
struct BabyDiagArgs {
  const uint32_t *key[kBdMaxBaby];
  uint32_t gal[kBdMaxBaby];
  const uint32_t *ct, *ext, *diags;  // [2][level][N], [beta][nlimb][N], [n_diag][nlimb][N]
  const uint2 *pmod;
  uint32_t *out;                     // [giant][2][nlimb][N]
  int giant, nlimb, level, L, K, alpha, beta;
  uint32_t idmask;                   // the baby steps without rotation
  uint32_t gmask[kBdGiant];          // bit b: giant step g meets baby step b
  int16_t didx[kBdGiant][kBdMaxBaby];
};
__host__ __device__ constexpr int baby_diag_stage_words(int beta) { return kIhUnit * (3 * beta + 1 + kBdGiant); }

template <bool DEP>
__global__ void __launch_bounds__(kBdMaxWarps * 32, 1)
    k_baby_diag(const __grid_constant__ BabyDiagArgs a, const PrimeC *pc, int logn) {
  constexpr int D = kBdStages;
  extern __shared__ __align__(128) uint8_t smem[];
  const int warp = threadIdx.x >> 5, l = threadIdx.x & 31;
  const size_t N = (size_t)1 << logn, poly = (size_t)a.nlimb * N, half = (size_t)(a.L + a.K) * N;
  const int lpl = logn - 7;  // log2 of the units per limb (kIhUnit = 2^7)
  const int total = a.nlimb << lpl;
  const int beta = a.beta, sw = baby_diag_stage_words(beta);
  const int PR = beta * kIhUnit, KR = PR + kIhUnit, GR = KR + 2 * beta * kIhUnit;
  uint32_t *ring = reinterpret_cast<uint32_t *>(smem) + (size_t)warp * D * sw;
  const uint32_t ring_s = smem_addr(ring);
  const int wpc = (int)(blockDim.x >> 5);
  const int gw = (int)blockIdx.x * wpc + warp, nw = (int)gridDim.x * wpc;
  const uint64_t once = l2_evict_first_policy();  // keys and diagonals are read exactly once
  const int eb = l >> 3, part = l & 7;                 // staging: this lane's block and 16-byte piece
  const uint32_t pw = (uint32_t)(eb * 32 + 4 * part);  // that piece's word within a staged row
  const uint32_t all = a.gmask[0] | a.gmask[1] | a.gmask[2] | a.gmask[3];
  auto steps = [&](int i) { return i < a.level ? all : all & ~a.idmask; };  // the baby steps of limb i

  // the staging cursor: unit su and its baby steps still to be staged
  int su = gw, ring_at = 0;
  uint32_t sm = su < total ? steps(su >> lpl) : 0u;
  auto stage = [&] {
    while (!sm && su < total) {
      su += nw;
      if (su < total) sm = steps(su >> lpl);
    }
    if (sm) {
      const int b = __ffs(sm) - 1, i = su >> lpl;
      sm &= sm - 1;
      const uint32_t c0 = (uint32_t)(su & ((1 << lpl) - 1)) * kIhUnit;
      const uint32_t dst = ring_s + (uint32_t)(ring_at * sw + pw) * 4u;
      auto row = [&](int words) { return dst + (uint32_t)words * 4u; };
      const size_t at = ((size_t)(galois_src(c0 + 32u * (uint32_t)eb, a.gal[b], logn) >> 5) << 5) + 4 * part;
      const size_t lim = (size_t)i * N;
      if (i < a.level) cp_async_plain16(row(PR), a.ct + lim + at);
      const uint32_t *own = a.ct + (size_t)a.level * N + lim;
      if ((a.idmask >> b) & 1u) {
        cp_async_plain16(row(0), own + at);
      } else {
        const int jown = i < a.level ? i / a.alpha : -1;
        const uint32_t *kp = a.key[b] + (size_t)(i < a.level ? i : a.L + (i - a.level)) * N + c0 + pw;
#pragma unroll
        for (int r = 0; r < 4; r++)
          if (r < beta) {
            cp_async_plain16(row(r * kIhUnit), (r == jown ? own : a.ext + (size_t)r * poly + lim) + at);
            cp_async16_hint(row(KR + 2 * r * kIhUnit), kp + (size_t)(2 * r) * half, once);
            cp_async16_hint(row(KR + (2 * r + 1) * kIhUnit), kp + (size_t)(2 * r + 1) * half, once);
          }
      }
#pragma unroll
      for (int g = 0; g < kBdGiant; g++)
        if ((a.gmask[g] >> b) & 1u)
          cp_async16_hint(row(GR + g * kIhUnit), a.diags + (size_t)a.didx[g][b] * poly + lim + c0 + pw, once);
    }
    if (++ring_at == D) ring_at = 0;
    cp_async_commit();  // (an empty group past the end keeps the group count uniform)
  };

  if (DEP) dep_wait();
#pragma unroll
  for (int k = 0; k < D - 1; k++) stage();
  int at = 0;
  for (int u = gw; u < total; u += nw) {
    const int i = u >> lpl;
    const uint32_t c0 = (uint32_t)(u & ((1 << lpl) - 1)) * kIhUnit;
    const PrimeC P = pc[i < a.level ? i : a.L + (i - a.level)];
    const uint2 pm = i < a.level ? a.pmod[i] : make_uint2(0, 0);
    uint64_t acc[2][kBdGiant][4] = {};
    int since = 0;  // products added to each accumulator since the last fold
    for (uint32_t live = steps(i); live; live &= live - 1) {
      const int b = __ffs(live) - 1;
      stage();
      cp_async_wait_group<D - 1>();  // this lane's pieces of the step have landed ...
      __syncwarp();                  // ... and every lane's
      const uint32_t *st = ring + (size_t)at * sw;
      if (++at == D) at = 0;
      uint32_t x0[4], x1[4];
      if ((a.idmask >> b) & 1u) {
#pragma unroll
        for (int e = 0; e < 4; e++) {
          x0[e] = shoup(st[PR + 32 * e + l], pm, P.q);
          x1[e] = shoup(st[32 * e + l], pm, P.q);
        }
      } else {
        int off[4];
        uint64_t a0[4] = {}, a1[4] = {};
#pragma unroll
        for (int e = 0; e < 4; e++) off[e] = e * 32 + (int)(galois_src(c0 + 32u * e + l, a.gal[b], logn) & 31u);
#pragma unroll
        for (int r = 0; r < 4; r++)
          if (r < beta) {
            const uint32_t *dr = st + r * kIhUnit, *kb = st + KR + 2 * r * kIhUnit + l;
#pragma unroll
            for (int e = 0; e < 4; e++) {
              const uint32_t ev = dr[off[e]];
              a0[e] += (uint64_t)ev * kb[32 * e];
              a1[e] += (uint64_t)ev * kb[kIhUnit + 32 * e];
            }
          }
#pragma unroll
        for (int e = 0; e < 4; e++) {
          x0[e] = reduce_u64(a0[e], P);
          x1[e] = reduce_u64(a1[e], P);
          if (i < a.level) x0[e] = add_mod(x0[e], shoup(st[PR + off[e]], pm, P.q), P.q);
        }
      }
#pragma unroll
      for (int g = 0; g < kBdGiant; g++)
        if ((a.gmask[g] >> b) & 1u)
#pragma unroll
          for (int e = 0; e < 4; e++) {
            const uint32_t d = st[GR + g * kIhUnit + 32 * e + l];
            acc[0][g][e] += (uint64_t)d * x0[e];
            acc[1][g][e] += (uint64_t)d * x1[e];
          }
      if (++since == 3) {
        since = 0;
#pragma unroll
        for (int g = 0; g < kBdGiant; g++)
#pragma unroll
          for (int e = 0; e < 4; e++) {
            acc[0][g][e] = fold34(acc[0][g][e], P.r34);
            acc[1][g][e] = fold34(acc[1][g][e], P.r34);
          }
      }
      __syncwarp();  // every lane is done with the stage before it is refilled
    }
    uint32_t *o = a.out + (size_t)i * N + c0 + l;
#pragma unroll
    for (int g = 0; g < kBdGiant; g++)
      if (g < a.giant)
#pragma unroll
        for (int e = 0; e < 4; e++) {
          o[(size_t)(2 * g) * poly + 32 * e] = reduce_u64(acc[0][g][e], P);
          o[(size_t)(2 * g + 1) * poly + 32 * e] = reduce_u64(acc[1][g][e], P);
        }
  }
  cp_async_wait_group<0>();  // nothing in flight when the warp leaves
}

// Giant steps of a double-hoisted transform, in the extended basis:
//   out_0 = sum_g sigma_g(inner_g,0) + u_g,0,   out_1 = sum_g u_g,1,
// u_g the key switch's inner product over the digits of ModDown(inner_g,1) read through sigma_g; a
// giant step without rotation adds inner_g itself.  The same warp pipelines, one giant step per
// stage: beta digit rows, the c0 row, 2 beta key rows.  The sums stay in registers, so the u_g
// (two extended polynomials each) are neither written nor read back.  Bound by HBM: the CoeffToSlot
// level above (3 rotating giant steps) reads 0.38 GB of keys and 0.27 GB of digits and c0 halves in
// 113 us, where an inner product and a sum kernel took 150 us (the level 1105 -> 1062 us, the one at
// N = 2^12 58 -> 50 us); 12 warps instead of 16 differ by less than the runs do.
constexpr int kGiMaxGiant = 16, kGiMaxWarps = 16, kGiStages = 2;
struct GiantIpArgs {
  const uint32_t *key[kGiMaxGiant];    // null: no rotation
  const uint32_t *ext[kGiMaxGiant];    // [beta][nlimb][N]
  const uint32_t *own[kGiMaxGiant];    // [level][N]
  const uint32_t *inner[kGiMaxGiant];  // [2][nlimb][N]
  uint32_t gal[kGiMaxGiant];
  uint32_t *out;                       // [2][nlimb][N]
  int giant, nlimb, level, L, K, alpha, beta;
};
__host__ __device__ constexpr int giant_ip_stage_words(int beta) { return kIhUnit * (3 * beta + 1); }

template <bool DEP>
__global__ void __launch_bounds__(kGiMaxWarps * 32, 1)
    k_giant_ip(const __grid_constant__ GiantIpArgs a, const PrimeC *pc, int logn) {
  constexpr int D = kGiStages;
  extern __shared__ __align__(128) uint8_t smem[];
  const int warp = threadIdx.x >> 5, l = threadIdx.x & 31;
  const size_t N = (size_t)1 << logn, poly = (size_t)a.nlimb * N, half = (size_t)(a.L + a.K) * N;
  const int lpl = logn - 7;
  const int total = a.nlimb << lpl;
  const int beta = a.beta, sw = giant_ip_stage_words(beta);
  const int PR = beta * kIhUnit, KR = PR + kIhUnit;
  uint32_t *ring = reinterpret_cast<uint32_t *>(smem) + (size_t)warp * D * sw;
  const uint32_t ring_s = smem_addr(ring);
  const int wpc = (int)(blockDim.x >> 5);
  const int gw = (int)blockIdx.x * wpc + warp, nw = (int)gridDim.x * wpc;
  const uint64_t once = l2_evict_first_policy();  // keys are read exactly once
  const int eb = l >> 3, part = l & 7;
  const uint32_t pw = (uint32_t)(eb * 32 + 4 * part);

  int su = gw, sg = 0, ring_at = 0;  // the staging cursor: unit and giant step
  auto stage = [&] {
    if (su < total) {
      const int i = su >> lpl;
      const uint32_t c0 = (uint32_t)(su & ((1 << lpl) - 1)) * kIhUnit;
      const uint32_t dst = ring_s + (uint32_t)(ring_at * sw + pw) * 4u;
      auto row = [&](int words) { return dst + (uint32_t)words * 4u; };
      const size_t lim = (size_t)i * N;
      const size_t at = ((size_t)(galois_src(c0 + 32u * (uint32_t)eb, a.gal[sg], logn) >> 5) << 5) + 4 * part;
      cp_async_plain16(row(PR), a.inner[sg] + lim + at);
      if (!a.key[sg]) {
        cp_async_plain16(row(0), a.inner[sg] + poly + lim + at);
      } else {
        const int jown = i < a.level ? i / a.alpha : -1;
        const uint32_t *kp = a.key[sg] + (size_t)(i < a.level ? i : a.L + (i - a.level)) * N + c0 + pw;
#pragma unroll
        for (int r = 0; r < 4; r++)
          if (r < beta) {
            cp_async_plain16(row(r * kIhUnit), (r == jown ? a.own[sg] : a.ext[sg] + (size_t)r * poly) + lim + at);
            cp_async16_hint(row(KR + 2 * r * kIhUnit), kp + (size_t)(2 * r) * half, once);
            cp_async16_hint(row(KR + (2 * r + 1) * kIhUnit), kp + (size_t)(2 * r + 1) * half, once);
          }
      }
      if (++sg == a.giant) {
        sg = 0;
        su += nw;
      }
    }
    if (++ring_at == D) ring_at = 0;
    cp_async_commit();
  };

  if (DEP) dep_wait();
#pragma unroll
  for (int k = 0; k < D - 1; k++) stage();
  int at = 0;
  for (int u = gw; u < total; u += nw) {
    const int i = u >> lpl;
    const uint32_t c0 = (uint32_t)(u & ((1 << lpl) - 1)) * kIhUnit;
    const PrimeC P = pc[i < a.level ? i : a.L + (i - a.level)];
    uint32_t s0[4] = {}, s1[4] = {};
    for (int g = 0; g < a.giant; g++) {
      stage();
      cp_async_wait_group<D - 1>();
      __syncwarp();
      const uint32_t *st = ring + (size_t)at * sw;
      if (++at == D) at = 0;
      if (!a.key[g]) {
#pragma unroll
        for (int e = 0; e < 4; e++) {
          s0[e] = add_mod(s0[e], st[PR + 32 * e + l], P.q);
          s1[e] = add_mod(s1[e], st[32 * e + l], P.q);
        }
      } else {
        int off[4];
        uint64_t a0[4] = {}, a1[4] = {};
#pragma unroll
        for (int e = 0; e < 4; e++) off[e] = e * 32 + (int)(galois_src(c0 + 32u * e + l, a.gal[g], logn) & 31u);
#pragma unroll
        for (int r = 0; r < 4; r++)
          if (r < beta) {
            const uint32_t *dr = st + r * kIhUnit, *kb = st + KR + 2 * r * kIhUnit + l;
#pragma unroll
            for (int e = 0; e < 4; e++) {
              const uint32_t ev = dr[off[e]];
              a0[e] += (uint64_t)ev * kb[32 * e];
              a1[e] += (uint64_t)ev * kb[kIhUnit + 32 * e];
            }
          }
#pragma unroll
        for (int e = 0; e < 4; e++) {
          s0[e] = add_mod(s0[e], add_mod(reduce_u64(a0[e], P), st[PR + off[e]], P.q), P.q);
          s1[e] = add_mod(s1[e], reduce_u64(a1[e], P), P.q);
        }
      }
      __syncwarp();
    }
    uint32_t *o = a.out + (size_t)i * N + c0 + l;
#pragma unroll
    for (int e = 0; e < 4; e++) {
      o[32 * e] = s0[e];
      o[poly + 32 * e] = s1[e];
    }
  }
  cp_async_wait_group<0>();
}

}  // namespace fhe
