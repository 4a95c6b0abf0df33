// Shared device definitions of the GB300 key-switching library: word-sized
// modular arithmetic on 31-bit primes and the launch descriptors every kernel
// reads.  Device-only (plus plain structs the host fills in).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace fhe {

constexpr int kMaxPrimes = 64;
constexpr int kMaxSeg = 96;       // segments passed by value per launch (kernel parameters up to 32 KB)
constexpr int kTile = 4096;       // elements per NTT tile (16 KB)
constexpr int kNttThreads = 256;  // 16 elements per thread

// Per-prime constants (host-computed).  q < 2^31 so that 2q fits in 32 bits.
struct PrimeC {
  uint32_t q;
  uint32_t r32, r32s;   // 2^32 mod q and its Shoup companion floor(r32 2^32 / q)
  uint32_t div32;       // floor(2^32 / q) = Shoup companion of 1
  uint32_t r64, r64s;   // 2^64 mod q and companion
  uint32_t r34;         // 2^34 mod q (the diagonal pass's fold constant)
  uint32_t pad1;
};

// ---------------------------------------------------------------- dependent launches
// A stage kernel of a single-call program may start before the one it follows has ended
// (programmatic dependent launch): it stages its constants, then dep_wait() holds it until the
// previous kernel has completed and its writes are visible, and lets the next kernel start its
// own prologue (one kernel ahead at most).  What an earlier kernel of the program wrote is read only after dep_wait, with ld_dep (L2;
// ordered after the wait): ld.global.nc may be moved above it and may hit a line that L1 kept
// from before the write.  Only the DEP forms of the kernels wait: the wait also holds back the
// loads behind a CTA's constants, which cost the 8-rotation graph step 512 -> 552 us when every
// launch had it.
__device__ __forceinline__ void dep_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ uint32_t ld_dep(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint4 ld_dep4(const uint32_t *p) {
  uint4 v;
  asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

template <bool DEP>
__device__ __forceinline__ uint32_t ld_in(const uint32_t *p) { return DEP ? ld_dep(p) : __ldg(p); }
template <bool DEP>
__device__ __forceinline__ uint4 ld_in4(const uint32_t *p) {
  return DEP ? ld_dep4(p) : __ldg(reinterpret_cast<const uint4 *>(p));
}

// ---------------------------------------------------------------- arithmetic
// [0, 2q) -> [0, q): if x < q then x - q wraps above x and min keeps x.
__device__ __forceinline__ uint32_t red2(uint32_t x, uint32_t q) { return min(x, x - q); }

// Shoup product a * w mod q in [0, 2q) for any a < 2^32, w < q, ws = floor(w 2^32 / q).
__device__ __forceinline__ uint32_t shoup_lazy(uint32_t a, uint32_t w, uint32_t ws, uint32_t q) {
  return a * w - __umulhi(a, ws) * q;
}
__device__ __forceinline__ uint32_t shoup(uint32_t a, uint32_t w, uint32_t ws, uint32_t q) {
  return red2(shoup_lazy(a, w, ws, q), q);
}
__device__ __forceinline__ uint32_t shoup(uint32_t a, uint2 w, uint32_t q) { return shoup(a, w.x, w.y, q); }

__device__ __forceinline__ uint32_t add_mod(uint32_t a, uint32_t b, uint32_t q) { return red2(a + b, q); }
__device__ __forceinline__ uint32_t sub_mod(uint32_t a, uint32_t b, uint32_t q) { return red2(a + q - b, q); }

// Exact x mod q for any 64-bit x: x = xh 2^32 + xl, xh * (2^32 mod q) and xl
// each reduced with a Shoup product (the second with w = 1).
__device__ __forceinline__ uint32_t reduce_u64(uint64_t x, const PrimeC &P) {
  const uint32_t xh = (uint32_t)(x >> 32), xl = (uint32_t)x;
  const uint32_t t1 = red2(shoup_lazy(xh, P.r32, P.r32s, P.q), P.q);
  const uint32_t t2 = red2(xl - __umulhi(xl, P.div32) * P.q, P.q);
  return red2(t1 + t2, P.q);
}

__device__ __forceinline__ uint32_t mul_mod(uint32_t a, uint32_t b, const PrimeC &P) {
  return reduce_u64((uint64_t)a * b, P);
}

// a = hi 2^34 + lo  ->  hi r34 + lo with r34 = 2^34 mod q: the same residue, below 2^61 + 2^34
// for any 64-bit a (hi < 2^30, r34 < 2^31), so three more products below 2^62 still fit
__device__ __forceinline__ uint64_t fold34(uint64_t a, uint32_t r34) {
  return (uint64_t)(uint32_t)(a >> 34) * r34 + (a & ((1ull << 34) - 1));
}

// ---------------------------------------------------------------- automorphism
// NTT-form Galois map sigma_k: slot i (value at psi^(2 brv(i)+1)) of the
// output is slot j of the input with 2 brv(j) + 1 = (2 brv(i) + 1) k mod 2N,
// i.e. brv(j) = brv(i) k + (k - 1)/2 mod N.
__device__ __forceinline__ uint32_t galois_src(uint32_t i, uint32_t k, int logn) {
  const uint32_t r = __brev(i) >> (32 - logn);
  const uint32_t rj = (r * k + (k >> 1)) & ((1u << logn) - 1u);
  return __brev(rj) >> (32 - logn);
}

// ---------------------------------------------------------------- descriptors
// A segment is a run of n limbs whose primes are consecutive (prime, prime+1,
// ...).  Limb l of the run reads src + l * src_stride * N and writes dst + l * N.
struct Seg {
  const uint32_t *src;
  uint32_t *dst;
  const uint32_t *src2;  // second operand (element-wise kernels), limb stride N, or null
  int n;             // limbs in the run
  int prime;         // prime index (into q_0.., p_0..) of the first limb
  int src_stride;    // in limbs (0: every limb reads the same source limb)
  const uint2 *scale;  // per-limb Shoup constant pairs (inverse-NTT output scale), or null
  int t0;            // extended-basis index of the first limb (inner product)
  int key_row0;      // key row of the first limb
  int c;             // small ring's inner product: 1 where the limb's inverse transform follows
  int item;          // index of this segment's key-switching arguments
  uint32_t galois;   // Galois element applied when src is gathered (1: none)
  int n_in;          // PRO_BCONV: src is n_in limbs, T the first limb's row of the conversion table
  const uint32_t *T;
};

// Key-switching arguments of one item (one key switch) for the inner product,
// the automorphism gathers and the ModDown combine.
struct KsArgs {
  const uint32_t *ext;   // [beta][n_ext][N] ModUp outputs (NTT form); own-digit limbs unused
  const uint32_t *own;   // [level][N] the key-switched polynomial in NTT form (own-digit limbs)
  const uint32_t *key;   // [dnum][2][L+K][N]
  const uint32_t *addp;  // [2][level][N] pass-through polynomial (c = 0, 1) of the output, or null; the
                         // inner product adds P * addp to u's q-limbs, so ModDown's (u - r) P^-1 carries it
  const uint32_t *mul_a, *mul_b;  // HMult's factors [2][level][N] when the tensor product is formed on the fly
                         // (own limbs a1 b1, pass-through (a0 b0, a0 b1 + a1 b0)), else null
  const uint32_t *r, *u; // the item's converted special limbs and inner product (PRO_SUM, EPI_SUM)
  const uint2 *pinv;     // [L] Shoup pairs of P^-1 mod q_i
  const uint2 *pmod;     // [L] Shoup pairs of P mod q_i
  int level, n_ext, beta, alpha, L, K;
  uint32_t galois_own;   // sigma applied when reading `own` (1 = none)
  uint32_t galois_ext;   // sigma applied when reading `ext` (hoisted rotations; 1 = none)
  uint32_t galois_add;   // sigma applied when reading `addp` (1 = none)
  int add_c1;            // addp's second polynomial also goes to c = 1 (HMult); a rotation adds c0 only
};

constexpr int kMaxInlineItems = 16;
constexpr int kMaxInlineLimbs = 2048;  // limbs of a by-value list (its limb -> segment map)

// One limb of a launch, as the transform passes and element-wise kernels need it.  Device
// lists hold one per limb, in launch order, so that a CTA reaches its operands through one
// load instead of three dependent ones (vmap, segment, arguments); with the by-value lists'
// limb -> segment map (below) in place of a walk over up to 96 segments, the level-24 dense
// transform went from 1403 to 1335 us and the 8-rotation graph step from 564 to 554 us.
struct alignas(16) Limb {
  const uint32_t *src;
  uint32_t *dst;
  const uint32_t *src2;
  const uint2 *scale;  // the limb's own constant (output scale, or P^-1 for a combine), or null
  const uint32_t *T;   // PRO_BCONV: its row of the conversion table, over n_in input limbs at src
  int prime;
  uint32_t galois;     // sigma applied when reading src (PRO_GATHER, EW_GATHER)
  int n;               // limbs in the segment (the HMult tensor's polynomial stride)
  int n_in;
};

// A launch's work list: segments and per-item arguments, either inline (by
// value, single operations) or in device memory (batched plans).
struct SegList {
  int nseg;
  int total;              // total limbs over all segments
  const Seg *dev;         // if non-null: segments in device memory
  const int2 *vmap;       // optional [total] (segment, limb within) for device lists
  const Limb *limbs;      // optional [total] limb descriptors for device lists
  const KsArgs *ksdev;    // if non-null: per-item arguments in device memory
  // optional limb-major order of an inline list, read by the hoisted inner product (0 groups:
  // list order): group g is lm_count[g] consecutive segments from lm_first[g], all of one size
  // and first extended-basis index, whose limbs are taken limb by limb across the segments
  int lm_groups;
  int lm_first[4], lm_count[4];
  int sum_n;                 // PRO_SUM, EPI_SUM: items ks[0..sum_n) are summed
  Seg seg[kMaxSeg];
  KsArgs ks[kMaxInlineItems];
  uint16_t first[kMaxSeg];          // inline lists: the segment's first limb, and each limb's segment
  uint8_t segof[kMaxInlineLimbs];   // (two constant loads instead of a walk over up to 96 segments)
};
static_assert(kMaxSeg <= 256, "segof holds a segment index in a byte");

// an empty by-value list: the header alone (the arrays hold what their counts say; clearing the
// 12 KB of them before each launch was a third of a small call's host time)
inline void seg_clear(SegList &l) {
  l.nseg = l.total = l.lm_groups = l.sum_n = 0;
  l.dev = nullptr;
  l.vmap = nullptr;
  l.limbs = nullptr;
  l.ksdev = nullptr;
}

// append a segment to a by-value list (the caller keeps within kMaxSeg and kMaxInlineLimbs)
inline void seg_push(SegList &l, const Seg &s) {
  l.first[l.nseg] = (uint16_t)l.total;
  for (int i = 0; i < s.n; i++) l.segof[l.total + i] = (uint8_t)l.nseg;
  l.seg[l.nseg++] = s;
  l.total += s.n;
}

__device__ __forceinline__ const Seg &seg_at(const SegList &L, int i) { return L.dev ? L.dev[i] : L.seg[i]; }
__device__ __forceinline__ const KsArgs &item_ks(const SegList &L, const Seg &s) {
  return L.ksdev ? L.ksdev[s.item] : L.ks[s.item];
}

// Locate limb v (0 <= v < total) of a segment list: returns segment index and limb within it.
__device__ __forceinline__ int seg_find(const SegList &L, int v, int &within) {
  if (L.vmap) {
    const int2 m = L.vmap[v];
    within = m.y;
    return m.x;
  }
  const int s = L.segof[v];
  within = v - L.first[s];
  return s;
}

// Limb v's descriptor; dflt: the per-prime constants a segment without its own scale uses.
// COMBINE: the scale is P^-1 mod the limb's prime.
template <bool COMBINE>
__device__ __forceinline__ Limb limb_at(const SegList &L, int v, const uint2 *dflt, int logn) {
  if (L.limbs) {
    const uint4 *p = reinterpret_cast<const uint4 *>(L.limbs + v);
    static_assert(sizeof(Limb) == 64, "a limb descriptor is four 16-byte loads");
    union { uint4 w[4]; Limb d; } u;
#pragma unroll
    for (int i = 0; i < 4; i++) u.w[i] = __ldg(p + i);
    return u.d;
  }
  int within;
  const Seg &s = L.seg[seg_find(L, v, within)];
  const size_t off = (size_t)within << logn;
  Limb d;
  d.src = s.src ? s.src + s.src_stride * off : nullptr;
  d.dst = s.dst + off;
  d.src2 = s.src2 ? s.src2 + off : nullptr;
  d.prime = s.prime + within;
  d.scale = COMBINE ? L.ks[s.item].pinv + d.prime : s.scale ? s.scale + within : dflt ? dflt + d.prime : nullptr;
  d.galois = s.galois;
  d.n = s.n;
  d.T = s.T + (size_t)within * s.n_in;
  d.n_in = s.n_in;
  return d;
}

}  // namespace fhe
