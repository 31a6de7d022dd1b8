// Ly-alpha packet transport on the GPU.
//
// Method (arXiv:2312.11448, Sec. III.B and Appendix A): packets are emitted
// per cell in proportion to the local recombination rate alpha_e n_e^2 (the
// integrand of the global loss-rate Monte Carlo), injected at a random point
// of the cell (step (1)), streamed in a straight line while the expansion
// redshifts them by dx = -H dl / v_th (step (4)), with the gas-frame frequency
// shifted by the bulk flow, omega_r = omega (1 - U_par).  A packet is absorbed
// into the integer tally of the first cell in which it comes back into line
// resonance.
//
// Kernels (one lya_transport call):
//   k_alloc_max     r_max over the emission weights (and a validity check), largest
//                   speeds
//   k_alloc_sum     Q_i = floor(2^31 r_i / r_max); compact velocity copy; block
//                   sums; last block scans them and draws the systematic-sampling
//                   offset u
//   k_alloc_prefix  packet prefix P_i = floor((N prefixQ_i + u) / sum Q), exact
//                   integer arithmetic; cell of every 32nd packet; packets per
//                   super-tile; last block: bucket offsets
//   k_emit          64 packets per warp and iteration: cell lookup in P, Philox
//                   draws; packets that are home by their quantile word are tallied,
//                   the others finished 32 at a time (resonance test in the home
//                   cell, warp-aggregated tally) or queued in their home
//                   super-tile's bucket; last block: chunks of the buckets
//   k_march         persistent warps march the queued packets (Amanatides-Woo),
//                   refilling idle lanes from the queue; tally atomics; last block
//                   closes the call
// The march is written operation by operation with round-to-nearest
// intrinsics (never contracted into FMA), in binary32 for the mixed form and
// binary64 for the FP64 form, so its integer results are reproducible.

#include <algorithm>
#include <cmath>
#include <cstring>

#include "rec_internal.cuh"
#include "rec_reduce.cuh"
#include "rec_velq.cuh"

namespace rec {
namespace {

constexpr int TT = 256;  // transport block size
constexpr int AT = kAllocThreads;

// ---- Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11) ----------------------
struct U4 {
  uint32_t a, b, c, d;
};

__device__ __forceinline__ U4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                            uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    // 32 x 32 -> 64-bit products (low and high words from one wide multiply)
    const uint64_t p0 = (uint64_t)0xD2511F53u * c0, p1 = (uint64_t)0xCD9E8D57u * c2;
    uint32_t lo0 = (uint32_t)p0, hi0 = (uint32_t)(p0 >> 32);
    uint32_t lo1 = (uint32_t)p1, hi1 = (uint32_t)(p1 >> 32);
    uint32_t n0 = hi1 ^ c1 ^ k0;
    uint32_t n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return U4{c0, c1, c2, c3};
}

// The keys of the ten rounds, (k0 + r W0, k1 + r W1), formed once on the host.
// Kernels read them from their parameters, so every round takes its key as a
// constant operand instead of adding the Weyl increments per packet.
struct Keys {
  uint32_t a[10], b[10];
};
inline Keys key_schedule(uint32_t k0, uint32_t k1) {
  Keys K;
  for (int r = 0; r < 10; ++r) {
    K.a[r] = k0;
    K.b[r] = k1;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return K;
}
__device__ __forceinline__ U4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const Keys& K) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)0xD2511F53u * c0, p1 = (uint64_t)0xCD9E8D57u * c2;
    uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ K.a[r];
    uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ K.b[r];
    c1 = (uint32_t)p1;
    c3 = (uint32_t)p0;
    c0 = n0;
    c2 = n2;
  }
  return U4{c0, c1, c2, c3};
}

// Streams: key (seed_lo, seed_hi ^ step), counter (cell, packet-in-cell, block, box).
struct Stream {
  uint32_t k0, k1, box;
};
__device__ __forceinline__ U4 draw(const Stream& s, uint32_t cell, uint32_t j, uint32_t block) {
  return philox4x32_10(cell, j, block, s.box, s.k0, s.k1);
}
// The same draw with the keys from a schedule (emission).
struct KStream {
  const Keys& K;
  uint32_t box;
};
__device__ __forceinline__ U4 draw(const KStream& s, uint32_t cell, uint32_t j, uint32_t block) {
  return philox4x32_10(cell, j, block, s.box, s.K);
}
constexpr uint32_t kAllocBlock = 0x000A110Cu;  // counter block of the allocation offset

// Uniform deviates strictly inside (0,1), exactly representable.
// Binary32: the float 1 + m 2^-23 with m the top 23 bits of r, minus 1 - 2^-24,
// is exactly (2m + 1) 2^-24 (Sterbenz: the operands are within a factor of
// two), with no integer-to-float conversion.
__device__ __forceinline__ float u01f(uint32_t r) {
  return __fsub_rn(__uint_as_float(0x3f800000u | (r >> 9)), 0x1.fffffep-1f);
}
// Binary64: the same with the top 52 bits of the word pair, 1 + m 2^-52 minus 1 - 2^-53:
// one operation on the binary64 pipe (a conversion and a product before).
__device__ __forceinline__ double u01d(uint32_t lo, uint32_t hi) {
  const uint64_t w = ((uint64_t)hi << 32) | lo;
  return __dsub_rn(__longlong_as_double((long long)(0x3ff0000000000000ull | (w >> 12))), 0x1.fffffffffffffp-1);
}

// ---- explicitly rounded arithmetic -----------------------------------------------
template <class R> struct Ar;
template <> struct Ar<float> {
  static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ float div(float a, float b) { return __fdiv_rn(a, b); }
  static __device__ __forceinline__ float rcp(float a) { return __frcp_rn(a); }  // correctly rounded 1/a
  static __device__ __forceinline__ float sqr(float a) { return __fsqrt_rn(a); }
  static __device__ __forceinline__ float inf() { return __int_as_float(0x7f800000); }
  static __device__ __forceinline__ int trunc(float a) { return __float2int_rz(a); }
};
template <> struct Ar<double> {
  static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
  static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
  static __device__ __forceinline__ double div(double a, double b) { return __ddiv_rn(a, b); }
  static __device__ __forceinline__ double rcp(double a) { return __drcp_rn(a); }  // correctly rounded 1/a
  static __device__ __forceinline__ double sqr(double a) { return __dsqrt_rn(a); }
  static __device__ __forceinline__ double inf() { return __longlong_as_double(0x7ff0000000000000ll); }
  static __device__ __forceinline__ int trunc(double a) { return __double2int_rz(a); }
};

template <class R> struct Vec4;
template <> struct Vec4<float> { using T = float4; };
template <> struct Vec4<double> { using T = double4_32a; };

// Per-precision draw layout.
template <class R> struct Draws;
template <> struct Draws<float> {
  // block 0: three cell offsets and the frequency quantile; blocks 1..16: two
  // direction pairs each
  static constexpr int kPairs = 2;
  static constexpr uint32_t kQuantBlock = 0;  // its last word leads the quantile's bits
  using Block = U4;
  static __device__ __forceinline__ bool first_of_block(int t) { return (t & 1) == 0; }
  template <class S>
  static __device__ __forceinline__ U4 block(const S& s, uint32_t c, uint32_t j, int t) {
    return draw(s, c, j, 1u + (uint32_t)(t >> 1));
  }
  static __device__ __forceinline__ void pair_from(const U4& r, int t, float* a, float* b) {
    if (t & 1) { *a = u01f(r.c); *b = u01f(r.d); }
    else { *a = u01f(r.a); *b = u01f(r.b); }
  }
};
template <> struct Draws<double> {
  // blocks 0, 1: three cell offsets and the quantile (two words per deviate);
  // blocks 2..33: one direction pair each
  static constexpr int kPairs = 1;
  static constexpr uint32_t kQuantBlock = 1;
  template <class S>
  static __device__ __forceinline__ void position(const S& s, uint32_t c, uint32_t j, double f[3], double* uq) {
    U4 r = draw(s, c, j, 0u), q = draw(s, c, j, 1u);
    f[0] = u01d(r.a, r.b); f[1] = u01d(r.c, r.d); f[2] = u01d(q.a, q.b); *uq = u01d(q.c, q.d);
  }
  using Block = U4;
  static __device__ __forceinline__ bool first_of_block(int) { return true; }
  template <class S>
  static __device__ __forceinline__ U4 block(const S& s, uint32_t c, uint32_t j, int t) {
    return draw(s, c, j, 2u + (uint32_t)t);
  }
  static __device__ __forceinline__ void pair_from(const U4& r, int, double* a, double* b) {
    *a = u01d(r.a, r.b); *b = u01d(r.c, r.d);
  }
};

// ---- allocation -------------------------------------------------------------------
// Velocity components for the compact copy (rec_velq.cuh), which the march's bound
// uses.  Binary64: bits moved to binary32 without the binary64 pipe, toward
// zero for the copy and one unit up for the maxima; the ends of binary32's
// range map to its smallest normal number and to infinity.
__device__ __forceinline__ float velq_value(float v) { return v; }
__device__ __forceinline__ float velq_upper(float v) { return fabsf(v); }
__device__ __forceinline__ uint32_t velq_abs_bits(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v) & 0x7fffffffu;
  if (hi >= 0x47e00000u) return 0x7f800000u;
  if (hi < 0x38100000u) return 0x00800000u;
  return __funnelshift_l((uint32_t)__double2loint(v), hi, 3) + 0x40000000u;
}
__device__ __forceinline__ float velq_value(double v) {
  return __uint_as_float(velq_abs_bits(v) | ((uint32_t)__double2hiint(v) & 0x80000000u));
}
__device__ __forceinline__ float velq_upper(double v) { return __uint_as_float(velq_abs_bits(v) + 1u); }

// Largest |component| and squared speed of a velocity vector, running maxima, and the
// sum of |component| over the cells that are finite.
struct VelMax {
  float u = 0.0f, v2 = 0.0f, sum = 0.0f;
  int bad = 0;
  template <class V>
  __device__ __forceinline__ void add(const V& U) {
    const float x = velq_upper(U.x), y = velq_upper(U.y), z = velq_upper(U.z);
    const bool fin = x < 3e38f && y < 3e38f && z < 3e38f;
    bad |= !fin;
    sum += fin ? x + y + z : 0.0f;
    u = fmaxf(u, fmaxf(x, fmaxf(y, z)));
    v2 = fmaxf(v2, x * x + y * y + z * z);
  }
};
// Bits of a non-negative number; as unsigned integers they order like the numbers.
__device__ __forceinline__ uint64_t order_bits(float v) { return __float_as_uint(v) & 0x7fffffffu; }
__device__ __forceinline__ uint64_t order_bits(double v) {
  return (uint64_t)__double_as_longlong(v) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ float from_order_bits(uint64_t b, float) { return __uint_as_float((uint32_t)b); }
__device__ __forceinline__ double from_order_bits(uint64_t b, double) { return __longlong_as_double((long long)b); }

// Largest weight and velocity of a block into the box's running maxima: warp
// maxima by integer reductions of the ordered bits (a maximum in binary64 would go
// through the slow pipe five times per value), one atomic maximum per block and value.
// bad: bit 0 an invalid weight, bit 1 a velocity that is not finite.
template <int NTH>
__device__ __forceinline__ void block_maxima(DevScalars* sc, uint64_t w, const VelMax& vm, bool bad) {
  __shared__ uint32_t sm[NTH / 32][5];
  __shared__ float part[NTH / 32];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto max64 = [&](uint32_t hi, uint32_t lo, uint32_t* h, uint32_t* l) {
    *h = __reduce_max_sync(full, hi);
    *l = __reduce_max_sync(full, hi == *h ? lo : 0u);
  };
  uint32_t h, l;
  max64((uint32_t)(w >> 32), (uint32_t)w, &h, &l);
  const uint32_t u = __reduce_max_sync(full, __float_as_uint(vm.u));
  const uint32_t v2 = __reduce_max_sync(full, __float_as_uint(vm.v2));
  const uint32_t b = __reduce_or_sync(full, (bad ? 1u : 0u) | (vm.bad ? 2u : 0u));
  float sum = vm.sum;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(full, sum, o);
  __syncthreads();  // sm may still be read by a previous call
  if (lane == 0) { sm[warp][0] = h; sm[warp][1] = l; sm[warp][2] = u; sm[warp][3] = v2; sm[warp][4] = b; part[warp] = sum; }
  __syncthreads();
  if (warp == 0) {
    const bool in = lane < NTH / 32;
    max64(in ? sm[lane][0] : 0u, in ? sm[lane][1] : 0u, &h, &l);
    const uint32_t bu = __reduce_max_sync(full, in ? sm[lane][2] : 0u);
    const uint32_t bv = __reduce_max_sync(full, in ? sm[lane][3] : 0u);
    const uint32_t bb = __reduce_or_sync(full, in ? sm[lane][4] : 0u);
    if (lane == 0) {
      for (int w = 1; w < NTH / 32; ++w) sum += part[w];
      atomicAdd(&sc->mx_sum, sum);  // in any order: the scale of the copy changes no result
      atomicMax(&sc->mx_w, ((unsigned long long)h << 32) | l);
      atomicMax(&sc->mx_u, bu);
      atomicMax(&sc->mx_v2, bv);
      if (bb) atomicOr(&sc->mx_bad, bb);
    }
  }
}
// The box's maxima once every block has added its own (one thread); ready for the next call.
template <class R>
__device__ __forceinline__ void take_maxima(DevScalars* sc, int64_t n3, float kappa) {
  const uint32_t bad = __ldcg(&sc->mx_bad);
  const unsigned long long w = __ldcg(&sc->mx_w);
  const float umax = __uint_as_float(__ldcg(&sc->mx_u)), v2 = __uint_as_float(__ldcg(&sc->mx_v2));
  const float u = velq_scale(umax, __ldcg(&sc->mx_sum) / (3.0f * (float)n3), kappa);
  sc->rmax = bad & 1u ? 0.0 : (double)from_order_bits(w, (R)0);  // invalid weights: emit nothing
  sc->flags = (sc->flags & ~(2 | 4 | 16)) | (bad & 1u ? 4 : 0);  // transport flags describe this call only
  sc->vq_u = u;
  sc->vq_v = bad & 2u ? __int_as_float(0x7f800000) : sqrtf(v2) * 1.00001f;
  sc->vq_out = (bad & 2u) || umax > u;
  sc->vel_plain = !(bad & 2u) && umax < 1e15f;
  sc->mx_sum = 0.0f;
  sc->mx_w = 0;
  sc->mx_u = sc->mx_v2 = sc->mx_bad = 0;
}

// Reads the emission weights once (their maximum, exact in the working precision)
// and the velocities once (the scale of their compact copy); clears the bucket capacities.
template <class R>
__global__ void __launch_bounds__(kPassThreads) k_alloc_max(const R* emis, const typename Vec4<R>::T* vel, int64_t n3,
                                                            float kappa, DevScalars* sc, unsigned long long* bcap,
                                                            int nb) {
  R m = (R)0;
  bool bad = false;
  VelMax vm;
  for (int i = blockIdx.x * kPassThreads + threadIdx.x; i < nb; i += gridDim.x * kPassThreads) bcap[i] = 0ull;
#pragma unroll 4
  for (int64_t i = (int64_t)blockIdx.x * kPassThreads + threadIdx.x; i < n3; i += (int64_t)gridDim.x * kPassThreads) {
    const R r = emis[i];
    if (!(r >= (R)0) || isinf(r)) bad = true;
    else m = m < r ? r : m;
    vm.add(vel[i]);
  }
  block_maxima<kPassThreads>(sc, order_bits(m), vm, bad);
  if (!last_block_done(&sc->counter)) return;
  if (threadIdx.x == 0) {
    take_maxima<R>(sc, n3, kappa);
    sc->counter = 0;
  }
}

template <class R>
__device__ __forceinline__ uint64_t quantised(R r, R rmax) {
  // Q = floor(2^31 r / r_max), the ratio rounded once in the working precision.
  // Q <= 2^31 fits 32 bits: the 32-bit truncation gives the same integer as a
  // 64-bit one without the 64-bit conversion (a binary64-pipe instruction).
  return (uint64_t)(uint32_t)Ar<R>::mul(Ar<R>::div(r, rmax), (R)2147483648.0);
}

// The FP64 form keeps Q (at most 2^31) in the prefix array between its two passes: a
// binary64 quotient per cell costs 16 us of the slow pipe per 1e6 cells.
template <class R> constexpr bool kKeepQ = sizeof(R) == 8;

// Inclusive block scan of 64-bit counts (thread order); returns the block total.
__device__ __forceinline__ uint64_t block_scan_incl(uint64_t v, uint64_t* incl) {
  __shared__ uint64_t wsum[AT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    uint64_t t = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += t;
  }
  __syncthreads();
  if (lane == 31) wsum[warp] = v;
  __syncthreads();
  uint64_t before = 0, total = 0;
  for (int w = 0; w < AT / 32; ++w) {
    uint64_t s = wsum[w];
    if (w < warp) before += s;
    total += s;
  }
  *incl = v + before;
  return total;
}

// Super-tiles of 2^tlg cells per side group the march queue: packets are queued in
// the bucket of their home super-tile, and the march takes the buckets in
// order, so the rays in flight at any time start in a compact region.

// Cell coordinates: shifts and masks for power-of-two sides, otherwise the
// quotients by n and n^2 from 64-bit multiply-high with precomputed
// multipliers ceil(2^64 / d), exact for every 32-bit dividend (Lemire, Kaser &
// Kurz 2019, "Faster remainder by direct computation").
struct Tiles {
  uint32_t n, nt, lg;  // box side, super-tiles per axis, log2 n (power-of-two sides)
  uint64_t mn, mn2;    // multipliers for the division by n and by n^2 (unused when n = 1: cell = 0)
  uint32_t tlg;        // log2 of the super-tile side
  template <bool P2>
  __device__ __forceinline__ void coords(uint32_t cell, uint32_t* ix, uint32_t* iy, uint32_t* iz) const {
    if (P2) {
      const uint32_t m = n - 1u;
      *ix = cell & m; *iy = (cell >> lg) & m; *iz = cell >> (2u * lg);
    } else {
      const uint32_t q = (uint32_t)__umul64hi(mn, (uint64_t)cell);   // cell / n
      const uint32_t z = (uint32_t)__umul64hi(mn2, (uint64_t)cell);  // cell / n^2
      *ix = cell - q * n; *iy = q - z * n; *iz = z;
    }
  }
  template <bool P2>
  __device__ __forceinline__ uint32_t at(uint32_t cell) const {
    uint32_t ix, iy, iz;
    coords<P2>(cell, &ix, &iy, &iz);
    return tile_of(ix, iy, iz);
  }
  __device__ __forceinline__ uint32_t tile_of(uint32_t ix, uint32_t iy, uint32_t iz) const {
    return ((iz >> tlg) * nt + (iy >> tlg)) * nt + (ix >> tlg);
  }
  // lg = 0: no power of two (or one cell, which the divisions take as well)
  __device__ __forceinline__ uint32_t of(uint32_t cell) const { return lg ? at<true>(cell) : at<false>(cell); }
};

// Multiplier ceil(2^64 / d) of the exact 32-bit division by d >= 2.
inline uint64_t fastdiv_multiplier(uint64_t d) { return d >= 2 ? UINT64_MAX / d + 1 : 0; }
inline uint32_t log2_of(uint32_t v) {
  uint32_t l = 0;
  while ((1u << l) < v) ++l;
  return l;
}
inline Tiles make_tiles(int n, int tile) {
  Tiles t;
  t.n = (uint32_t)n;
  t.tlg = log2_of((uint32_t)tile);
  t.nt = (uint32_t)((n + tile - 1) / tile);
  t.lg = 0;
  if ((n & (n - 1)) == 0)
    while ((1 << t.lg) < n) ++t.lg;
  t.mn = fastdiv_multiplier((uint64_t)n);
  t.mn2 = fastdiv_multiplier((uint64_t)n * (uint64_t)n);
  return t;
}

// The sum S > 0 of the weights as a divisor, prepared once per call: its
// normalised form d = S 2^shift (top bit set) with the reciprocal word
// v = floor((2^128 - 1) / d) - 2^64 of Moeller & Granlund, "Improved division by
// invariant integers" (IEEE Trans. Comput. 60, 165 (2011)), and m = floor((2^64 - 1) / S).
__device__ __forceinline__ void set_divisor(DevScalars* sc, uint64_t S) {
  sc->sumQ = S;
  if (S == 0) return;
  const int k = __clzll((long long)S);
  const uint64_t d = S << k;
  // v = floor((2^128 - 1 - 2^64 d) / d): long division of (2^64 - 1 - d) 2^64 + (2^64 - 1) by d, bit by bit
  uint64_t r = ~0ull - d, v = 0;
  for (int i = 0; i < 64; ++i) {
    const uint64_t top = r >> 63;
    r = (r << 1) | 1ull;
    v <<= 1;
    if (top || r >= d) { r -= d; v |= 1ull; }
  }
  sc->div_shift = k;
  sc->div_v = v;
  sc->div_m = ~0ull / S;
}
struct Divisor {
  uint64_t S, v, m;
  int shift;
};

// floor((N * pre + u) / S) and the remainder, for N < 2^32, pre <= S < 2^63, u < S:
// their algorithm 4 (two words by one) in integers.
__device__ __forceinline__ uint32_t sys_floor(uint64_t N, uint64_t pre, uint64_t u, const Divisor& dv, uint64_t* rem) {
  uint64_t lo = N * pre, hi = __umul64hi(N, pre);
  lo += u;
  hi += lo < u;
  const int k = dv.shift;  // >= 1: S < 2^63
  const uint64_t d = dv.S << k, u1 = (hi << k) | (lo >> (64 - k)), u0 = lo << k;
  uint64_t q0 = dv.v * u1, q1 = __umul64hi(dv.v, u1);
  q0 += u0;
  q1 += u1 + (q0 < u0) + 1ull;
  uint64_t r = u0 - q1 * d;
  if (r > q0) { --q1; r += d; }
  if (r >= d) { ++q1; r -= d; }
  *rem = r >> k;
  return (uint32_t)q1;
}

// Compact copy of the velocities of AT * IT consecutive cells (one block).
template <class R, int IT, class V>
__device__ __forceinline__ void velq_write(const V* vel, int64_t n3, int64_t c0, float u, uint32_t* velq, uint32_t bx,
                                           const Tiles& tl) {
  if (!velq || !(u > 0.0f)) return;
  const float qs = 127.0f / u;
#pragma unroll 4
  for (int k = 0; k < IT; ++k) {
    const int64_t i = c0 + (int64_t)k * AT + threadIdx.x;
    if (i >= n3) break;
    const V U = vel[i];
    uint32_t ix, iy, iz;
    if (tl.lg) tl.template coords<true>((uint32_t)i, &ix, &iy, &iz);
    else tl.template coords<false>((uint32_t)i, &ix, &iy, &iz);
    const bool in = velq_upper(U.x) <= u && velq_upper(U.y) <= u && velq_upper(U.z) <= u;
    velq[velq_x(ix) | velq_y(iy, bx) | velq_z(iz, bx)] =
        in ? velq_pack(velq_value(U.x), velq_value(U.y), velq_value(U.z), qs) : kVelqOut;
  }
}

// The allocation kernels give each thread IT consecutive cells.
template <class R, int IT>
__device__ __forceinline__ void load_items(const R* p, int64_t c0, int64_t n3, R (&v)[IT]) {
  if (IT >= 4 && c0 + IT <= n3 && (reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
    if (sizeof(R) == 4) {
      const float4* q = reinterpret_cast<const float4*>(p + c0);
#pragma unroll
      for (int k = 0; k < IT / 4; ++k) {
        float4 t = q[k];
        v[4 * k] = (R)t.x; v[4 * k + 1] = (R)t.y; v[4 * k + 2] = (R)t.z; v[4 * k + 3] = (R)t.w;
      }
    } else {
      const double2* q = reinterpret_cast<const double2*>(p + c0);
#pragma unroll
      for (int k = 0; k < IT / 2; ++k) {
        double2 t = q[k];
        v[2 * k] = (R)t.x; v[2 * k + 1] = (R)t.y;
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < IT; ++k) v[k] = (c0 + k < n3) ? p[c0 + k] : (R)0;
  }
}

template <class R, int IT>
__global__ void __launch_bounds__(AT) k_alloc_sum(const R* emis, const typename Vec4<R>::T* vel, int64_t n3,
                                                  uint64_t n_packets, Stream strm, DevScalars* sc,
                                                  unsigned long long* partQ, uint32_t* P, uint32_t* velq, uint32_t vbx,
                                                  Tiles tl) {
  const R rmax = (R)sc->rmax;
  velq_write<R, IT>(vel, n3, (int64_t)blockIdx.x * (AT * IT), sc->vq_u, velq, vbx, tl);
  uint64_t acc = 0;
  if (rmax > (R)0) {
    R v[IT];
    const int64_t c0 = (int64_t)blockIdx.x * (AT * IT) + (int64_t)threadIdx.x * IT;
    load_items<R, IT>(emis, c0, n3, v);
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const uint64_t q = quantised<R>(v[k], rmax);
      acc += q;
      if (kKeepQ<R> && c0 + k < n3) P[c0 + k] = (uint32_t)q;
    }
  }
  uint64_t incl;
  uint64_t tot = block_scan_incl(acc, &incl);
  if (threadIdx.x == 0) partQ[blockIdx.x] = tot;
  if (!last_block_done(&sc->alloc_counter)) return;
  // exclusive scan of the block sums, in block order
  const int nb = gridDim.x;
  const int per = (nb + AT - 1) / AT;
  uint64_t seg = 0;
  for (int b = threadIdx.x * per; b < min(nb, (threadIdx.x + 1) * per); ++b) seg += __ldcg(&partQ[b]);
  uint64_t sincl;
  uint64_t sumQ = block_scan_incl(seg, &sincl);
  uint64_t run = sincl - seg;
  for (int b = threadIdx.x * per; b < min(nb, (threadIdx.x + 1) * per); ++b) {
    uint64_t q = __ldcg(&partQ[b]);
    partQ[b] = run;
    run += q;
  }
  if (threadIdx.x == 0) {
    U4 r = draw(strm, 0u, 0u, kAllocBlock);
    uint64_t w = ((uint64_t)r.b << 32) | r.a;
    uint64_t npk = (sumQ > 0) ? n_packets : 0;
    set_divisor(sc, sumQ);
    sc->alloc_u = sumQ > 0 ? w % sumQ : 0;
    P[n3] = (uint32_t)npk;
    sc->emitted = npk;
    sc->absorbed = 0;
    sc->capped = 0;
    sc->crossings = 0;
    sc->qtail = 0;
    sc->alloc_counter = 0;
    if (sumQ == 0 && n_packets > 0) sc->flags |= 4;
  }
}

// floor(t / S) and t mod S for t < 2^64, given m = floor((2^64 - 1) / S): the
// multiply-high estimate is short by at most 2, then corrected exactly
// (replaces a 64-bit division per cell).
__device__ __forceinline__ uint64_t div_small(uint64_t t, uint64_t S, uint64_t m, uint64_t* r) {
  uint64_t q = __umul64hi(t, m);
  uint64_t rr = t - q * S;
#pragma unroll
  for (int i = 0; i < 3; ++i)
    if (rr >= S) { ++q; rr -= S; }
  *r = rr;
  return q;
}

// Packet prefix P_i = floor((N prefixQ_i + u) / S) of the thread's consecutive
// cells: one 128-bit division for the first, then exact 64-bit remainder
// updates, (R + N Q_i) / S.  The same pass writes the coarse index first[w] =
// cell of packet 32 w (each cell writes the multiples of 32 in its packet
// range, so a warp of 32 consecutive packets finds its first cell with one
// load) and the packets per super-tile (the capacity of its march-queue bucket).
template <class R, int IT>
__device__ __forceinline__ void alloc_prefix_block(const R* emis, int64_t n3, uint64_t n_packets, const Divisor& dv,
                                                   uint64_t u, R rmax, uint64_t pre_block, int64_t c0, uint32_t* P,
                                                   uint32_t* first, const Tiles& tl, uint32_t bk0,
                                                   unsigned long long* bcap) {
  const uint64_t S = dv.S;
  uint64_t Q[IT];
  uint64_t acc = 0;
  if (kKeepQ<R>) {  // left in P by the pass before
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      Q[k] = (rmax > (R)0 && c0 + k < n3) ? __ldcg(P + c0 + k) : 0u;
      acc += Q[k];
    }
  } else {
    R v[IT];
    load_items<R, IT>(emis, c0, n3, v);
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      Q[k] = (rmax > (R)0 && c0 + k < n3) ? quantised<R>(v[k], rmax) : 0;
      acc += Q[k];
    }
  }
  uint64_t incl;
  block_scan_incl(acc, &incl);
  uint32_t out[IT];
  uint32_t bk = 0xffffffffu, bcount = 0;  // packets of the thread's last super-tile
  if (S == 0) {
#pragma unroll
    for (int k = 0; k < IT; ++k) out[k] = 0u;
  } else {
    uint64_t rem;
    uint32_t pk = sys_floor(n_packets, pre_block + incl - acc, u, dv, &rem);
    const uint64_t minv = dv.m;
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      out[k] = pk;
      const uint64_t t = rem + n_packets * Q[k];  // < S + 2^63 <= 2^64
      const uint64_t dq = div_small(t, S, minv, &rem);
      const uint32_t p1 = pk + (uint32_t)dq;
      if (p1 > pk && c0 + k < n3) {
        for (uint32_t w = (pk + 31u) >> 5; 32ull * w < p1; ++w) first[w] = (uint32_t)(c0 + k);
        const uint32_t b = bk0 + tl.of((uint32_t)(c0 + k));
        if (b != bk) {
          if (bcount) atomicAdd(&bcap[bk], (unsigned long long)bcount);
          bk = b;
          bcount = 0;
        }
        bcount += p1 - pk;
      }
      pk = p1;
    }
  }
  // the lanes of a warp are mostly in one super-tile: one addition per warp and super-tile
  const unsigned same = __match_any_sync(0xffffffffu, bk);
  const uint32_t sum = __reduce_add_sync(same, bcount);
  if (sum && (int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&bcap[bk], (unsigned long long)sum);
  if (c0 >= n3) return;
  if (IT >= 4 && c0 + IT <= n3 && (reinterpret_cast<uintptr_t>(P + c0) & 15u) == 0) {
    uint4* q = reinterpret_cast<uint4*>(P + c0);
#pragma unroll
    for (int k = 0; k < IT / 4; ++k) q[k] = make_uint4(out[4 * k], out[4 * k + 1], out[4 * k + 2], out[4 * k + 3]);
  } else {
#pragma unroll
    for (int k = 0; k < IT; ++k)
      if (c0 + k < n3) P[c0 + k] = out[k];
  }
}

// Exclusive prefix of one value per thread over the block (thread order); the total in *total.
template <int NTH>
__device__ __forceinline__ unsigned long long block_prefix(unsigned long long v, unsigned long long* total) {
  __shared__ unsigned long long warp_sum[NTH / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();  // warp_sum may still be read by a previous call
  if (lane == 31) warp_sum[warp] = incl;
  __syncthreads();
  unsigned long long before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < NTH / 32; ++w) {
    const unsigned long long t = warp_sum[w];
    if (w < warp) before += t;
    all += t;
  }
  *total = all;
  return before + incl - v;
}

// One block: bucket capacities -> offsets (in place); fill counters cleared.
template <int NTH>
__device__ __forceinline__ void bucket_offsets_block(unsigned long long* bcap, unsigned long long* bfill, int nb) {
  const int per = (nb + NTH - 1) / NTH;
  unsigned long long s = 0, total;
  for (int b = threadIdx.x * per; b < min(nb, (int)(threadIdx.x + 1) * per); ++b) s += __ldcg(&bcap[b]);
  unsigned long long run = block_prefix<NTH>(s, &total);
  for (int b = threadIdx.x * per; b < min(nb, (int)(threadIdx.x + 1) * per); ++b) {
    unsigned long long v = __ldcg(&bcap[b]);
    bcap[b] = run;
    run += v;
    bfill[b] = 0;
  }
}

// One block: the march works through the queue in chunks of `chunk` packets
// that never straddle a bucket; cpre[b] = first chunk of bucket b, cpre[nb] =
// all chunks.  Also the total queued.
template <int NTH>
__device__ __forceinline__ void bucket_scan_block(const unsigned long long* bfill, unsigned long long* cpre, int nb,
                                                  DevScalars* sc, uint32_t chunk) {
  const int per = (nb + NTH - 1) / NTH;
  unsigned long long s = 0, q = 0, chunks, queued;
  for (int b = threadIdx.x * per; b < min(nb, (int)(threadIdx.x + 1) * per); ++b) {
    const unsigned long long f = __ldcg(&bfill[b]);
    s += (f + chunk - 1) / chunk;
    q += f;
  }
  unsigned long long run = block_prefix<NTH>(s, &chunks);
  block_prefix<NTH>(q, &queued);
  if (threadIdx.x == 0) {
    cpre[nb] = chunks;
    sc->qtail = queued;
    sc->march_next = 0;
    sc->requeued = 0;
  }
  for (int b = threadIdx.x * per; b < min(nb, (int)(threadIdx.x + 1) * per); ++b) {
    cpre[b] = run;
    run += (__ldcg(&bfill[b]) + chunk - 1) / chunk;
  }
}
// The last block to finish turns the bucket capacities into offsets.
template <class R, int IT>
__global__ void __launch_bounds__(AT, 3) k_alloc_prefix(const R* emis, int64_t n3, uint64_t n_packets, DevScalars* sc,
                                                     const unsigned long long* partQ, uint32_t* P, uint32_t* first,
                                                     Tiles tl, unsigned long long* bcap, unsigned long long* bfill,
                                                     int nb) {
  const int64_t c0 = (int64_t)blockIdx.x * (AT * IT) + (int64_t)threadIdx.x * IT;
  alloc_prefix_block<R, IT>(emis, n3, n_packets, Divisor{sc->sumQ, sc->div_v, sc->div_m, sc->div_shift}, sc->alloc_u,
                            (R)sc->rmax, partQ[blockIdx.x], c0, P, first, tl, 0u, bcap);
  if (!last_block_done(&sc->alloc_counter)) return;
  bucket_offsets_block<AT>(bcap, bfill, nb);
  if (threadIdx.x == 0) sc->alloc_counter = 0;
}

// The launches of their own of a batch without the persistent front.
__global__ void __launch_bounds__(1024) k_bucket_offsets(unsigned long long* bcap, unsigned long long* bfill, int nb) {
  bucket_offsets_block<1024>(bcap, bfill, nb);
}
__global__ void __launch_bounds__(1024) k_bucket_scan(const unsigned long long* bfill, unsigned long long* cpre, int nb,
                                                      DevScalars* sc, uint32_t chunk) {
  bucket_scan_block<1024>(bfill, cpre, nb, sc, chunk);
}

// ---- transport ----------------------------------------------------------------------
// A queued packet: the march state right after it left its home cell.
// Binary32 form (two float4):
//   q0 = {cell bits, tMax_x, tMax_y, tMax_z},  q1 = {n_x, n_y, n_z, u0};
// the march recomputes tDelta = 1/|n| and kappa n with the same rounded
// operations as the emission, so it continues bit for bit.
// Binary64 form (three double4): q0 as above, q1 = {tDelta (sign = step
// direction), u0}, q2 = {kappa n, -}: recomputing them would cost three
// correctly rounded binary64 reciprocals per packet on the slow binary64 pipe.
template <class R> struct QueueVecs { static constexpr int value = sizeof(R) == 4 ? 2 : 3; };
template <class R>
struct TransportArgs {
  const uint32_t* P;
  const uint32_t* first;  // cell of packet 32 w
  int64_t n3;
  int n;
  const typename Vec4<R>::T* vel;
  const R* T;
  const R* quant;
  int M;
  R kappa, cth;
  Keys ks;  // round keys of the step's stream (emission)
  uint32_t early;  // packets whose quantile word is below it have xi <= 0 (early_word)
  uint32_t* tally;
  DevScalars* sc;
  typename Vec4<R>::T* queue;  // QueueVecs entries per queued packet (3 where a sweep resumes)
  Tiles tl;
  int nb;                          // buckets (super-tiles)
  unsigned long long* boff;        // bucket start in the queue (capacity prefix)
  unsigned long long* bfill;       // packets queued per bucket
  unsigned long long* cpre;        // first march chunk of each bucket [nb + 1]
  uint32_t chunk;                  // queued packets per march chunk
  int refill;                      // idle lanes of a warp that trigger a refill
  // region sweeps (single box, power-of-two side)
  typename Vec4<R>::T* rq;         // second queue: full traversal states, 3 vectors per entry
  unsigned long long* rcount;      // entries per bucket appended to the second queue
  unsigned long long* rqn;         // entries appended per part of the second queue [kRqParts]
  uint64_t rq_part;                // entries one part holds
  uint32_t halo;                   // region of a bucket: its super-tile and halo cells around it; 0: no limit
  int closes;                      // this march is the call's last
  int resumed;                     // the queue holds full states of an earlier sweep (3 vectors per entry)
  // compact velocity copy (rec_velq.cuh) and its index masks
  const uint32_t* velq;
  VelqMasks vm;
  uint32_t vbx;
};

// Loads of the packet prefix and coarse index: the read-only path, or through
// L2 (FRESH) when they were written earlier in the same launch.
template <bool FRESH>
__device__ __forceinline__ uint32_t ld_index(const uint32_t* p) {
  return FRESH ? __ldcg(p) : __ldg(p);
}

// First index k in [lo, hi] with P[k] > key (P[hi] > key holds).
template <bool FRESH = false>
__device__ __forceinline__ uint32_t upper_bound(const uint32_t* P, uint32_t lo, uint32_t hi, uint32_t key) {
  while (lo < hi) {
    uint32_t mid = lo + ((hi - lo) >> 1);
    if (ld_index<FRESH>(P + mid) > key) hi = mid;
    else lo = mid + 1;
  }
  return lo;
}

template <class R> __device__ __forceinline__ R bits_to(uint32_t v);
template <> __device__ __forceinline__ float bits_to<float>(uint32_t v) { return __uint_as_float(v); }
template <> __device__ __forceinline__ double bits_to<double>(uint32_t v) { return __longlong_as_double((long long)v); }
template <class R> __device__ __forceinline__ uint32_t to_bits(R v);
template <> __device__ __forceinline__ uint32_t to_bits<float>(float v) { return __float_as_uint(v); }
template <> __device__ __forceinline__ uint32_t to_bits<double>(double v) { return (uint32_t)__double_as_longlong(v); }

// Lower table node of the frequency quantile: k = min(trunc(tq), M - 2) (0 <= tq
// < M - 1) and k as a value of R.  Binary32: adding 2^23 rounded toward zero
// leaves 2^23 + trunc(tq) exactly, whose bits give k without a conversion.
template <class R>
__device__ __forceinline__ R quant_node(R tq, int M, int* k) {
  int kk = Ar<R>::trunc(tq);
  if (kk > M - 2) kk = M - 2;
  *k = kk;
  return (R)kk;
}
template <>
__device__ __forceinline__ float quant_node<float>(float tq, int M, int* k) {
  const float t = __fadd_rz(tq, 0x1p23f);
  int kk = __float_as_int(t) - 0x4b000000;
  float kf = __fsub_rn(t, 0x1p23f);
  if (kk > M - 2) { kk = M - 2; kf = (float)(M - 2); }
  *k = kk;
  return kf;
}

// Traversal state of one packet.
template <class R>
struct Ray {
  uint32_t ix, iy, iz, kc;
  R tMx, tMy, tMz, tDx, tDy, tDz, knx, kny, knz, u0;
  int sx, sy, sz;
};

__device__ __forceinline__ int step_sign(float v) { return (v > 0.0f) - (v < 0.0f); }
__device__ __forceinline__ int step_sign(double v) {  // by the bits
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  return ((hi & 0x7fffffffu) | lo) == 0u ? 0 : ((int)hi < 0 ? -1 : 1);
}

// tDelta and step of one axis from the direction cosine (Amanatides-Woo).
template <class R>
// Written without branches: 1/|n_d| correctly rounded (the same value as the
// division 1/|n_d|) is +inf for n_d = 0, which is the tDelta of an axis never
// crossed.
__device__ __forceinline__ void axis_setup(R nd, R* tD, int* st) {
  using A = Ar<R>;
  *st = step_sign(nd);
  *tD = A::rcp(fabs(nd));
}

// One cell of the march: resonance test in the current cell, then a step
// across the nearest face (ties x < y < z, periodic wrap).  Returns 1 when
// absorbed in the current cell, 2 when the crossing cap is hit, 0 otherwise.
// The step is written with selects rather than branches so that the lanes of
// a warp stepping along different axes do not serialise.
// Periodic neighbour index along one axis; a mask when the side is a power of two.
template <bool P2>
__device__ __forceinline__ uint32_t wrap_step(uint32_t i, int s, uint32_t n) {
  if (P2) return (i + (uint32_t)s) & (n - 1u);
  return s > 0 ? (i + 1 == n ? 0 : i + 1) : (i == 0 ? n - 1 : i - 1);
}

// Order of two positive numbers or +inf; binary64 by the bits, off the binary64 pipe.
__device__ __forceinline__ bool le_pos(float a, float b) { return a <= b; }
__device__ __forceinline__ bool le_pos(double a, double b) { return __double_as_longlong(a) <= __double_as_longlong(b); }

// Path length along the ray at which the packet leaves its current cell: the
// nearest face, ties broken x < y < z.
template <class R>
__device__ __forceinline__ R dda_exit(const Ray<R>& r, bool* ax0, bool* ax1, bool* ax2) {
  *ax0 = le_pos(r.tMx, r.tMy) && le_pos(r.tMx, r.tMz);
  *ax1 = !*ax0 && le_pos(r.tMy, r.tMz);
  *ax2 = !*ax0 && !*ax1;
  return *ax0 ? r.tMx : (*ax1 ? r.tMy : r.tMz);
}

// Gas-frame resonance distance offset kappa n.U_c of a cell.
template <class R, class V>
__device__ __forceinline__ R doppler(const Ray<R>& r, const V& U) {
  using A = Ar<R>;
  return A::add(A::add(A::mul(r.knx, U.x), A::mul(r.kny, U.y)), A::mul(r.knz, U.z));
}

// The step across the exit face: periodic neighbour along the exit axis and
// its next face distance.
template <class R, bool P2>
__device__ __forceinline__ void dda_advance(Ray<R>& r, bool ax0, bool ax1, bool ax2, R s_exit, uint32_t n) {
  using A = Ar<R>;
  const uint32_t wx = wrap_step<P2>(r.ix, r.sx, n);
  const uint32_t wy = wrap_step<P2>(r.iy, r.sy, n);
  const uint32_t wz = wrap_step<P2>(r.iz, r.sz, n);
  r.ix = ax0 ? wx : r.ix;
  r.iy = ax1 ? wy : r.iy;
  r.iz = ax2 ? wz : r.iz;
  const R tD = ax0 ? r.tDx : (ax1 ? r.tDy : r.tDz);
  const R tn = A::add(s_exit, tD);
  r.tMx = ax0 ? tn : r.tMx;
  r.tMy = ax1 ? tn : r.tMy;
  r.tMz = ax2 ? tn : r.tMz;
  ++r.kc;
}

__device__ __forceinline__ void add_counters(DevScalars* sc, uint64_t ab, uint64_t cap, uint64_t cross) {
  __shared__ unsigned long long s_abs, s_cap, s_cross;
  if (threadIdx.x == 0) { s_abs = 0; s_cap = 0; s_cross = 0; }
  __syncthreads();
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    ab += __shfl_down_sync(0xffffffffu, ab, off);
    cap += __shfl_down_sync(0xffffffffu, cap, off);
    cross += __shfl_down_sync(0xffffffffu, cross, off);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&s_abs, (unsigned long long)ab);
    atomicAdd(&s_cap, (unsigned long long)cap);
    atomicAdd(&s_cross, (unsigned long long)cross);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_abs) atomicAdd(&sc->absorbed, s_abs);
    if (s_cap) atomicAdd(&sc->capped, s_cap);
    if (s_cross) atomicAdd(&sc->crossings, s_cross);
  }
}

// Batched contexts: per-box event counters of one block in shared memory
// (absorbed, capped, crossings), added to the boxes' scalars at the block's end.
struct BoxCounters {
  unsigned long long v[3][kMaxBoxes];
};
__device__ __forceinline__ void box_counters_clear(BoxCounters& c, int B) {
  for (int i = threadIdx.x; i < 3 * kMaxBoxes; i += blockDim.x) c.v[i / kMaxBoxes][i % kMaxBoxes] = 0ull;
  __syncthreads();
}
__device__ __forceinline__ void box_counters_add(BoxCounters& c, int b, uint64_t ab, uint64_t cap, uint64_t cross) {
  if (ab) atomicAdd(&c.v[0][b], (unsigned long long)ab);
  if (cap) atomicAdd(&c.v[1][b], (unsigned long long)cap);
  if (cross) atomicAdd(&c.v[2][b], (unsigned long long)cross);
}
__device__ __forceinline__ void box_counters_flush(BoxCounters& c, const BoxDev* bxs, int B) {
  __syncthreads();
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    DevScalars* sc = bxs[b].sc;
    if (c.v[0][b]) atomicAdd(&sc->absorbed, c.v[0][b]);
    if (c.v[1][b]) atomicAdd(&sc->capped, c.v[1][b]);
    if (c.v[2][b]) atomicAdd(&sc->crossings, c.v[2][b]);
  }
}

// Last index i in [0, B) with key(i) <= v (key non-decreasing, key(0) <= v).
template <class F>
__device__ __forceinline__ int last_le(int B, uint64_t v, F key) {
  int lo = 0, hi = B;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if ((uint64_t)key(mid) <= v) lo = mid;
    else hi = mid;
  }
  return lo;
}

// One box as the emission sees it: its fields, packet prefix and coarse index,
// transport scalars, random stream, super-tiles and first queue bucket.
template <class R>
struct EmitBox {
  const uint32_t* P;
  const uint32_t* first;
  uint32_t n3, n;
  const typename Vec4<R>::T* vel;
  const R* T;
  uint32_t* tally;
  R kappa, cth;
  uint32_t box;  // fourth Philox counter word
  Tiles tl;
  uint32_t bk0;
  uint32_t early;  // TransportArgs::early, or 0 where not all velocities are plain (DevScalars::vel_plain)
};

// Emission of one packet, in three parts: the cell of each of a warp's 32
// packets (warp-collective), the packet's first Philox block, frequency and
// thermal speed (per lane), and the rest (warp-collective): direction, the
// resonance test in the home cell, the home tally or the queue entry.

// Cell and index within the cell of packet base + lane (< N): the coarse index
// gives the cell c0 of the warp's first packet, and the prefix values of the 32 cells
// after it, those below base + 32, mark where in the warp a new cell begins (bit s of
// *starts for a cell that begins at packet base + s; at[s], shared memory of the
// warp, names it).  The packets of a cell are neighbouring lanes: *starts also
// groups the warp by cells, if *whole (no packet lies beyond those 32 cells).
template <class R, bool FRESH>
__device__ __forceinline__ bool emit_locate(const EmitBox<R>& e, uint32_t base, uint32_t N, uint32_t* at,
                                            uint32_t* cell_out, uint32_t* j_out, uint32_t* starts, bool* whole) {
  const int lane = threadIdx.x & 31;
  const uint32_t n3 = e.n3;
  const uint32_t p = base + lane;
  const bool act = p < N;
  const uint32_t c0 = ld_index<FRESH>(e.first + (base >> 5));
  const uint32_t Pc0 = ld_index<FRESH>(e.P + c0);
  const uint32_t widx = c0 + 1u + lane;
  const uint32_t wv = (widx <= n3) ? ld_index<FRESH>(e.P + widx) : 0xffffffffu;
  const uint32_t next = __shfl_down_sync(0xffffffffu, wv, 1);
  const uint32_t s = wv - base;  // >= 1: the warp's first packet lies in c0
  const uint32_t m = __reduce_or_sync(0xffffffffu, s < 32u ? 1u << s : 0u);
  __syncwarp();  // at is read no more
  if (s < 32u && (lane == 31 || next != wv)) at[s] = (uint32_t)lane + 1u;  // the last of the cells that begin there
  __syncwarp();
  const uint32_t mine = m & (0xffffffffu >> (31 - lane));
  const uint32_t b = 31u - (uint32_t)__clz((int)mine);  // where the packet's cell begins
  const uint32_t off = mine ? at[b & 31u] : 0u;
  uint32_t cell = c0 + off, j = mine ? (uint32_t)lane - b : p - Pc0;
  *whole = !__any_sync(0xffffffffu, act && off == 32u);
  if (act && off == 32u) {
    cell = upper_bound<FRESH>(e.P, c0 + 32u, n3, p) - 1u;
    j = p - ld_index<FRESH>(e.P + cell);
  }
  *cell_out = cell;
  *j_out = j;
  *starts = m;
  return act;
}

// Lanes of the group of neighbouring lanes that a lane belongs to, from the
// lanes where groups start (lane 0 always starts one).
__device__ __forceinline__ unsigned lane_group(uint32_t starts) {
  const int lane = threadIdx.x & 31;
  const uint32_t upto = 0xffffffffu >> (31 - lane);
  const uint32_t low = (starts | 1u) & upto, high = starts & ~upto;
  const uint32_t from = 0xffffffffu << (31 - __clz((int)low));
  return from & (high ? (high & (0u - high)) - 1u : 0xffffffffu);
}
// The same from keys: neighbouring lanes with equal keys.
__device__ __forceinline__ unsigned key_group(uint32_t key) {
  const uint32_t before = __shfl_up_sync(0xffffffffu, key, 1);
  return lane_group(__ballot_sync(0xffffffffu, key != before));
}

// (1) the emission frequency from the tabulated inverse CDF at the packet's
// quantile, and the thermal speed in cells.
template <class R>
__device__ __forceinline__ void emit_draw0(const TransportArgs<R>& a, const EmitBox<R>& e, uint32_t cell, R uq, R* xi,
                                           R* vt) {
  using A = Ar<R>;
  R tq = A::mul(uq, (R)(a.M - 1));
  int k;
  const R fr = A::sub(tq, quant_node<R>(tq, a.M, &k));
  R q0 = __ldg(a.quant + k), q1 = __ldg(a.quant + k + 1);
  *xi = A::add(q0, A::mul(fr, A::sub(q1, q0)));
  *vt = A::sqr(A::mul(__ldg(e.T + cell), e.cth));
}

// 2 u - 1 (2 u is exact, so one rounding as in the separate operations), and
// 0 < s < 1 for a sum of squares (binary64 by the bits).
__device__ __forceinline__ float centred(float u) { return __fmaf_rn(2.0f, u, -1.0f); }
__device__ __forceinline__ double centred(double u) { return __fma_rn(2.0, u, -1.0); }
__device__ __forceinline__ bool in_disk(float s) { return s < 1.0f && s > 0.0f; }
__device__ __forceinline__ bool in_disk(double s) {
  const uint64_t b = (uint64_t)__double_as_longlong(s);
  return b - 1u < 0x3ff0000000000000ull - 1u;
}

// The rest of a packet's emission (all lanes of the warp call it; lanes with
// act false take no part): isotropic direction (Philox blocks 1, 2, ...),
// u0, the Amanatides-Woo set-up and the resonance test in the home cell;
// packets resonant at home are tallied (warp-aggregated), the others take
// their first step and are queued in their home super-tile's bucket.
template <class R, bool P2>
__device__ __forceinline__ void emit_rest(const TransportArgs<R>& a, const EmitBox<R>& e, bool act, uint32_t cell,
                                          uint32_t j, const R f[3], R xi, R vt, uint64_t& my_abs,
                                          uint64_t& my_cross) {
  using A = Ar<R>;
  using V = typename Vec4<R>::T;
  const int lane = threadIdx.x & 31;
  const uint32_t n = e.n;
  const R one = (R)1, two = (R)2, zero = (R)0;
  bool home = false, queued = false;
  Ray<R> r;
  R nx = zero, ny = zero, nz = one;
  e.tl.template coords<P2>(cell, &r.ix, &r.iy, &r.iz);
  const uint32_t bk = e.bk0 + e.tl.tile_of(r.ix, r.iy, r.iz);  // bucket of the home cell
  if (act) {
    const KStream ks{a.ks, e.box};
    // isotropic direction (Marsaglia 1972): the first accepted of the candidate
    // pairs t = 0, 1, ... (each Philox block is computed once for the pairs it
    // holds).  The pairs of the first block are tested side by side; the loop
    // over later blocks runs for the few packets that reject all of them.
    {
      typename Draws<R>::Block blk = Draws<R>::block(ks, cell, j, 0);
      R ua, ub;
      Draws<R>::pair_from(blk, 0, &ua, &ub);
      R v1 = centred(ua), v2 = centred(ub);
      R s = A::add(A::mul(v1, v1), A::mul(v2, v2));
      bool ok = in_disk(s);
      int t = 1;
      if (Draws<R>::kPairs == 2) {  // the block's second pair
        Draws<R>::pair_from(blk, 1, &ua, &ub);
        const R w1 = centred(ua), w2 = centred(ub);
        const R sw = A::add(A::mul(w1, w1), A::mul(w2, w2));
        if (!ok && in_disk(sw)) { v1 = w1; v2 = w2; s = sw; ok = true; }
        t = 2;
      }
      for (; !ok && t < 32; ++t) {
        if (Draws<R>::first_of_block(t)) blk = Draws<R>::block(ks, cell, j, t);
        Draws<R>::pair_from(blk, t, &ua, &ub);
        v1 = centred(ua);
        v2 = centred(ub);
        s = A::add(A::mul(v1, v1), A::mul(v2, v2));
        ok = in_disk(s);
      }
      if (ok) {
        R fac = A::mul(two, A::sqr(A::sub(one, s)));
        nx = A::mul(v1, fac); ny = A::mul(v2, fac); nz = A::sub(one, A::mul(two, s));
      }
    }
    r.knx = A::mul(e.kappa, nx); r.kny = A::mul(e.kappa, ny); r.knz = A::mul(e.kappa, nz);
    V Uh = e.vel[cell];
    const R dh = doppler(r, Uh);
    r.u0 = A::add(A::mul(xi, vt), dh);
    axis_setup<R>(nx, &r.tDx, &r.sx);
    axis_setup<R>(ny, &r.tDy, &r.sy);
    axis_setup<R>(nz, &r.tDz, &r.sz);
    // distance to the first face along each axis (f in (0,1): an axis with
    // tDelta = inf gets tMax = inf)
    r.tMx = A::mul(r.sx < 0 ? f[0] : A::sub(one, f[0]), r.tDx);
    r.tMy = A::mul(r.sy < 0 ? f[1] : A::sub(one, f[1]), r.tDy);
    r.tMz = A::mul(r.sz < 0 ? f[2] : A::sub(one, f[2]), r.tDz);
    r.kc = 0;
    // home cell: resonance at path length u0 - kappa n.U_home, absorb unless beyond the exit
    bool ax0, ax1, ax2;
    const R s_exit = dda_exit(r, &ax0, &ax1, &ax2);
    home = A::sub(r.u0, dh) <= s_exit;
    queued = !home;
    if (home) ++my_abs;
    else {
      dda_advance<R, P2>(r, ax0, ax1, ax2, s_exit, n);
      ++my_cross;
    }
  }
  // warp-aggregated tally of the packets resonant at home (mostly one cell per warp)
  const unsigned m = key_group(cell) & __ballot_sync(0xffffffffu, home);
  if (home && lane == __ffs(m) - 1) atomicAdd(e.tally + cell, (uint32_t)__popc(m));
  // queue the others after their first step, in their home super-tile's bucket
  const unsigned qm = __ballot_sync(0xffffffffu, queued);
  if (qm) {
    const unsigned gm = key_group(bk) & qm;
    unsigned long long qb = 0;
    const int leader = __ffs(gm) - 1;
    if (queued && lane == leader) qb = atomicAdd(&a.bfill[bk], (unsigned long long)__popc(gm));
    qb = __shfl_sync(0xffffffffu, qb, leader < 0 ? 0 : leader);
    if (queued) {
      uint64_t slot = a.boff[bk] + qb + __popc(gm & ((1u << lane) - 1u));
      uint32_t c1 = P2 ? (((r.iz << e.tl.lg) | r.iy) << e.tl.lg) | r.ix : (r.iz * n + r.iy) * n + r.ix;
      constexpr int QV = QueueVecs<R>::value;
      V q0v, q1v;
      q0v.x = bits_to<R>(c1); q0v.y = r.tMx; q0v.z = r.tMy; q0v.w = r.tMz;
      if (QV == 2) {
        q1v.x = nx; q1v.y = ny; q1v.z = nz; q1v.w = r.u0;
      } else {
        q1v.x = r.sx < 0 ? -r.tDx : r.tDx; q1v.y = r.sy < 0 ? -r.tDy : r.tDy; q1v.z = r.sz < 0 ? -r.tDz : r.tDz;
        q1v.w = r.u0;
        V q2v;
        q2v.x = r.knx; q2v.y = r.kny; q2v.z = r.knz; q2v.w = zero;
        a.queue[QV * slot + 2] = q2v;
      }
      a.queue[QV * slot] = q0v;
      a.queue[QV * slot + 1] = q1v;
    }
  }
}

// A packet emitted at or below the line centre (xi <= 0) is resonant in its
// home cell whatever its direction: u0 - kappa n.U_home = (xi v_t + d) - d
// with d = kappa n.U_home is <= 0 by the monotonicity of rounding, and the
// exit distance is >= 0.  This holds exactly when xi v_t is not NaN (v_t
// finite) and d is finite; such packets need no direction and are tallied at once.
// - xi: the packet's quantile deviate u lies below a bound known to the host
//   (early_word), so the word that leads u's bits decides, without the table.
// - v_t = sqrt(T cth): T in [0, 1e15] by its bits, with cth <= 1e15 (early_word is 0 otherwise).
// - d: kappa < 1e15 (early_word is 0 otherwise) and |U| components below 1e15 km/s: the whole
//   box's (EmitBox::early), or the home cell's (256^3, 1e8 packets with one infinite cell:
//   1.73 ms of emission, 2.54 with the direction of every packet drawn, 1.65 where the box is plain).
__device__ __forceinline__ bool temperature_plain(float T) { return __float_as_uint(T) <= 0x58635fa9u; }
__device__ __forceinline__ bool temperature_plain(double T) { return (uint32_t)__double2hiint(T) < 0x430c6bf5u; }
template <class V>
__device__ __forceinline__ bool velocity_plain(const V& U) {
  return velq_upper(U.x) < 1e15f && velq_upper(U.y) < 1e15f && velq_upper(U.z) < 1e15f;
}

// Emission in 64-packet windows.  The first Philox block of every packet
// gives its frequency; the packets with xi <= 0 (about half) are absorbed at
// home without a direction.  The others wait in a per-warp ring in shared
// memory and are finished 32 at a time, so the warp's lanes stay busy in the
// costly part (direction, ray set-up, home test); leftovers carry over to the
// next window and are flushed at the end (and, in batches, at a change of box).
// A waiting binary32 packet keeps its first block's words; the binary64 form is
// bound by its arithmetic and draws its two blocks again.
constexpr uint32_t kStash = 96;  // < 32 left over + 64 new
template <class R> struct EmitStash;
template <> struct EmitStash<float> {
  uint32_t at[32];
  uint32_t cell[kStash], j[kStash], w0[kStash], w1[kStash], w2[kStash], w3[kStash];
  __device__ __forceinline__ void put(uint32_t k, uint32_t c, uint32_t jj, const U4& r) {
    cell[k] = c; j[k] = jj; w0[k] = r.a; w1[k] = r.b; w2[k] = r.c; w3[k] = r.d;
  }
  template <class S>
  __device__ __forceinline__ void position(uint32_t k, const S&, uint32_t, uint32_t, float f[3], float* uq) const {
    f[0] = u01f(w0[k]); f[1] = u01f(w1[k]); f[2] = u01f(w2[k]); *uq = u01f(w3[k]);
  }
};
template <> struct EmitStash<double> {
  uint32_t at[32];
  uint32_t cell[kStash], j[kStash];
  __device__ __forceinline__ void put(uint32_t k, uint32_t c, uint32_t jj, const U4&) { cell[k] = c; j[k] = jj; }
  template <class S>
  __device__ __forceinline__ void position(uint32_t, const S& s, uint32_t c, uint32_t jj, double f[3], double* uq) const {
    Draws<double>::position(s, c, jj, f, uq);
  }
};

// Finish up to 32 packets from the head of the ring (head, count: warp-uniform).
template <class R, bool P2>
__device__ __forceinline__ void emit_finish32(const TransportArgs<R>& a, const EmitBox<R>& e, EmitStash<R>& st,
                                              uint32_t& head, uint32_t& count, uint64_t& my_abs,
                                              uint64_t& my_cross) {
  const int lane = threadIdx.x & 31;
  const uint32_t take = count < 32u ? count : 32u;
  const bool act = (uint32_t)lane < take;
  uint32_t k = head + lane;
  if (k >= kStash) k -= kStash;
  uint32_t cell = 0, j = 0;
  R f[3] = {(R)0, (R)0, (R)0}, xi = (R)0, vt = (R)0;
  if (act) {
    R uq;
    cell = st.cell[k];
    j = st.j[k];
    st.position(k, KStream{a.ks, e.box}, cell, j, f, &uq);
    emit_draw0<R>(a, e, cell, uq, &xi, &vt);
  }
  __syncwarp();  // read before the slots are reused
  head += take;
  if (head >= kStash) head -= kStash;
  count -= take;
  emit_rest<R, P2>(a, e, act, cell, j, f, xi, vt, my_abs, my_cross);
}

template <class R, bool P2>
__device__ __forceinline__ void emit_flush(const TransportArgs<R>& a, const EmitBox<R>& e, EmitStash<R>& st,
                                           uint32_t& head, uint32_t& count, uint64_t& my_abs, uint64_t& my_cross) {
  while (count > 0) emit_finish32<R, P2>(a, e, st, head, count, my_abs, my_cross);
}

template <class R, bool P2, bool FRESH = false>
__device__ __forceinline__ void emit_window64(const TransportArgs<R>& a, const EmitBox<R>& e, EmitStash<R>& st,
                                              uint32_t base, uint32_t N, uint32_t& head, uint32_t& count,
                                              uint64_t& my_abs, uint64_t& my_cross) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (base + 32u * h >= N) break;  // the coarse index ends at the last packet
    uint32_t cell, j, starts;
    bool whole;
    const bool act = emit_locate<R, FRESH>(e, base + 32u * h, N, st.at, &cell, &j, &starts, &whole);
    U4 r{0, 0, 0, 0};
    bool early = false;
    if (act) {
      r = draw(KStream{a.ks, e.box}, cell, j, Draws<R>::kQuantBlock);
      early = r.d < e.early && temperature_plain(__ldg(e.T + cell));
      if (e.early == 0u) early = r.d < a.early && temperature_plain(__ldg(e.T + cell)) && velocity_plain(e.vel[cell]);
    }
    // home tally of the early packets (warp-aggregated)
    const unsigned em = __ballot_sync(0xffffffffu, early);
    const unsigned m = em & (whole ? lane_group(starts) : key_group(cell));
    if (early && (m & lt) == 0u) atomicAdd(e.tally + cell, (uint32_t)__popc(m));
    if (early) ++my_abs;
    // the others to the ring, in lane order after the waiting ones
    const bool pend = act && !early;
    const unsigned pm = __ballot_sync(0xffffffffu, pend);
    if (pend) {
      uint32_t k = head + count + __popc(pm & lt);
      if (k >= kStash) k -= kStash;
      st.put(k, cell, j, r);
    }
    count += __popc(pm);
  }
  __syncwarp();
  while (count >= 32u) emit_finish32<R, P2>(a, e, st, head, count, my_abs, my_cross);
}

// What bounds the emission: the half-rate integer pipe (wide multiplies of Philox) and
// issue in binary32, 1.65 -> 1.59 ms at 256^3 with 1e8 packets when the packets
// settled by their quantile word skip the table; the binary64 pipe in the FP64
// form, 15.1 -> 8.8 ms with those packets, the ring and quotients saved.
// Resident blocks per SM of the emission (registers and the shared-memory ring:
// with the ring a sixth block measured slower, 1.83 against 1.74 ms at 256^3).
template <class R> constexpr int emit_occupancy() { return sizeof(R) == 4 ? 5 : 4; }

template <class R, bool P2>
__global__ void __launch_bounds__(TT, emit_occupancy<R>()) k_emit(TransportArgs<R> a) {
  const EmitBox<R> e{a.P, a.first, (uint32_t)a.n3, (uint32_t)a.n, a.vel, a.T, a.tally, a.kappa, a.cth, 0u, a.tl, 0u,
                     a.sc->vel_plain ? a.early : 0u};
  const uint32_t N = __ldg(a.P + a.n3);  // packets actually allocated
  __shared__ EmitStash<R> stash[TT / 32];
  EmitStash<R>& st = stash[threadIdx.x >> 5];
  uint64_t my_abs = 0, my_cross = 0;
  uint32_t head = 0, count = 0;
  const uint64_t warps_total = (uint64_t)gridDim.x * (TT / 32);
  for (uint64_t base = ((uint64_t)blockIdx.x * (TT / 32) + (threadIdx.x >> 5)) * 64; base < N;
       base += warps_total * 64)
    emit_window64<R, P2>(a, e, st, (uint32_t)base, N, head, count, my_abs, my_cross);
  emit_flush<R, P2>(a, e, st, head, count, my_abs, my_cross);
  add_counters(a.sc, my_abs, 0, my_cross);
  // the last block to finish prepares the march's chunks
  if (!last_block_done(&a.sc->counter)) return;
  bucket_scan_block<TT>(a.bfill, a.cpre, a.nb, a.sc, a.chunk);
  if (threadIdx.x == 0) a.sc->counter = 0;
}

// March of the queued packets.  Persistent warps take chunks of a.chunk queued
// packets (never straddling a bucket) from a shared counter in queue order, so
// the warps advance through the super-tile buckets together and the cells
// they touch stay close in memory; each warp refills its idle lanes from its
// current chunk, so that lanes stay busy whatever the spread of path lengths.
//
// A lane walks a few cells per round.  For every cell it asks the bound of
// rec_velq.cuh, one 32-bit word of the compact velocity copy and one integer dot
// product, whether the packet can be absorbed there at all; a cell whose
// threshold exceeds any possible dot product is not even loaded.  A lane with
// a candidate cell parks.  Once `refill` lanes of a warp are parked or idle, the
// parked ones read the exact velocity of their candidate and take the exact
// resonance test (tally and done, or on to the rest of the round), and the idle
// ones take new packets, so that both run with many lanes at once.
// What bounds it: with flows of 1 km/s, requests from L1 to L2 (72 % busy), instruction
// issue (68 %) and the integer pipe (66 %) together; once Compton drag has slowed the
// flow most cells need no load, and it is issue (74 %) and the integer pipe (73 %).  With
// the velocity vector read in every cell it was the requests alone (87 %): 256^3, 1e8 packets 5.34 -> 3.36 ms, FP64 47.4 -> 7.9 ms;
// 512^3, 1e9 packets with sweeps 111 -> 65.7 ms.
// Cells a lane walks per round, with their words in flight together (256^3 mixed: 3 / 4 /
// 5 / 6 cells 4.07 / 3.57 / 3.60 / 3.43 ms, 8 cells 3.69 at three blocks per SM; FP64: 4 / 6
// cells 7.97 / 8.28 ms; region sweeps of 512^3, 1e9 packets, leaving packets queued after every
// round: 6 / 8 / 10 cells 76.3 / 72.0 / 70.5 ms, 12 spill).
template <class R, bool RS> struct MarchAhead { static constexpr int value = sizeof(R) == 4 ? (RS ? 10 : 6) : 4; };

// Resident blocks per SM of the march (register budget per thread; a batch
// keeps the box of each lane's packet in registers).
template <class R, bool MB, bool RS = false> constexpr int march_occupancy() {
  return RS ? (sizeof(R) == 4 ? 3 : 2) : (MB ? 3 : (sizeof(R) == 4 ? 4 : 3));
}

// The exit distance in binary32 for the bound: binary64 truncates toward zero
// (its bits moved, 2^-23 relative).  Every exit distance is a normal binary32
// number: at least 2^-53 (offset in the cell times tDelta >= 1), at most sqrt(3) per
// crossing (one direction cosine is at least 1/sqrt(3)) times the crossing cap.
__device__ __forceinline__ float bound_exit(float s) { return s; }
__device__ __forceinline__ float bound_exit(double s) {
  return __uint_as_float(__funnelshift_l((uint32_t)__double2loint(s), (uint32_t)__double2hiint(s), 3) + 0x40000000u);
}

// Word of a cell whose threshold some dot product may reach; predicated, not
// branched around.
__device__ __forceinline__ void load_word(uint32_t& w, const uint32_t* q, uint32_t cell, int thr, int top) {
  asm("{\n\t.reg .pred p;\n\t.reg .u64 a;\n\t"
      "setp.le.s32 p, %3, %4;\n\t"
      "mad.wide.u32 a, %2, 4, %1;\n\t"
      "@p ld.global.nc.u32 %0, [a];\n\t}"
      : "+r"(w)
      : "l"(q), "r"(cell), "r"(thr), "r"(top));
}

// Loads that are not used again: past L1, which the words then have to themselves
// (256^3: 3.43 -> 3.38 ms; a batch, short of registers, keeps plain loads).
__device__ __forceinline__ float4 ld_stream(const float4* p) {
  float4 v;
  asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ double4_32a ld_stream(const double4_32a* p) { return *p; }

// One cell of the walk: returns the exit distance (the nearest face, ties
// broken x < y < z) and steps across that face: its next distance, and its part
// of the word index (an addition with a mask, which wraps power-of-two sides).
// The three axes are predicated instructions, written out: as selects they
// cost twice as many, and the march is bound by instruction issue.
__device__ __forceinline__ float walk_step(float& tMx, float& tMy, float& tMz, float tDx, float tDy, float tDz,
                                           uint32_t& X, uint32_t& Y, uint32_t& Z, uint32_t Sx, uint32_t Sy,
                                           uint32_t Sz, uint32_t mx, uint32_t my, uint32_t mz) {
  float s;
  asm("{\n\t.reg .pred px, py, pz;\n\t"
      "min.f32 %0, %1, %2, %3;\n\t"
      "setp.eq.f32 px, %1, %0;\n\t"
      "setp.eq.and.f32 py|pz, %2, %0, !px;\n\t"
      "@px add.rn.f32 %1, %1, %7;\n\t"
      "@py add.rn.f32 %2, %2, %8;\n\t"
      "@pz add.rn.f32 %3, %3, %9;\n\t"
      "@px add.u32 %4, %4, %10;\n\t"
      "@py add.u32 %5, %5, %11;\n\t"
      "@pz add.u32 %6, %6, %12;\n\t"
      "@px and.b32 %4, %4, %13;\n\t"
      "@py and.b32 %5, %5, %14;\n\t"
      "@pz and.b32 %6, %6, %15;\n\t}"
      : "=&f"(s), "+f"(tMx), "+f"(tMy), "+f"(tMz), "+r"(X), "+r"(Y), "+r"(Z)
      : "f"(tDx), "f"(tDy), "f"(tDz), "r"(Sx), "r"(Sy), "r"(Sz), "r"(mx), "r"(my), "r"(mz));
  return s;
}
// Binary64: face distances are positive or +inf, so their bits order as
// integers and no comparison goes to the slow binary64 pipe; the addition is the
// walk's only binary64 operation.
__device__ __forceinline__ double walk_step(double& tMx, double& tMy, double& tMz, double tDx, double tDy, double tDz,
                                            uint32_t& X, uint32_t& Y, uint32_t& Z, uint32_t Sx, uint32_t Sy,
                                            uint32_t Sz, uint32_t mx, uint32_t my, uint32_t mz) {
  const long long a = __double_as_longlong(tMx), b = __double_as_longlong(tMy), c = __double_as_longlong(tMz);
  const bool px = a <= b && a <= c, py = !px && b <= c, pz = !px && !py;
  const double s = __longlong_as_double(px ? a : (py ? b : c));
  const double t = __dadd_rn(s, px ? tDx : (py ? tDy : tDz));
  if (px) { tMx = t; X = (X + Sx) & mx; }
  if (py) { tMy = t; Y = (Y + Sy) & my; }
  if (pz) { tMz = t; Z = (Z + Sz) & mz; }
  return s;
}
// Sides that are no power of two: from the last cell in the direction of travel
// (end, offset E) the step goes to the first one (last ^ E, since one of the two is
// offset 0), where the mask would not wrap.
__device__ __forceinline__ float walk_step_any(float& tMx, float& tMy, float& tMz, float tDx, float tDy, float tDz,
                                               uint32_t& X, uint32_t& Y, uint32_t& Z, uint32_t Sx, uint32_t Sy,
                                               uint32_t Sz, uint32_t mx, uint32_t my, uint32_t mz, uint32_t Ex,
                                               uint32_t Ey, uint32_t Ez, uint32_t lx, uint32_t ly, uint32_t lz) {
  float s;
  asm("{\n\t.reg .pred px, py, pz, ex, ey, ez;\n\t"
      "min.f32 %0, %1, %2, %3;\n\t"
      "setp.eq.f32 px, %1, %0;\n\t"
      "setp.eq.and.f32 py|pz, %2, %0, !px;\n\t"
      "@px add.rn.f32 %1, %1, %7;\n\t"
      "@py add.rn.f32 %2, %2, %8;\n\t"
      "@pz add.rn.f32 %3, %3, %9;\n\t"
      "setp.eq.and.u32 ex, %4, %16, px;\n\t"
      "setp.eq.and.u32 ey, %5, %17, py;\n\t"
      "setp.eq.and.u32 ez, %6, %18, pz;\n\t"
      "@px add.u32 %4, %4, %10;\n\t"
      "@py add.u32 %5, %5, %11;\n\t"
      "@pz add.u32 %6, %6, %12;\n\t"
      "@px and.b32 %4, %4, %13;\n\t"
      "@py and.b32 %5, %5, %14;\n\t"
      "@pz and.b32 %6, %6, %15;\n\t"
      "@ex xor.b32 %4, %16, %19;\n\t"
      "@ey xor.b32 %5, %17, %20;\n\t"
      "@ez xor.b32 %6, %18, %21;\n\t}"
      : "=&f"(s), "+f"(tMx), "+f"(tMy), "+f"(tMz), "+r"(X), "+r"(Y), "+r"(Z)
      : "f"(tDx), "f"(tDy), "f"(tDz), "r"(Sx), "r"(Sy), "r"(Sz), "r"(mx), "r"(my), "r"(mz), "r"(Ex), "r"(Ey), "r"(Ez),
        "r"(lx), "r"(ly), "r"(lz));
  return s;
}
__device__ __forceinline__ double walk_step_any(double& tMx, double& tMy, double& tMz, double tDx, double tDy,
                                                double tDz, uint32_t& X, uint32_t& Y, uint32_t& Z, uint32_t Sx,
                                                uint32_t Sy, uint32_t Sz, uint32_t mx, uint32_t my, uint32_t mz,
                                                uint32_t Ex, uint32_t Ey, uint32_t Ez, uint32_t lx, uint32_t ly,
                                                uint32_t lz) {
  const uint32_t x0 = X, y0 = Y, z0 = Z;
  const double s = walk_step(tMx, tMy, tMz, tDx, tDy, tDz, X, Y, Z, Sx, Sy, Sz, mx, my, mz);
  if (X != x0 && x0 == Ex) X = lx ^ Ex;
  if (Y != y0 && y0 == Ey) Y = ly ^ Ey;
  if (Z != z0 && z0 == Ez) Z = lz ^ Ez;
  return s;
}

// End of a transport call of a single box (one thread; the counters were added by
// other blocks' atomics: read through L2).
__device__ __forceinline__ void transport_end(DevScalars* sc, rec_stats* st) {
  const unsigned long long absorbed = __ldcg(&sc->absorbed), capped = __ldcg(&sc->capped);
  sc->tally_total = __ldcg(&sc->tally_total) + absorbed;
  if (capped) atomicOr(&sc->flags, 2);
  if (st) {
    st->emitted = __ldcg(&sc->emitted);
    st->absorbed = absorbed;
    st->capped = capped;
    st->crossings = __ldcg(&sc->crossings);
    st->queued = __ldcg(&sc->qtail);
    st->requeued = __ldcg(&sc->requeued);
    st->flags = __ldcg(&sc->flags);
  }
}

__device__ __forceinline__ void transport_end_batch(const BoxDev* bxs, int B, const unsigned long long* bfill,
                                                    rec_stats* st);

// P2: the box side is a power of two (periodic wrap by masks).
// MB: batched context; the lanes of a warp may hold packets of different boxes.
// F: kCopyOut: cells beyond the scale of the copy exist, which are candidates whatever
// their threshold (a body of its own: the test costs the others 2 %).  kDirect: a context
// without the copy reads the velocity of every cell, a few cells ahead of the tests.
enum MarchForm { kCopy, kCopyOut, kDirect };
template <class R, bool P2, bool MB, bool RS, MarchForm F>
__device__ __forceinline__ void march_body(const TransportArgs<R>& a, const BoxDev* bxs, int B, const BoxStep* bst,
                                           BoxCounters& cnt) {
  static_assert(!RS || (P2 && !MB), "region sweeps: single box of power-of-two side");
  static_assert(!MB || !P2, "a batch mixes sides");
  using V = typename Vec4<R>::T;
  constexpr int kA = F != kDirect ? MarchAhead<R, RS>::value : (sizeof(R) == 4 ? 4 : 2);
  const int lane = threadIdx.x & 31;
  const uint32_t n = (uint32_t)a.n;
  // region sweeps: bucket of the open chunk (its super-tile); path length at
  // which the lane's packet leaves the region around it (+inf: no limit)
  uint32_t cbk = 0;
  float leave = 0.0f;
  bool gone = false;  // it has left, and waits to be queued again
  // box of the lane's packet and of the open chunk
  int lbox = -1, cbox = 0;
  const uint32_t* q = a.velq;
  uint32_t bx = a.vbx, ln = n;
  // A cell as three parts, one per axis, that a step adds to under a mask: of the copy's
  // word index, or without the copy of the cell index (power-of-two side) or ten bits per axis.
  const uint32_t sh = P2 ? a.tl.lg : 10u, low = P2 ? n - 1u : 1023u;
  auto part_x = [&](uint32_t i) { return F == kDirect ? i : velq_x(i); };
  auto part_y = [&](uint32_t i) { return F == kDirect ? i << sh : velq_y(i, bx); };
  auto part_z = [&](uint32_t i) { return F == kDirect ? i << (2u * sh) : velq_z(i, bx); };
  auto coords = [&](uint32_t c, uint32_t* ix, uint32_t* iy, uint32_t* iz) {
    if (F != kDirect) return velq_coords(c, bx, ix, iy, iz);
    *ix = c & low; *iy = (c >> sh) & low; *iz = c >> (2u * sh);
  };
  VelqMasks lm = F == kDirect ? VelqMasks{low, low << sh, low << (2u * sh)} : a.vm;
  uint32_t lastx = 0, lasty = 0, lastz = 0;
  R lkappa = a.kappa;
  if (!MB) { lastx = part_x(n - 1u); lasty = part_y(n - 1u); lastz = part_z(n - 1u); }
  uint64_t pos = 0;   // next queue slot of the open chunk
  uint32_t left = 0;  // slots left in it
  bool more = true;
  bool active = false, parked = false;
  // the packet: cell (three parts of the word index), face distances, steps, resonance
  uint32_t X = 0, Y = 0, Z = 0, Sx = 0, Sy = 0, Sz = 0, Ex = 0, Ey = 0, Ez = 0, kc = 0;
  R tMx = 0, tMy = 0, tMz = 0, tDx = 0, tDy = 0, tDz = 0, knx = 0, kny = 0, knz = 0, u0 = 0;
  VelqPacket vp;
  vp.m = 0; vp.c1 = vp.c2 = 0.0f; vp.top = 0;
  // the last round: cells, exit distances, words, first cell not yet cleared
  uint32_t cl[kA] = {}, qw[kA] = {}, kfrom = 0;
  R se[kA] = {};
  // counters of the lane; crossings are flushed before 32 bits could overflow
  uint32_t my_abs = 0, my_cap = 0, my_cross = 0;
  for (;;) {
    const unsigned stop = __ballot_sync(0xffffffffu, !active || parked);
    if (__popc(stop) >= a.refill || stop == 0xffffffffu) {
      // exact test of the parked lanes' first candidate cell
      if (F != kDirect && parked && !(RS && gone)) {
        uint32_t cand = 0;
#pragma unroll
        for (int k = 0; k < kA; ++k) {
          const int thr = __float_as_int(fmaf(-bound_exit(se[k]), vp.c1, vp.c2));
          if (velq_dot(qw[k], vp.m, kVelqBiasBits) >= thr || (F == kCopyOut && velq_is_out(qw[k])) ||
              kc - (uint32_t)(kA - k) >= kMaxCrossings)
            cand |= 1u << k;
        }
        cand &= 0xffffffffu << kfrom;
        if (cand == 0) {
          parked = false;
        } else {
          const uint32_t k = (uint32_t)__ffs((int)cand) - 1u;
          uint32_t c = cl[0];
          R s = se[0];
#pragma unroll
          for (int i = 1; i < kA; ++i)
            if (k == (uint32_t)i) { c = cl[i]; s = se[i]; }
          uint32_t ix, iy, iz;
          velq_coords(c, bx, &ix, &iy, &iz);
          const uint32_t lin = (iz * ln + iy) * ln + ix;
          const V* vel = MB ? (const V*)bxs[lbox].vel4 : a.vel;
          const V U = MB ? vel[lin] : ld_stream(vel + lin);
          Ray<R> r;
          r.knx = knx; r.kny = kny; r.knz = knz;
          // resonance in the cell at path length u0 - kappa n.U: absorb unless beyond its exit
          const uint32_t kcell = kc - (uint32_t)kA + k;  // crossings before this cell
          const bool hit = Ar<R>::sub(u0, doppler(r, U)) <= s;
          if (hit || kcell >= kMaxCrossings) {
            active = parked = false;
            my_cross += kcell - 1;  // crossings up to this cell; the first was counted at emission
            if (my_cross >= 0x80000000u) {
              if (MB) box_counters_add(cnt, lbox, 0, 0, my_cross);
              else atomicAdd(&a.sc->crossings, (unsigned long long)my_cross);
              my_cross = 0;
            }
            if (hit) { atomicAdd((MB ? bxs[lbox].tally : a.tally) + lin, 1u); ++my_abs; }
            else ++my_cap;
          } else {
            kfrom = k + 1u;
            parked = (cand >> kfrom) != 0u;
          }
        }
        if (RS) gone = active && !parked && bound_exit(se[kA - 1]) >= leave;
      }
      if (RS) {
        // packets that left their region: appended to the second queue as full
        // states (the current cell is the next to test), counted in the bucket
        // of the super-tile they have reached
        const unsigned rm = __ballot_sync(0xffffffffu, gone);
        if (rm) {
          uint32_t ix, iy, iz;
          coords(X | Y | Z, &ix, &iy, &iz);
          const uint32_t cell = (((iz << a.tl.lg) | iy) << a.tl.lg) | ix;
          // the warp's part of the second queue
          const uint32_t part = (blockIdx.x * (TT / 32) + (threadIdx.x >> 5)) & (uint32_t)(kRqParts - 1);
          unsigned long long qb = 0;
          const int leader = __ffs(rm) - 1;
          if (lane == leader) qb = atomicAdd(&a.rqn[part], (unsigned long long)__popc(rm));
          qb = __shfl_sync(0xffffffffu, qb, leader);
          const uint64_t k = qb + __popc(rm & ((1u << lane) - 1u));
          const bool stored = gone && k < a.rq_part;
          if (stored) {
            const uint64_t slot = (uint64_t)part * a.rq_part + k;
            V q0v, q1v, q2v;
            q0v.x = bits_to<R>(cell); q0v.y = tMx; q0v.z = tMy; q0v.w = tMz;
            q1v.x = copysign(tDx, knx); q1v.y = copysign(tDy, kny); q1v.z = copysign(tDz, knz); q1v.w = u0;
            q2v.x = knx; q2v.y = kny; q2v.z = knz; q2v.w = bits_to<R>(kc);
            a.rq[3 * slot] = q0v;
            a.rq[3 * slot + 1] = q1v;
            a.rq[3 * slot + 2] = q2v;
            active = false;
          }
          const unsigned sm = __ballot_sync(0xffffffffu, stored);
          const uint32_t bk = stored ? a.tl.template at<true>(cell) : 0xffffffffu;
          const unsigned gm = __match_any_sync(0xffffffffu, bk) & sm;
          if (stored && lane == __ffs(gm) - 1) atomicAdd(&a.rcount[bk], (unsigned long long)__popc(gm));
          if (gone && !stored) leave = __int_as_float(0x7f800000);  // the second queue is full: march on without a limit
          if (__any_sync(0xffffffffu, gone && !stored) && lane == 0) atomicOr(&a.sc->flags, 16);
          if (gone) gone = parked = false;
        }
      }
      // refill idle lanes in lane order from the warp's chunks
      unsigned idle = __ballot_sync(0xffffffffu, !active);
      while (idle && more) {
        if (left == 0) {
          // next chunk in queue order, shared by all warps: the warps in flight
          // stay on neighbouring chunks, so their rays start close together
          unsigned long long nc = 0;
          if (lane == 0) nc = atomicAdd(&a.sc->march_next, 1ull);
          const uint64_t chunk = __shfl_sync(0xffffffffu, nc, 0);
          if (chunk >= __ldg(a.cpre + a.nb)) { more = false; break; }
          // bucket of this chunk: last b with cpre[b] <= chunk (cpre[0] = 0).  A binary search, the
          // same in every lane (the lanes probing 32 places at once: 3.60 against 3.43 ms at 256^3)
          uint32_t lo = 0, hi = (uint32_t)a.nb;
          while (hi - lo > 1) {
            uint32_t mid = (lo + hi) >> 1;
            if (__ldg(a.cpre + mid) <= chunk) lo = mid;
            else hi = mid;
          }
          const uint64_t k0 = (chunk - __ldg(a.cpre + lo)) * a.chunk;
          pos = a.boff[lo] + k0;
          left = (uint32_t)min((uint64_t)a.chunk, (uint64_t)(a.bfill[lo] - k0));
          if (RS) cbk = lo;
          if (MB) cbox = last_le(B, lo, [&](int i) { return bxs[i].bk0; });  // last b with bk0 <= lo
        }
        const uint32_t take = min((uint32_t)__popc(idle), left);
        const uint32_t rank = __popc(idle & ((1u << lane) - 1u));
        if (((idle >> lane) & 1u) && rank < take) {
          const uint64_t slot = pos + rank;
          constexpr int QV = QueueVecs<R>::value;
          if (MB) {
            if (lbox != cbox) {  // counters of the previous box to shared memory
              if (lbox >= 0) box_counters_add(cnt, lbox, my_abs, my_cap, my_cross);
              my_abs = my_cap = my_cross = 0;
              lbox = cbox;
              const BoxDev& d = bxs[lbox];
              ln = d.n;
              bx = d.vbx;
              if (F != kDirect) lm = velq_masks(ln, bx, false);
              q = d.velq;
              lkappa = (R)bst[lbox].kappa;
              lastx = part_x(ln - 1u); lasty = part_y(ln - 1u); lastz = part_z(ln - 1u);
            }
          }
          uint32_t cell;
          int sx, sy, sz;
          if (RS && a.resumed) {
            // a full state queued again by an earlier sweep
            const V q0v = a.queue[3 * slot], q1v = a.queue[3 * slot + 1], q2v = a.queue[3 * slot + 2];
            cell = to_bits<R>(q0v.x);
            tMx = q0v.y; tMy = q0v.z; tMz = q0v.w;
            sx = q1v.x < (R)0 ? -1 : 1; tDx = fabs(q1v.x);
            sy = q1v.y < (R)0 ? -1 : 1; tDy = fabs(q1v.y);
            sz = q1v.z < (R)0 ? -1 : 1; tDz = fabs(q1v.z);
            u0 = q1v.w;
            knx = q2v.x; kny = q2v.y; knz = q2v.z;
            kc = to_bits<R>(q2v.w);
          } else {
            const V* entry = a.queue + QV * slot;
            const V q0v = MB ? entry[0] : ld_stream(entry), q1v = MB ? entry[1] : ld_stream(entry + 1);
            cell = to_bits<R>(q0v.x);
            tMx = q0v.y; tMy = q0v.z; tMz = q0v.w;
            u0 = q1v.w;
            if (QV == 2) {  // tDelta and kappa n exactly as the emission formed them
              axis_setup<R>(q1v.x, &tDx, &sx);
              axis_setup<R>(q1v.y, &tDy, &sy);
              axis_setup<R>(q1v.z, &tDz, &sz);
              knx = Ar<R>::mul(lkappa, q1v.x); kny = Ar<R>::mul(lkappa, q1v.y); knz = Ar<R>::mul(lkappa, q1v.z);
            } else {
              const V q2v = a.queue[QV * slot + 2];
              sx = q1v.x < (R)0 ? -1 : 1; tDx = fabs(q1v.x);
              sy = q1v.y < (R)0 ? -1 : 1; tDy = fabs(q1v.y);
              sz = q1v.z < (R)0 ? -1 : 1; tDz = fabs(q1v.z);
              knx = q2v.x; kny = q2v.y; knz = q2v.z;
            }
            kc = 1;  // the step out of the home cell
          }
          uint32_t ix, iy, iz;
          if (MB) {
            const BoxDev& d = bxs[lbox];
            Tiles{d.n, d.nt, d.lg, d.mn, d.mn2, d.tlg}.template coords<false>(cell, &ix, &iy, &iz);
          } else {
            a.tl.template coords<P2>(cell, &ix, &iy, &iz);
          }
          X = part_x(ix); Y = part_y(iy); Z = part_z(iz);
          if (RS) {
            // the region: the bucket's super-tile widened by the halo (periodic:
            // offsets from its low corner modulo n).  Along an axis the packet leaves
            // after the cells that are left of it in the direction of travel.
            leave = __int_as_float(0x7f800000);
            if (a.halo) {
              const uint32_t tlg = a.tl.tlg, ntl = a.tl.lg - tlg, ntm = (1u << ntl) - 1u, m = n - 1u;
              const uint32_t far = (1u << tlg) + 2u * a.halo - 1u;
              const uint32_t rx = (ix - (((cbk & ntm) << tlg) - a.halo)) & m;
              const uint32_t ry = (iy - ((((cbk >> ntl) & ntm) << tlg) - a.halo)) & m;
              const uint32_t rz = (iz - (((cbk >> (2u * ntl)) << tlg) - a.halo)) & m;
              leave = fminf(leave, (float)tMx + (float)(sx > 0 ? far - rx : rx) * (float)tDx);
              leave = fminf(leave, (float)tMy + (float)(sy > 0 ? far - ry : ry) * (float)tDy);
              leave = fminf(leave, (float)tMz + (float)(sz > 0 ? far - rz : rz) * (float)tDz);
            }
          }
          Sx = sx > 0 ? 0u - lm.x : 0u - 1u;
          Sy = sy > 0 ? 0u - lm.y : 0u - (F == kDirect ? 1u << sh : 2u);
          Sz = sz > 0 ? 0u - lm.z : 0u - (F == kDirect ? 1u << (2u * sh) : 4u);
          if (!P2) { Ex = sx > 0 ? lastx : 0u; Ey = sy > 0 ? lasty : 0u; Ez = sz > 0 ? lastz : 0u; }
          if (F != kDirect) {
            const DevScalars* bsc = MB ? bxs[lbox].sc : a.sc;
            const VelqBox vb = velq_box(bsc->vq_u, bsc->vq_v, (float)lkappa);
            vp = velq_packet<F == kCopyOut>(vb, (float)knx, (float)kny, (float)knz, (float)u0);
          }
          active = true;
        }
        pos += take;
        left -= take;
        idle = __ballot_sync(0xffffffffu, !active);
      }
    }
    if (!__any_sync(0xffffffffu, active)) break;  // no packet left in the warp
    if (F == kDirect && active && !parked) {
      // one round: walk kA cells and read their velocities, then test them in order
      uint32_t lin[kA];
      V U[kA];
      const V* vel = MB ? (const V*)bxs[lbox].vel4 : a.vel;
#pragma unroll
      for (int k = 0; k < kA; ++k) {
        lin[k] = P2 ? X | Y | Z : ((Z >> 20) * ln + (Y >> 10)) * ln + X;
        U[k] = vel[lin[k]];
        if (P2)
          se[k] = walk_step(tMx, tMy, tMz, tDx, tDy, tDz, X, Y, Z, Sx, Sy, Sz, lm.x, lm.y, lm.z);
        else
          se[k] = walk_step_any(tMx, tMy, tMz, tDx, tDy, tDz, X, Y, Z, Sx, Sy, Sz, lm.x, lm.y, lm.z, Ex, Ey, Ez, lastx,
                                lasty, lastz);
      }
      Ray<R> r;
      r.knx = knx; r.kny = kny; r.knz = knz;
      bool hit = false;
      uint32_t at = 0, kcell = kc;
#pragma unroll
      for (int k = 0; k < kA; ++k) {
        if (!active) continue;
        hit = Ar<R>::sub(u0, doppler(r, U[k])) <= se[k];
        if (hit || kc + (uint32_t)k >= kMaxCrossings) { active = false; at = lin[k]; kcell = kc + (uint32_t)k; }
      }
      kc += kA;
      if (!active) {
        my_cross += kcell - 1;
        if (my_cross >= 0x80000000u) {
          if (MB) box_counters_add(cnt, lbox, 0, 0, my_cross);
          else atomicAdd(&a.sc->crossings, (unsigned long long)my_cross);
          my_cross = 0;
        }
        if (hit) { atomicAdd((MB ? bxs[lbox].tally : a.tally) + at, 1u); ++my_abs; }
        else ++my_cap;
      } else if (RS && bound_exit(se[kA - 1]) >= leave) {
        gone = parked = true;
      }
    } else if (F != kDirect && active && !parked) {
      // one round: walk kA cells, loading the words that matter, then ask the bound
#pragma unroll
      for (int k = 0; k < kA; ++k) {
        cl[k] = X | Y | Z;
        if (P2)
          se[k] = walk_step(tMx, tMy, tMz, tDx, tDy, tDz, X, Y, Z, Sx, Sy, Sz, lm.x, lm.y, lm.z);
        else
          se[k] = walk_step_any(tMx, tMy, tMz, tDx, tDy, tDz, X, Y, Z, Sx, Sy, Sz, lm.x, lm.y, lm.z, Ex, Ey, Ez, lastx,
                                lasty, lastz);
        load_word(qw[k], q, cl[k], __float_as_int(fmaf(-bound_exit(se[k]), vp.c1, vp.c2)), vp.top);
      }
      kc += kA;
      kfrom = 0;
      parked = kc > kMaxCrossings;
#pragma unroll
      for (int k = 0; k < kA; ++k)
        parked |= velq_dot(qw[k], vp.m, kVelqBiasBits) >= __float_as_int(fmaf(-bound_exit(se[k]), vp.c1, vp.c2));
      if (F == kCopyOut) {
        uint32_t any = 0;
#pragma unroll
        for (int k = 0; k < kA; ++k) any |= qw[k];
        parked |= velq_is_out(any);
      }
      // a packet that left its region waits for the warp's next stop, so that the
      // append runs with many lanes: with one or two lanes after each round
      // the sweeps of 512^3, 1e9 packets took 70.9 ms, with this 65.3
      if (RS && !parked && bound_exit(se[kA - 1]) >= leave) gone = parked = true;
    }
  }
  if (!MB) add_counters(a.sc, my_abs, my_cap, my_cross);
  else if (lbox >= 0) box_counters_add(cnt, lbox, my_abs, my_cap, my_cross);
}

template <class R, bool P2, bool MB, bool RS, bool COPY>
__global__ void __launch_bounds__(TT, (march_occupancy<R, MB, RS>())) k_march(TransportArgs<R> a, const BoxDev* bxs,
                                                                              int B, const BoxStep* bst,
                                                                              rec_stats* st) {
  __shared__ BoxCounters cnt;
  bool out = COPY && !MB && a.sc->vq_out != 0;
  if (MB) {
    box_counters_clear(cnt, B);
    if (COPY)
      for (int b = threadIdx.x & 31; b < B; b += 32) out |= bxs[b].sc->vq_out != 0;
    out = __any_sync(0xffffffffu, out);
  }
  if (!COPY) march_body<R, P2, MB, RS, kDirect>(a, bxs, B, bst, cnt);
  else if (!out) march_body<R, P2, MB, RS, kCopy>(a, bxs, B, bst, cnt);
  else march_body<R, P2, MB, RS, kCopyOut>(a, bxs, B, bst, cnt);
  if (MB) {
    box_counters_flush(cnt, bxs, B);
    // the last block to finish closes the call: queued counts, tally totals, statistics
    if (last_block_done(&a.sc->counter)) {
      transport_end_batch(bxs, B, a.bfill, st);
      if (threadIdx.x == 0) a.sc->counter = 0;
    }
  } else {
    // the last block of the last march closes the call: tally total, statistics
    if (!a.closes || !last_block_done(&a.sc->counter)) return;
    if (threadIdx.x == 0) {
      transport_end(a.sc, st);
      a.sc->counter = 0;
    }
  }
}

// Region sweeps, between two march launches (one block): the entries each
// bucket received in the second queue become the march queue of the next
// sweep: bucket offsets (exclusive prefix of the counts), fills, march-chunk
// prefix; the counts and the placement fills are reset.
__global__ void __launch_bounds__(1024) k_requeue_scan(unsigned long long* rcount, unsigned long long* boff,
                                                       unsigned long long* bfill, unsigned long long* cpre,
                                                       unsigned long long* scnt, unsigned long long* rqn, int nb,
                                                       DevScalars* sc, uint32_t chunk, uint64_t part_cap) {
  constexpr int NTH = 1024;
  static_assert(kRqParts <= NTH, "one thread per part");
  __shared__ unsigned long long stored;
  if (threadIdx.x == 0) stored = 0;
  __syncthreads();
  if (threadIdx.x < kRqParts) {  // entries each part holds for the placement; append counters reset
    const unsigned long long m = rqn[threadIdx.x], c = m < part_cap ? m : part_cap;
    rqn[kRqParts + threadIdx.x] = c;
    rqn[threadIdx.x] = 0;
    atomicAdd(&stored, c);
  }
  const int per = (nb + NTH - 1) / NTH;
  const int b0 = threadIdx.x * per, b1 = min(nb, (int)(threadIdx.x + 1) * per);
  unsigned long long se = 0, sc_ = 0, all, chunks;
  for (int b = b0; b < b1; ++b) {
    const unsigned long long f = __ldcg(&rcount[b]);
    se += f;
    sc_ += (f + chunk - 1) / chunk;
  }
  unsigned long long re = block_prefix<NTH>(se, &all);
  unsigned long long rc = block_prefix<NTH>(sc_, &chunks);
  if (threadIdx.x == 0) {
    cpre[nb] = chunks;
    sc->requeued += stored;
    sc->march_next = 0;
  }
  for (int b = b0; b < b1; ++b) {
    const unsigned long long f = __ldcg(&rcount[b]);
    boff[b] = re;
    bfill[b] = f;
    cpre[b] = rc;
    re += f;
    rc += (f + chunk - 1) / chunk;
    rcount[b] = 0;
    scnt[b] = 0;
  }
}

// Region sweeps: every entry of the second queue to its bucket's range of the
// march queue (order within a bucket is free: the march of a packet does not
// depend on the others).
template <class R>
__global__ void __launch_bounds__(TT) k_requeue_place(TransportArgs<R> a, unsigned long long* scnt) {
  using V = typename Vec4<R>::T;
  const int lane = threadIdx.x & 31;
  for (int part = blockIdx.x; part < kRqParts; part += gridDim.x) {
  const uint64_t m = a.rqn[kRqParts + part], off = (uint64_t)part * a.rq_part;
  for (uint64_t base = (uint64_t)(threadIdx.x >> 5) * 32; base < m; base += TT) {
    const uint64_t i = base + lane;
    const bool act = i < m;
    V q0v, q1v, q2v;
    uint32_t bk = 0xffffffffu;
    if (act) {
      q0v = a.rq[3 * (off + i)]; q1v = a.rq[3 * (off + i) + 1]; q2v = a.rq[3 * (off + i) + 2];
      bk = a.tl.template at<true>(to_bits<R>(q0v.x));
    }
    const unsigned am = __ballot_sync(0xffffffffu, act);
    const unsigned gm = __match_any_sync(0xffffffffu, bk) & am;
    const int leader = __ffs(gm) - 1;
    unsigned long long qb = 0;
    if (act && lane == leader) qb = atomicAdd(&scnt[bk], (unsigned long long)__popc(gm));
    qb = __shfl_sync(0xffffffffu, qb, leader < 0 ? 0 : leader);
    if (act) {
      const uint64_t slot = a.boff[bk] + qb + __popc(gm & ((1u << lane) - 1u));
      a.queue[3 * slot] = q0v;
      a.queue[3 * slot + 1] = q1v;
      a.queue[3 * slot + 2] = q2v;
    }
  }
  }
}

// Consecutive cells per thread of the single-box allocation: few for small
// boxes, whose time is one thread's serial chain (quotients, remainders) on a
// part of the chip, many for large ones, where the passes stream and the
// prefix's 128-bit division is shared.  Whole passes with 16 cells per thread
// against the rule's: 32^3 FP64 step 250 / 217 us, 100^3 transport 326 / 318 us.
int alloc_items(int64_t n3) { return n3 <= (1 << 17) ? 1 : (n3 <= (1 << 21) ? 4 : kAllocItems); }

template <class R, int IT>
void alloc_launch(rec_ctx* c, int blocks, const typename Vec4<R>::T* vel, const Stream& s, const Tiles& tl, int nb) {
  const R* emis = (const R*)c->box.emis;
  const uint64_t npk = c->box.n_packets;
  k_alloc_sum<R, IT><<<blocks, AT, 0, c->stream>>>(emis, vel, c->n3, npk, s, c->sc, c->partQ, c->P, c->velq,
                                                   velq_bits((uint32_t)c->box.n), tl);
  k_alloc_prefix<R, IT><<<blocks, AT, 0, c->stream>>>(emis, c->n3, npk, c->sc, c->partQ, c->P, c->first, tl, c->bcap,
                                                      c->bfill, nb);
}

// Without the copy (256^3, 1e8 packets) the march takes 6.2 ms; as a bound that excludes
// nothing, so that six cells cost a round and six stops, it took 21.6.
template <class R, bool P2, bool MB, bool RS>
void march_launch(rec_ctx* c, const TransportArgs<R>& a, int blocks, const BoxDev* bxs, int B, const BoxStep* bst,
                  rec_stats* st) {
  if (c->velq) k_march<R, P2, MB, RS, true><<<blocks, TT, 0, c->stream>>>(a, bxs, B, bst, st);
  else k_march<R, P2, MB, RS, false><<<blocks, TT, 0, c->stream>>>(a, bxs, B, bst, st);
}

// Bound of the quantile's leading word w below which xi <= 0 (0: none).  The deviate
// u < (w + 257) 2^-32 (binary32 keeps the top 23 bits and adds half a unit), the table node k = trunc(u (M - 1)) after
// one rounding (2^-23 relative covers both precisions), and a node is safe if
// interpolation from it cannot pass zero by rounding: its upper end q1 = 0 (then q1 - q0 is
// exact), or q1 <= -2^-20 |q0|.
uint32_t early_word(const rec_ctx* c, double kappa, double cth) {
  if (!(cth <= 1e15) || !(kappa < 1e15)) return 0u;
  const double w = std::floor((double)c->early_nodes / (double)(c->params.n_quantiles - 1) * (1.0 - 0x1p-22) * 0x1p32) - 258.0;
  return w > 0.0 ? (uint32_t)std::min(w, 4294967295.0) : 0u;
}

template <class R>
cudaError_t run_transport(rec_ctx* c, int step, double z, rec_stats* st) {
  const rec_box& b = c->box;
  Stream s{(uint32_t)c->params.seed, (uint32_t)(c->params.seed >> 32) ^ (uint32_t)step, 0u};
  const bool p2 = (b.n & (b.n - 1)) == 0;
  const rec_tuning& tu = c->tune;
  const Tiles tl = make_tiles(b.n, tu.tile);
  const int nb = (int)(tl.nt * tl.nt * tl.nt);
  double kappa, cth;
  transport_scalars(c->cosmo, b.n, z, &kappa, &cth);
  {
    GroupTimer t(c, kTAlloc, 3);
    const typename Vec4<R>::T* vel = (const typename Vec4<R>::T*)b.vel4;
    k_alloc_max<R><<<c->grid, kPassThreads, 0, c->stream>>>((const R*)b.emis, vel, c->n3, (float)kappa, c->sc, c->bcap, nb);
    const int it = alloc_items(c->n3), ab = c->alloc_blocks;
    if (it == 1) alloc_launch<R, 1>(c, ab, vel, s, tl, nb);
    else if (it == 4) alloc_launch<R, 4>(c, ab, vel, s, tl, nb);
    else alloc_launch<R, kAllocItems>(c, ab, vel, s, tl, nb);
  }
  TransportArgs<R> a;
  a.P = c->P;
  a.first = c->first;
  a.n3 = c->n3;
  a.n = b.n;
  a.vel = (const typename Vec4<R>::T*)b.vel4;
  a.T = (const R*)b.T;
  a.quant = (const R*)c->quant;
  a.M = c->params.n_quantiles;
  a.kappa = (R)kappa;
  a.cth = (R)cth;
  a.ks = key_schedule(s.k0, s.k1);
  a.early = early_word(c, kappa, cth);
  a.tally = b.tally;
  a.sc = c->sc;
  a.queue = (typename Vec4<R>::T*)c->queue;
  a.tl = tl;
  a.nb = nb;
  a.boff = c->bcap;
  a.bfill = c->bfill;
  a.cpre = c->cpre;
  a.chunk = (uint32_t)tu.march_chunk;
  a.refill = tu.march_refill;
  a.rq = nullptr;
  a.rcount = nullptr;
  a.rqn = nullptr;
  a.rq_part = 0;
  a.halo = 0;
  a.resumed = 0;
  a.closes = 1;
  a.velq = c->velq;
  a.vbx = velq_bits((uint32_t)b.n);
  a.vm = velq_masks((uint32_t)b.n, a.vbx, p2);
  {
    GroupTimer t(c, kTEmit, 1);
    const int eb = c->sm_count * tu.emit_blocks_per_sm;
    if (p2) k_emit<R, true><<<eb, TT, 0, c->stream>>>(a);
    else k_emit<R, false><<<eb, TT, 0, c->stream>>>(a);
  }
  const uint32_t halo = (uint32_t)tu.march_halo;
  const bool sweeps = p2 && halo > 0 && c->rqueue && ((uint32_t)tu.tile + 2u * halo) < (uint32_t)b.n;
  if (!sweeps) {
    GroupTimer t(c, kTMarch, 1);
    const int mb = c->sm_count * tu.march_blocks_per_sm;
    if (p2) march_launch<R, true, false, false>(c, a, mb, nullptr, 1, nullptr, st);
    else march_launch<R, false, false, false>(c, a, mb, nullptr, 1, nullptr, st);
  } else {
    // region sweeps: each march leaves the packets that stray beyond the halo of
    // their bucket's super-tile in the second queue; those are placed by the
    // super-tile they reached and marched by the next sweep; the last sweep has
    // no limit, so every packet ends
    GroupTimer t(c, kTMarch, 3 * kMaxSweeps - 2);
    const int mb = c->sm_count * tu.march_blocks_per_sm;
    a.rq = (typename Vec4<R>::T*)c->rqueue;
    a.rcount = c->rcount;
    a.rqn = c->rqn;
    a.rq_part = c->rq_cap / kRqParts;
    cudaMemsetAsync(c->rqn, 0, sizeof(unsigned long long) * kRqParts, c->stream);
    for (int k = 0; k < kMaxSweeps; ++k) {
      if (k > 0) {
        k_requeue_scan<<<1, 1024, 0, c->stream>>>(c->rcount, c->bcap, c->bfill, c->cpre, c->scnt, c->rqn, nb, c->sc,
                                                  a.chunk, a.rq_part);
        k_requeue_place<R><<<kRqParts, TT, 0, c->stream>>>(a, c->scnt);
      }
      a.resumed = k > 0;
      a.closes = k + 1 == kMaxSweeps;
      a.halo = a.closes ? 0u : halo;
      march_launch<R, true, false, true>(c, a, mb, nullptr, 1, nullptr, st);
    }
  }
  return cudaGetLastError();
}

// ---- batched contexts: every phase is one launch over all boxes ------------------

// Transport scalars of every box, a kernel parameter.
struct BoxStepArgs {
  BoxStep s[kMaxBoxes];
};

// Allocation blocks: kAllocChunk cells of one box each; box of block g = last b
// with ablk0 <= g.
__device__ __forceinline__ int alloc_box(const BoxDev* bxs, int B, uint32_t g) {
  return last_le(B, g, [&](int i) { return bxs[i].ablk0; });
}

// Allocation phases of a batch as functions of the allocation block g of ng
// (blockIdx.x of a per-phase launch, or a virtual block of the persistent one).
template <class R>
__device__ __forceinline__ void alloc_max_batch(const BoxDev* bxs, const BoxStepArgs& bs, int B, DevScalars* gsc,
                                                uint32_t g, uint32_t ng) {
  using V = typename Vec4<R>::T;
  const int b = alloc_box(bxs, B, g);
  const BoxDev& d = bxs[b];
  const int64_t c0 = (int64_t)(g - d.ablk0) * kAllocChunk + (int64_t)threadIdx.x * kAllocItems;
  R v[kAllocItems];
  load_items<R, kAllocItems>((const R*)d.emis, c0, d.n3, v);
  R m = (R)0;
  bool bad = false;
#pragma unroll
  for (int k = 0; k < kAllocItems; ++k) {
    if (c0 + k >= d.n3) continue;
    const R r = v[k];
    if (!(r >= (R)0) || isinf(r)) bad = true;
    else m = m < r ? r : m;
  }
  VelMax vm;
  for (int k = 0; k < kAllocItems; ++k) {
    const int64_t i = (int64_t)(g - d.ablk0) * kAllocChunk + (int64_t)k * AT + threadIdx.x;
    if (i < d.n3) vm.add(((const V*)d.vel4)[i]);
  }
  block_maxima<AT>(d.sc, order_bits(m), vm, bad);
  if (!last_block_done(&gsc->counter, ng)) return;
  for (int i = threadIdx.x; i < B; i += AT) take_maxima<R>(bxs[i].sc, bxs[i].n3, (float)(R)bs.s[i].kappa);
  if (threadIdx.x == 0) gsc->counter = 0;
}
template <class R>
__global__ void __launch_bounds__(AT) k_alloc_max_batch(const BoxDev* bxs, BoxStepArgs bs, int B,
                                                        DevScalars* gsc) {
  alloc_max_batch<R>(bxs, bs, B, gsc, blockIdx.x, gridDim.x);
}

template <class R>
__device__ __forceinline__ void alloc_sum_batch(const BoxDev* bxs, int B, uint32_t k0, uint32_t k1, DevScalars* gsc,
                                                unsigned long long* partQ, uint32_t g, uint32_t ng) {
  const int b = alloc_box(bxs, B, g);
  const BoxDev& d = bxs[b];
  const R rmax = (R)__ldcg(&d.sc->rmax);
  velq_write<R, kAllocItems>((const typename Vec4<R>::T*)d.vel4, d.n3, (int64_t)(g - d.ablk0) * kAllocChunk, __ldcg(&d.sc->vq_u),
                d.velq, d.vbx, Tiles{d.n, d.nt, d.lg, d.mn, d.mn2, d.tlg});
  uint64_t acc = 0;
  if (rmax > (R)0) {
    const int64_t c0 = (int64_t)(g - d.ablk0) * kAllocChunk + (int64_t)threadIdx.x * kAllocItems;
    R v[kAllocItems];
    load_items<R, kAllocItems>((const R*)d.emis, c0, d.n3, v);
#pragma unroll
    for (int k = 0; k < kAllocItems; ++k) {
      const uint64_t q = quantised<R>(v[k], rmax);
      acc += q;
      if (kKeepQ<R> && c0 + k < d.n3) d.P[c0 + k] = (uint32_t)q;
    }
  }
  uint64_t incl;
  uint64_t tot = block_scan_incl(acc, &incl);
  if (threadIdx.x == 0) partQ[g] = tot;
  if (!last_block_done(&gsc->alloc_counter, ng)) return;
  // one warp per box: exclusive scan of its block sums (in place), the
  // systematic-sampling offset and the box's packet total
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = warp; i < B; i += AT / 32) {
    const BoxDev& e = bxs[i];
    const uint32_t g0 = e.ablk0;
    const uint32_t g1 = (i + 1 < B) ? bxs[i + 1].ablk0 : ng;
    uint64_t run = 0;
    for (uint32_t gb = g0; gb < g1; gb += 32) {
      const uint32_t g = gb + lane;
      uint64_t q = g < g1 ? __ldcg(&partQ[g]) : 0ull, v = q;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        uint64_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
      }
      if (g < g1) partQ[g] = run + v - q;
      run += __shfl_sync(0xffffffffu, v, 31);
    }
    if (lane == 0) {
      DevScalars* sc = e.sc;
      const uint64_t sumQ = run;
      U4 r = draw(Stream{k0, k1, (uint32_t)i}, 0u, 0u, kAllocBlock);
      uint64_t w = ((uint64_t)r.b << 32) | r.a;
      uint64_t npk = (sumQ > 0) ? e.npk : 0;
      set_divisor(sc, sumQ);
      sc->alloc_u = sumQ > 0 ? w % sumQ : 0;
      e.P[e.n3] = (uint32_t)npk;
      sc->emitted = npk;
      sc->absorbed = 0;
      sc->capped = 0;
      sc->crossings = 0;
      sc->qtail = 0;
      if (sumQ == 0 && e.npk > 0) sc->flags |= 4;
    }
  }
  if (threadIdx.x == 0) gsc->alloc_counter = 0;
}
template <class R>
__global__ void __launch_bounds__(AT) k_alloc_sum_batch(const BoxDev* bxs, int B, uint32_t k0, uint32_t k1,
                                                        DevScalars* gsc, unsigned long long* partQ) {
  alloc_sum_batch<R>(bxs, B, k0, k1, gsc, partQ, blockIdx.x, gridDim.x);
}

template <class R>
__device__ __forceinline__ void alloc_prefix_batch(const BoxDev* bxs, int B, const unsigned long long* partQ,
                                                   unsigned long long* bcap, uint32_t g) {
  const int b = alloc_box(bxs, B, g);
  const BoxDev& d = bxs[b];
  const DevScalars* sc = d.sc;
  const int64_t c0 = (int64_t)(g - d.ablk0) * kAllocChunk + (int64_t)threadIdx.x * kAllocItems;
  const Divisor dv{__ldcg(&sc->sumQ), __ldcg(&sc->div_v), __ldcg(&sc->div_m), __ldcg(&sc->div_shift)};
  alloc_prefix_block<R, kAllocItems>((const R*)d.emis, d.n3, d.npk, dv, __ldcg(&sc->alloc_u), (R)__ldcg(&sc->rmax),
                                     __ldcg(&partQ[g]), c0, d.P, d.first,
                                     Tiles{d.n, d.nt, d.lg, d.mn, d.mn2, d.tlg}, d.bk0, bcap);
}
template <class R>
__global__ void __launch_bounds__(AT) k_alloc_prefix_batch(const BoxDev* bxs, int B, const unsigned long long* partQ,
                                                           unsigned long long* bcap) {
  alloc_prefix_batch<R>(bxs, B, partQ, bcap, blockIdx.x);
}

// Emission over the batch packet space (each box padded to a multiple of 64,
// so a warp's 64-packet window belongs to one box): the ring is flushed at each change of
// box; one cell-coordinate path (exact multiply-high divisions) for every side keeps
// the kernel within its registers.  FRESH: the packet prefixes and box scalars were
// written earlier in the same launch (read through L2).
template <class R, bool FRESH>
__device__ __forceinline__ void emit_batch_body(const TransportArgs<R>& a, const BoxDev* bxs, const BoxStep* bst,
                                                     int B, uint64_t tot_pk) {
  using V = typename Vec4<R>::T;
  __shared__ BoxCounters cnt;
  __shared__ EmitStash<R> stash[TT / 32];
  EmitStash<R>& st = stash[threadIdx.x >> 5];
  box_counters_clear(cnt, B);
  uint64_t my_abs = 0, my_cross = 0;
  int cur = -1;
  uint64_t lo_pk = 1, hi_pk = 0;  // packet range of box cur (empty before the first lookup)
  uint32_t N = 0;
  uint32_t head = 0, count = 0;   // the warp's ring of packets waiting for their direction
  auto box_of = [&](int b) {
    const BoxDev& d = bxs[b];
    return EmitBox<R>{d.P, d.first, (uint32_t)d.n3, d.n, (const V*)d.vel4, (const R*)d.T, d.tally,
                      (R)__ldcg(&bst[b].kappa), (R)__ldcg(&bst[b].cth),
                      (uint32_t)b, Tiles{d.n, d.nt, d.lg, d.mn, d.mn2, d.tlg}, d.bk0,
                      __ldcg(&d.sc->vel_plain) ? a.early : 0u};
  };
  const uint64_t warps_total = (uint64_t)gridDim.x * (TT / 32);
  for (uint64_t gbase = ((uint64_t)blockIdx.x * (TT / 32) + (threadIdx.x >> 5)) * 64; gbase < tot_pk;
       gbase += warps_total * 64) {
    if (gbase < lo_pk || gbase >= hi_pk) {  // next box (uniform over the warp)
      if (count) emit_flush<R, false>(a, box_of(cur), st, head, count, my_abs, my_cross);
      const int b = last_le(B, gbase, [&](int i) { return bxs[i].pk0; });
      if (cur >= 0) box_counters_add(cnt, cur, my_abs, 0, my_cross);
      my_abs = my_cross = 0;
      cur = b;
      lo_pk = bxs[b].pk0;
      hi_pk = (b + 1 < B) ? bxs[b + 1].pk0 : tot_pk;
      N = ld_index<FRESH>(bxs[b].P + bxs[b].n3);  // packets actually allocated to this box
    }
    const uint64_t base = gbase - lo_pk;
    if (base >= N) continue;  // padding of the packet space
    emit_window64<R, false, FRESH>(a, box_of(cur), st, (uint32_t)base, N, head, count, my_abs, my_cross);
  }
  if (count) emit_flush<R, false>(a, box_of(cur), st, head, count, my_abs, my_cross);
  if (cur >= 0) box_counters_add(cnt, cur, my_abs, 0, my_cross);
  box_counters_flush(cnt, bxs, B);
}

template <class R>
__global__ void __launch_bounds__(TT, sizeof(R) == 4 ? 4 : 3) k_emit_batch(TransportArgs<R> a, const BoxDev* bxs, const BoxStep* bst,
                                                      int B, uint64_t tot_pk) {
  emit_batch_body<R, false>(a, bxs, bst, B, tot_pk);
}

__global__ void k_set_box_step(BoxStepArgs p, BoxStep* out, int B) {
  for (int b = threadIdx.x; b < B; b += blockDim.x) out[b] = p.s[b];
}

__device__ __forceinline__ void transport_end_batch(const BoxDev* bxs, int B, const unsigned long long* bfill,
                                                    rec_stats* st) {
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    const BoxDev& d = bxs[b];
    DevScalars* sc = d.sc;
    unsigned long long q = 0;
    const uint32_t nb = d.nt * d.nt * d.nt;
    for (uint32_t k = 0; k < nb; ++k) q += __ldcg(&bfill[d.bk0 + k]);
    // the counters were added by other blocks' atomics: read them through L2
    const unsigned long long absorbed = __ldcg(&sc->absorbed), capped = __ldcg(&sc->capped);
    sc->qtail = q;
    sc->tally_total = __ldcg(&sc->tally_total) + absorbed;
    if (capped) atomicOr(&sc->flags, 2);
    if (st) {
      st[b].emitted = __ldcg(&sc->emitted);
      st[b].absorbed = absorbed;
      st[b].capped = capped;
      st[b].crossings = __ldcg(&sc->crossings);
      st[b].queued = q;
      st[b].requeued = 0;
      st[b].flags = __ldcg(&sc->flags);
    }
  }
}

// The allocation and the emission of a batched transport call as phases of
// one persistent cooperative launch, separated by bounded grid barriers: box
// transport scalars, bucket capacities cleared and the allocation maxima;
// quantised sums and their scans; packet prefixes; bucket offsets; emission;
// march chunk prefix.  The allocation phases run the allocation blocks of the
// per-phase kernels as virtual blocks.  A barrier that gives up ends the launch
// (flags bit 3 of the batch record) and the march that follows finds no work.
template <class R>
__global__ void __launch_bounds__(AT, sizeof(R) == 4 ? 4 : 3) k_batch_front(TransportArgs<R> a, const BoxDev* bxs, BoxStep* bst,
                                                       BoxStepArgs bs, int B, uint32_t k0, uint32_t k1,
                                                       DevScalars* gsc, unsigned long long* partQ, unsigned long long* cpre,
                                                       uint32_t n_ablk, uint64_t tot_pk,
                                                       uint32_t limit) {
  if (blockIdx.x == 0)
    for (int b = threadIdx.x; b < B; b += AT) bst[b] = bs.s[b];
  for (int i = blockIdx.x * AT + threadIdx.x; i < a.nb; i += gridDim.x * AT) a.boff[i] = 0ull;
  if (blockIdx.x == 0 && threadIdx.x == 0) gsc->march_next = ~0ull >> 1;  // no march work until the chunks exist
  for (uint32_t g = blockIdx.x; g < n_ablk; g += gridDim.x) alloc_max_batch<R>(bxs, bs, B, gsc, g, n_ablk);
  if (!grid_barrier(&gsc->bar, &gsc->flags, limit)) return;
  for (uint32_t g = blockIdx.x; g < n_ablk; g += gridDim.x) alloc_sum_batch<R>(bxs, B, k0, k1, gsc, partQ, g, n_ablk);
  if (!grid_barrier(&gsc->bar, &gsc->flags, limit)) return;
  for (uint32_t g = blockIdx.x; g < n_ablk; g += gridDim.x) alloc_prefix_batch<R>(bxs, B, partQ, a.boff, g);
  if (!grid_barrier(&gsc->bar, &gsc->flags, limit)) return;
  if (blockIdx.x == 0) bucket_offsets_block<AT>(a.boff, a.bfill, a.nb);
  if (!grid_barrier(&gsc->bar, &gsc->flags, limit)) return;
  emit_batch_body<R, true>(a, bxs, bst, B, tot_pk);
  if (!grid_barrier(&gsc->bar, &gsc->flags, limit)) return;
  if (blockIdx.x == 0) bucket_scan_block<AT>(a.bfill, cpre, a.nb, gsc, a.chunk);
}

template <class R>
cudaError_t run_transport_batch(rec_ctx* c, int step, double z, rec_stats* st) {
  const int B = c->n_boxes;
  const uint32_t k0 = (uint32_t)c->params.seed, k1 = (uint32_t)(c->params.seed >> 32) ^ (uint32_t)step;
  const int nb = c->tot_buckets;
  BoxStepArgs bs;
  for (int b = 0; b < B; ++b) transport_scalars(c->cosmo, (int)c->hbx[b].n, z, &bs.s[b].kappa, &bs.s[b].cth);
  TransportArgs<R> a;
  std::memset(&a, 0, sizeof(a));
  a.quant = (const R*)c->quant;
  a.M = c->params.n_quantiles;
  a.ks = key_schedule(k0, k1);
  double kappa_max = 0.0, cth_max = 0.0;
  for (int b = 0; b < B; ++b) {
    kappa_max = std::max(kappa_max, (double)bs.s[b].kappa);
    cth_max = std::max(cth_max, (double)bs.s[b].cth);
  }
  a.early = early_word(c, kappa_max, cth_max);
  a.sc = c->gsc;
  a.queue = (typename Vec4<R>::T*)c->queue;
  a.nb = nb;
  a.boff = c->bcap;
  a.bfill = c->bfill;
  a.cpre = c->cpre;
  a.chunk = (uint32_t)c->tune.march_chunk;
  a.refill = c->tune.march_refill;
  if (c->batch_front_grid == 0) {  // resident blocks of the persistent front (cooperative launch)
    int per_sm = 0, coop = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch_front<R>, AT, 0);
    cudaGetLastError();
    c->batch_front_grid = (e == cudaSuccess && coop && per_sm > 0) ? per_sm * c->sm_count : -1;
  }
  if (c->batch_front_grid > 0) {
    // allocation + emission in one persistent launch, then the march (which closes the call)
    GroupTimer t(c, kTEmit, 1);
    const BoxDev* bxs = c->bx;
    BoxStep* bst = c->bstep;
    DevScalars* gsc = c->gsc;
    unsigned long long* partQ = c->partQ;
    unsigned long long* cpre = c->cpre;
    uint32_t n_ablk = (uint32_t)c->tot_ablk;
    uint64_t tot_pk = c->tot_pk;
    uint32_t limit = c->wait_limit;
    int Bv = B;
    uint32_t k0v = k0, k1v = k1;
    void* args[] = {&a, &bxs, &bst, &bs, &Bv, &k0v, &k1v, &gsc, &partQ, &cpre, &n_ablk, &tot_pk, &limit};
    cudaError_t e = cudaLaunchCooperativeKernel((void*)k_batch_front<R>, c->batch_front_grid, AT, args, 0, c->stream);
    if (e != cudaSuccess) return e;
  } else {
    {
      GroupTimer t(c, kTAlloc, 5);
      k_set_box_step<<<1, kMaxBoxes, 0, c->stream>>>(bs, c->bstep, B);
      k_alloc_max_batch<R><<<c->tot_ablk, AT, 0, c->stream>>>(c->bx, bs, B, c->gsc);
      k_alloc_sum_batch<R><<<c->tot_ablk, AT, 0, c->stream>>>(c->bx, B, k0, k1, c->gsc, c->partQ);
      cudaMemsetAsync(c->bcap, 0, sizeof(unsigned long long) * nb, c->stream);
      k_alloc_prefix_batch<R><<<c->tot_ablk, AT, 0, c->stream>>>(c->bx, B, c->partQ, c->bcap);
      k_bucket_offsets<<<1, 1024, 0, c->stream>>>(c->bcap, c->bfill, nb);
    }
    {
      GroupTimer t(c, kTEmit, 2);
      k_emit_batch<R><<<c->sm_count * c->tune.emit_blocks_per_sm, TT, 0, c->stream>>>(a, c->bx, c->bstep, B,
                                                                                      c->tot_pk);
      k_bucket_scan<<<1, 1024, 0, c->stream>>>(c->bfill, c->cpre, nb, c->gsc, a.chunk);
    }
  }
  {
    GroupTimer t(c, kTMarch, 1);
    march_launch<R, false, true, false>(c, a, c->sm_count * c->tune.march_blocks_per_sm, c->bx, B, c->bstep, st);
  }
  return cudaGetLastError();
}

}  // namespace

int alloc_blocks_single(int64_t n3) {
  const int64_t cells = (int64_t)AT * alloc_items(n3);
  return (int)((n3 + cells - 1) / cells);
}

// Largest resident blocks per SM of the emission and the march (their
// launch bounds), for the checks of rec_set_tuning.
int sweep_march_limit(bool mixed) {
  return mixed ? march_occupancy<float, false, true>() : march_occupancy<double, false, true>();
}

void transport_limits(bool mixed, bool batch, int* emit_max, int* march_max) {
  *emit_max = batch ? 4 : (mixed ? emit_occupancy<float>() : emit_occupancy<double>());
  *march_max = batch ? march_occupancy<float, true>()
                     : (mixed ? march_occupancy<float, false>() : march_occupancy<double, false>());
}

cudaError_t launch_transport(rec_ctx* c, int step, double z, rec_stats* st) {
  if (c->params.precision == REC_PREC_MIXED) return run_transport<float>(c, step, z, st);
  return run_transport<double>(c, step, z, st);
}

cudaError_t launch_transport_batch(rec_ctx* c, int step, double z, rec_stats* st) {
  if (c->params.precision == REC_PREC_MIXED) return run_transport_batch<float>(c, step, z, st);
  return run_transport_batch<double>(c, step, z, st);
}

}  // namespace rec
