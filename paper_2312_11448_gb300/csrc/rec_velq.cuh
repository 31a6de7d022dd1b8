// Compact velocity copy of the march: one signed byte per component, one
// 32-bit word per cell, in bricks.
//
// A marching packet is absorbed in the first cell with u0 - kappa n.U <= s
// (s its exit distance).  Almost every cell fails that test by a wide margin,
// so the march first asks a bound: with U ~ (u / 127) q, q integer in
// [-127, 127], and kappa n ~ (kappa / 127) m, the integer dot product m.q
// decides, and the exact velocity is read only where the bound cannot exclude
// absorption (about once per packet).  The results are those of the exact
// test, bit for bit: the copy only removes loads.
//
// A word per cell instead of a 16- or 32-byte vector makes the copy of a
// 256^3 box 67 MB (the vectors: 268 / 537 MB), which the 126 MB L2 holds, and the
// brick order puts 2 x 2 x 2 cells into a 32-byte sector and 4 x 4 x 2 into a
// 128-byte line, so that a ray stays about two cells in a sector whatever its
// direction.  Word index of cell (ix, iy, iz):
//   bits 0..2: ix0 iy0 iz0; bits 3, 4: ix1 iy1; then ix >> 2 (bx bits),
//   iy >> 2 (bx bits), iz >> 1.
// Every axis owns a fixed set of index bits, so that a step along an axis is
// an addition with a mask (the carry runs through the gaps) and no other
// coordinate has to be known.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rec {

// bits of the brick coordinates: 4 << bx >= n
__host__ __device__ inline uint32_t velq_bits(uint32_t n) {
  uint32_t b = 0;
  while ((4u << b) < n) ++b;
  return b;
}
__host__ __device__ inline uint32_t velq_x(uint32_t ix) { return (ix & 1u) | ((ix & 2u) << 2) | ((ix >> 2) << 5); }
__host__ __device__ inline uint32_t velq_y(uint32_t iy, uint32_t bx) {
  return ((iy & 1u) << 1) | ((iy & 2u) << 3) | ((iy >> 2) << (5u + bx));
}
__host__ __device__ inline uint32_t velq_z(uint32_t iz, uint32_t bx) {
  return ((iz & 1u) << 2) | ((iz >> 1) << (5u + 2u * bx));
}
// Words of the copy of an n^3 box (n <= 1024: at most 2^30).  x and y are padded to a power of
// two, so n^3 words for such sides and up to four times as many just above one.
__host__ __device__ inline uint64_t velq_words(uint32_t n) {
  return (uint64_t)((n + 1u) >> 1) << (5u + 2u * velq_bits(n));
}
// Cell coordinates of a word index.
__host__ __device__ inline void velq_coords(uint32_t o, uint32_t bx, uint32_t* ix, uint32_t* iy, uint32_t* iz) {
  const uint32_t m = (1u << bx) - 1u;
  *ix = (o & 1u) | ((o >> 2) & 2u) | (((o >> 5) & m) << 2);
  *iy = ((o >> 1) & 1u) | ((o >> 3) & 2u) | (((o >> (5u + bx)) & m) << 2);
  *iz = ((o >> 2) & 1u) | ((o >> (5u + 2u * bx)) << 1);
}

// Stepping masks of the three axes.  Power-of-two sides: the bits in use, so
// that the addition wraps periodically.  Other sides: every bit of the axis;
// the wrap is a comparison with the last cell's offset.
struct VelqMasks {
  uint32_t x, y, z;
};
__host__ __device__ inline VelqMasks velq_masks(uint32_t n, uint32_t bx, bool p2) {
  if (p2) return VelqMasks{velq_x(n - 1u), velq_y(n - 1u, bx), velq_z(n - 1u, bx)};
  const uint32_t x = velq_x((4u << bx) - 1u), y = velq_y((4u << bx) - 1u, bx);
  return VelqMasks{x, y, ~(x | y)};
}

// The integer dot product of four signed bytes, added to c.
__device__ __forceinline__ int velq_dot(uint32_t a, uint32_t b, int c) { return __dp4a((int)a, (int)b, c); }

// Quantised velocity: components rounded to units of u / 127 (qs = 127 / u),
// |component| <= u.  An error of half a unit per component, plus rounding.
__device__ __forceinline__ uint32_t velq_pack(float x, float y, float z, float qs) {
  const int a = __float2int_rn(fminf(fmaxf(x * qs, -127.0f), 127.0f));
  const int b = __float2int_rn(fminf(fmaxf(y * qs, -127.0f), 127.0f));
  const int c = __float2int_rn(fminf(fmaxf(z * qs, -127.0f), 127.0f));
  return ((uint32_t)a & 0xffu) | (((uint32_t)b & 0xffu) << 8) | (((uint32_t)c & 0xffu) << 16);
}
// Word of a cell with a component beyond u, or not finite: always a candidate.
constexpr uint32_t kVelqOut = 0x80000000u;
__device__ __forceinline__ bool velq_is_out(uint32_t w) { return (int)w < 0; }

// Scale of the copy for a box with largest |component| umax and mean |component|
// `mean` (of the cells that are finite): umax, but at most 16 means, so that a few fast cells
// do not coarsen the unit of all others (they are marked as kVelqOut instead; a
// Gaussian flow, whose largest component is about 7 means, has none; by Markov's
// inequality at most 3/16 of the cells are beyond).  256^3 mixed, 1e8 packets, 1 km/s: march 3.5 ms, and
// with one cell of 30 / 300 / 3e4 km/s 3.9 ms each (by umax alone 4.4 / 15.3 / 24.4); speeds that
// vary by a log-normal factor of width 1.5 from cell to cell: 16.2 -> 6.9 ms.
// Never below 0.1 cells of Hubble drift, so that the unit of the integer test
// stays representable when there is hardly any flow.  0: no usable copy.
__device__ __forceinline__ float velq_scale(float umax, float mean, float kappa) {
  if (!(kappa > 1e-15f) || !(kappa < 1e15f)) return 0.0f;
  const float u = fmaxf(fminf(umax, 16.0f * mean), 0.1f / kappa);
  return u < 1e15f ? u : 0.0f;
}

// The per-packet bound.  In units of kappa u / 127^2 cells (c1 units per cell) the
// packet is a candidate for absorption in a cell with exit distance s only if
//   kBias + m.q >= c2 - c1 s     (compared as the bits of binary32 numbers),
// where c2 = kBias + c1 u0 - slack and kBias = 1.5 2^23: integers up to 2^22 around
// it are exact, and binary32 bit patterns of positive numbers order as signed
// integers (negative ones below all of them), so one integer comparison of
// the dot product, started at kBias' bits, with the bits of c2 - c1 s decides.
// slack covers, in those units:
//   - the packet's rounded direction, |kappa n_i - (kappa/127) m_i| u per component (exact per packet),
//   - half a unit of velocity per component against |kappa n_i|,
//   - the rounding of the exact test itself, of c1, c2 and of c2 - c1 s: relative
//     2^-20 of c1 u0 and 4 units (each operation rounds to 2^-24 relative, and
//     c1 s exceeds c1 |u0| + 127^2 sqrt 3 only where every cell is a candidate anyway).
// top: no dot product of this packet with any cell exceeds it (the packet's own
// bytes against 127 each, or the largest speed of the box), so that a cell
// with c2 - c1 s beyond it needs no load at all.  Where cells are beyond the scale it
// is the largest speed that bounds them (c2 - c1 s, in units above the bias, is no less than
// the bits' distance from it, so the comparison by bits errs towards loading).
constexpr int kVelqBiasBits = 0x4B400000;
struct VelqPacket {
  uint32_t m;      // rounded direction, one signed byte per component
  float c1, c2;
  int top;         // kVelqBiasBits + largest possible dot product
};
struct VelqBox {
  float u, v, kinv, kq, c1;  // scale, largest speed, 127 / kappa, kappa / 127, 127^2 / (kappa u)
};
__device__ __forceinline__ VelqBox velq_box(float u, float v, float kappa) {
  VelqBox b;
  b.u = u;
  b.v = v;
  b.kinv = 127.0f / kappa;
  b.kq = kappa * (1.0f / 127.0f);
  b.c1 = u > 0.0f ? 16129.0f / (kappa * u) : 0.0f;
  return b;
}
// OUT: some cells (of any box of a batch) are beyond the scale.
template <bool OUT>
__device__ __forceinline__ VelqPacket velq_packet(const VelqBox& b, float kx, float ky, float kz, float u0) {
  VelqPacket p;
  if (!(b.u > 0.0f)) {  // no copy: every cell is a candidate, nothing is loaded from it
    p.m = 0u;
    p.c1 = 0.0f;
    p.c2 = -1.0f;
    p.top = (int)0x80000000;
    return p;
  }
  const float mx = rintf(kx * b.kinv), my = rintf(ky * b.kinv), mz = rintf(kz * b.kinv);
  p.m = ((uint32_t)(int)mx & 0xffu) | (((uint32_t)(int)my & 0xffu) << 8) | (((uint32_t)(int)mz & 0xffu) << 16);
  const float err = fabsf(kx - mx * b.kq) + fabsf(ky - my * b.kq) + fabsf(kz - mz * b.kq);
  const float sum = fabsf(kx) + fabsf(ky) + fabsf(kz);
  const float slack = b.c1 * b.u * (err + sum * (0.501f / 127.0f)) * 1.001f + 4.0f + fabsf(u0) * b.c1 * 0x1p-20f;
  p.c1 = b.c1;
  p.c2 = 12582912.0f + (u0 * b.c1 - slack);
  const float own = 127.0f * (fabsf(mx) + fabsf(my) + fabsf(mz));
  // |kappa n| <= 1.00001 kappa; the dot product differs from c1 kappa n.U by less than slack
  const float box = b.c1 * b.v * (b.kq * 127.0f) * 1.0001f + slack + 2.0f;
  if (OUT) p.top = box < 8e8f ? kVelqBiasBits + (int)box : 0x7fffffff;
  else p.top = kVelqBiasBits + (int)fminf(own, box);
  return p;
}

}  // namespace rec
