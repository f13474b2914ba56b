// Device helpers shared by the particle-mesh kernels: the fixed-point CIC coordinates.
#pragma once
#include "cola_internal.cuh"

namespace cola {

// v / np as a multiply-high and shifts (set_np_divider): integer-pipe instructions only
__device__ __forceinline__ unsigned div_np(const Geometry& g, unsigned v) {
  const unsigned t = __umulhi(g.np_mul, v);
  return (t + ((v - t) >> g.np_sh1)) >> g.np_sh2;
}

// Lattice index of particle p = (iz np + iy) np + ix.
__device__ __forceinline__ void lattice_index(const Geometry& g, int64_t p, int& ix, int& iy, int& iz) {
  if (g.np3 <= 0xFFFFFFFFLL) {
    const unsigned pu = (unsigned)p, n = (unsigned)g.np;
    const unsigned r = div_np(g, pu);
    ix = (int)(pu - r * n);
    iz = (int)div_np(g, r);
    iy = (int)(r - (unsigned)iz * n);
  } else {
    const int64_t r = p / g.np;
    ix = (int)(p - r * g.np);
    iz = (int)(r / g.np);
    iy = (int)(r - (int64_t)iz * g.np);
  }
}

// Fixed-point coordinate of one axis (the library's CIC quantisation, shared bit for bit
// with the deposit test oracle):
//   f = (floor(i ng 2^F / np) + floor(fl32(s * fl32(ng/L)) * 2^F)) mod (ng 2^F)
// returns the cell (f >> F) and the upper-neighbour weight t = f mod 2^F.
__device__ __forceinline__ void fixed_axis(const Geometry& g, int i, float s, int& cell, int& t) {
  const float w = __fmul_rn(s, g.scale32);
  // 2^F from its bit pattern (no 64-bit integer conversion); exact power-of-two scaling
  const float ws = __fmul_rn(w, __int_as_float((127 + g.fbits) << 23));
  if (g.fast32 && fabsf(ws) < 4194304.0f) {
    // the same in 32 bits: the lattice offset is below ng 2^F <= 2^30 and |floor(ws)| < 2^22 <=
    // ng 2^F, so f lies in (-2^22, 2^30 + 2^22) and one wrap brings it into [0, ng 2^F).
    // floor(ws) without a conversion instruction: ws + 1.5 2^23 rounded down lies in
    // [2^23, 2^24), where floats are the integers and their bit patterns consecutive.
    // One form of the lattice offset for every np: with a branch between i (ng / np) 2^F and two
    // multiply-high divisions the compiler kept the axes' loads apart (density's adjoint of 384^3
    // particles 1082 -> 1099 us with the branch; density of 384^3 on 512^3 1487 us, 1366 without).
    const int period = g.ng << g.fbits;
    const int q = (int)(((uint64_t)(unsigned)i * g.lattice_step) >> 32);
    int f = q + (__float_as_int(__fadd_rd(ws, 12582912.0f)) - 0x4B400000);
    if (f < 0) f += period;
    else if (f >= period) f -= period;
    cell = f >> g.fbits;
    t = f & ((1 << g.fbits) - 1);
    return;
  }
  const int64_t one = 1LL << g.fbits;
  const int64_t period = (int64_t)g.ng << g.fbits;
  const int64_t q = g.ratio ? ((int64_t)i * g.ratio) << g.fbits : (((int64_t)i * g.ng) << g.fbits) / g.np;
  int64_t f;
  if (fabsf(ws) < 4194304.0f) {
    f = q + (int64_t)(__float_as_int(__fadd_rd(ws, 12582912.0f)) - 0x4B400000);
  } else {
    f = q + (int64_t)floorf(ws);
  }
  if (f < 0) f += period;
  if (f >= period) f -= period;
  if (f < 0 || f >= period) {  // displacement beyond one box length
    f %= period;
    if (f < 0) f += period;
  }
  cell = (int)(f >> g.fbits);
  t = (int)(f & (one - 1));
}

__device__ __forceinline__ int wrap_inc(int c, int n) { return c + 1 == n ? 0 : c + 1; }

// float32 nearest to v (ties to even), v < 2^62, as __ull2float_rn but with 32-bit integer and
// float32 instructions only (a 64-bit conversion runs on the narrow float64 pipe of sm_103a):
// with lz leading zeros in the high word, m = the 32 bits of v from its leading one down, its
// lowest bit ORed with every bit below them (sticky); m's rounding to 24 bits is v's rounding,
// and the scale 2^(32 - lz) is exact.
__device__ __forceinline__ float u64_to_f32_rn(unsigned long long v) {
  const unsigned lo = (unsigned)v, hi = (unsigned)(v >> 32);
  const unsigned lz = __clz(hi);                       // 32 if hi == 0
  unsigned m = __funnelshift_lc(lo, hi, lz);           // top 32 bits of v << lz (lo when lz = 32)
  m |= __funnelshift_lc(0u, lo, lz) != 0u ? 1u : 0u;   // bits of lo shifted out below m
  return __fmul_rn(__uint2float_rn(m), __int_as_float((int)(127 + 32 - lz) << 23));
}

// Exact 64-bit accumulation in shared memory held as two 32-bit words per cell, the low words
// in one array and the high words in another: the low word is added with carry detection (the
// atomic returns the previous value; the add wrapped iff the new value is below it) and the
// high word receives the upper half plus that carry.  lo[i] + 2^32 hi[i] is the 64-bit sum
// modulo 2^64, whatever the order of the adds.  Two 32-bit shared atomics run at about twice
// the rate of one 64-bit shared atomic on sm_103a.
__device__ __forceinline__ void acc_add64(unsigned* lo, unsigned* hi, int i, unsigned long long w) {
  const unsigned l = (unsigned)w, h = (unsigned)(w >> 32);
  const unsigned old = atomicAdd(lo + i, l);
  const unsigned up = h + ((old + l < old) ? 1u : 0u);
  if (up) atomicAdd(hi + i, up);
}
// The cloud of one particle into the rows of a tile of TY x TZ rows from (y0, z0), rows of n cells
// (lo, hi as above): f its fixed-point coordinates, F = fbits.  BATCH: the low words of all the
// cloud's cells are added before the first high word needs a carry, eight atomics in flight per
// thread instead of one or two.  A block of one or two warps with a clump in its tile is bound by
// their latency (256^3 mesh, 192^3 clustered particles: 272 -> 248 us); larger blocks hide it and
// are better off with the fewer registers (512^3 mesh and particles, 2455 us, batched 2503).
template <int TY, int TZ, bool BATCH>
__device__ __forceinline__ void acc_cloud(unsigned* lo, unsigned* hi, const uint32_t (&f)[3], int fbits, int n, int y0,
                                          int z0) {
  const uint32_t one = 1u << fbits, fmask = one - 1u;
  const int cx = (int)(f[0] >> fbits), cy = (int)(f[1] >> fbits), cz = (int)(f[2] >> fbits);
  const uint32_t tx = f[0] & fmask, ty = f[1] & fmask, tz = f[2] & fmask;
  const int cx1 = wrap_inc(cx, n);
  if constexpr (BATCH) {
    int row[4];  // first cell of the tile's row of corner (dz, dy), -1 outside the tile
    unsigned long long w[4][2];
    unsigned old[4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int dz = k >> 1, dy = k & 1;
      const int lz = (dz ? wrap_inc(cz, n) : cz) - z0, ly = (dy ? wrap_inc(cy, n) : cy) - y0;
      row[k] = (unsigned)lz < (unsigned)TZ && (unsigned)ly < (unsigned)TY ? (lz * TY + ly) * n : -1;
      // (products of three weights of at most 2^F each)
      const unsigned long long wzy = (unsigned long long)(dz ? tz : one - tz) * (dy ? ty : one - ty);
      w[k][0] = wzy * (one - tx);
      w[k][1] = wzy * tx;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (row[k] >= 0) {
        old[k][0] = atomicAdd(lo + row[k] + cx, (unsigned)w[k][0]);
        old[k][1] = atomicAdd(lo + row[k] + cx1, (unsigned)w[k][1]);
      }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (row[k] >= 0) {
        const unsigned u0 = (unsigned)(w[k][0] >> 32) + (old[k][0] + (unsigned)w[k][0] < old[k][0] ? 1u : 0u);
        const unsigned u1 = (unsigned)(w[k][1] >> 32) + (old[k][1] + (unsigned)w[k][1] < old[k][1] ? 1u : 0u);
        if (u0) atomicAdd(hi + row[k] + cx, u0);
        if (u1) atomicAdd(hi + row[k] + cx1, u1);
      }
  } else {
    const unsigned long long wx0 = one - tx, wx1 = tx;
#pragma unroll
    for (int dz = 0; dz < 2; ++dz) {
      const int lz = (dz ? wrap_inc(cz, n) : cz) - z0;
      if (lz < 0 || lz >= TZ) continue;
      const unsigned long long wz = dz ? (unsigned long long)tz : one - tz;
#pragma unroll
      for (int dy = 0; dy < 2; ++dy) {
        const int ly = (dy ? wrap_inc(cy, n) : cy) - y0;
        if (ly < 0 || ly >= TY) continue;
        const unsigned long long wzy = wz * (dy ? (unsigned long long)ty : one - ty);
        const int row = (lz * TY + ly) * n;
        acc_add64(lo, hi, row + cx, wzy * wx0);
        acc_add64(lo, hi, row + cx1, wzy * wx1);
      }
    }
  }
}

}  // namespace cola
