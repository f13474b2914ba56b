// Device bodies of the mesh passes, shared by the single-box kernels and the multi-box
// (ensemble) kernels.  Each body processes one block's share of work given by explicit block
// indices and shared-memory pointers, so that a persistent kernel can run the bodies of
// different boxes (and mesh sizes) one after another.
#pragma once
#include "cola_internal.cuh"
#include "fft.cuh"
#include "pm_common.cuh"
#include "tma.cuh"
#include "tmem.cuh"

namespace cola {

// ---- helpers -----------------------------------------------------------------------------
__device__ __forceinline__ float sinc_pi_f(int n, int ng) {
  if (n == 0) return 1.0f;
  const float x = (float)n / (float)ng;
  return sinpif(x) / (3.14159265358979323846f * x);
}
__device__ __forceinline__ int signed_mode(int k, int n) { return k < n / 2 ? k : k - n; }

// first-derivative factor i k_j (zero on the Nyquist plane |n_j| = N/2)
__device__ __forceinline__ float2 mul_ik(float2 a, float k) { return make_float2(__fmul_rn(-k, a.y), __fmul_rn(k, a.x)); }

// ---- one or two columns per thread ---------------------------------------------------------
// The strided (column) passes run on strips of W columns, V = float2: one column per thread, V =
// cpair: two neighbouring columns per thread (fft.cuh).  A half spectrum's rows start on 32-byte
// boundaries and are padded to a multiple of 4 entries, so the pair that holds the last column
// (an even one, N/2) has its other lane in the padding, and pairs are 16-byte aligned.
template <class V>
__host__ __device__ constexpr int lanes_of() {
  return (int)(sizeof(V) / sizeof(float2));
}
__device__ __forceinline__ cpair c_interleave(float4 q) { return {make_float2(q.x, q.z), make_float2(q.y, q.w)}; }
__device__ __forceinline__ float4 c_deinterleave(cpair v) { return make_float4(v.re.x, v.im.x, v.re.y, v.im.y); }
template <class V>
__device__ __forceinline__ V c_load(const float2* p) {
  if constexpr (lanes_of<V>() == 1) return *p;
  else return c_interleave(*reinterpret_cast<const float4*>(p));
}
template <class V>
__device__ __forceinline__ V c_load_cg(const float2* p) {
  if constexpr (lanes_of<V>() == 1) return __ldcg(p);
  else return c_interleave(__ldcg(reinterpret_cast<const float4*>(p)));
}
template <class V>
__device__ __forceinline__ V c_zero() {
  return V{};
}
__device__ __forceinline__ void c_store(float2* p, float2 v) { *p = v; }
__device__ __forceinline__ void c_store(float2* p, cpair v) { *reinterpret_cast<float4*>(p) = c_deinterleave(v); }
__device__ __forceinline__ void c_store_cg(float2* p, float2 v) { __stcg(p, v); }
__device__ __forceinline__ void c_store_cg(float2* p, cpair v) { __stcg(reinterpret_cast<float4*>(p), c_deinterleave(v)); }
// first-derivative factor i k of both lanes
__device__ __forceinline__ cpair mul_ik(cpair a, float k) {
  return {p_mul_rn(p_dup(-k), a.im), p_mul_rn(p_dup(k), a.re)};
}

// row pitch (complex entries) of a half spectrum of an N^3 mesh: N/2 + 1 rounded up to a multiple
// of 4 (32-byte rows, the alignment the bulk copies need)
template <int N>
__host__ __device__ constexpr int half_pitch() {
  return ((N / 2 + 1) + 3) / 4 * 4;
}

// Strip width (columns per block), slabs per block, threads and resident blocks per SM of the
// single-box column passes, two columns per thread: 16 columns are 128-byte row segments, 8 where
// a strip of 16 would leave room for fewer than two blocks in shared memory.  The registers of E
// complex pairs (4 E) set the threads per SM.
template <int N>
__host__ __device__ constexpr int cols_width() {
  return N >= 512 ? 8 : 16;
}
// two slabs per block where one makes a block of one or two warps whose parked words take a
// quarter of the tensor memory
template <int N>
__host__ __device__ constexpr int cols_slabs() {
  return N == 192 || N == 96 ? 2 : 1;
}
template <int N>
__host__ __device__ constexpr int cols_threads() {
  return FFTConf<N>::T * cols_width<N>() / 2 * cols_slabs<N>();
}
template <int N>
__host__ __device__ constexpr int cols_min_blocks() {
  constexpr int E = FFTConf<N>::E, threads = cols_threads<N>();
  constexpr int per_sm = (E >= 24 ? 384 : (E >= 12 ? 512 : 768)) / threads;
  // (and no more blocks than have their parked words in the tensor memory at once)
  constexpr int parked = 512 / tmem_columns(threads, (4 * E + 15) / 16 * 16);
  return per_sm < 1 ? 1 : (per_sm < parked ? per_sm : parked);
}
// one thread's E elements, parked (tmem.cuh)
template <int THREADS, int E, class V>
using Park = TmemPark<THREADS, (E * lanes_of<V>() * 2 + 15) / 16 * 16>;
template <class P, int E, class V>
__device__ __forceinline__ void park_store(const P& park, const V (&u)[E]) {
  uint32_t r[(sizeof(u) / 4 + 15) / 16 * 16] = {};
#pragma unroll
  for (int m = 0; m < E; ++m) {
    if constexpr (lanes_of<V>() == 1) {
      r[2 * m] = __float_as_uint(u[m].x);
      r[2 * m + 1] = __float_as_uint(u[m].y);
    } else {
      r[4 * m] = __float_as_uint(u[m].re.x);
      r[4 * m + 1] = __float_as_uint(u[m].re.y);
      r[4 * m + 2] = __float_as_uint(u[m].im.x);
      r[4 * m + 3] = __float_as_uint(u[m].im.y);
    }
  }
  park.store(r);
}
template <class P, int E, class V>
__device__ __forceinline__ void park_load(const P& park, V (&u)[E]) {
  uint32_t r[(sizeof(u) / 4 + 15) / 16 * 16];
  park.load(r);
#pragma unroll
  for (int m = 0; m < E; ++m) {
    if constexpr (lanes_of<V>() == 1)
      u[m] = make_float2(__uint_as_float(r[2 * m]), __uint_as_float(r[2 * m + 1]));
    else
      u[m] = V{make_float2(__uint_as_float(r[4 * m]), __uint_as_float(r[4 * m + 1])),
               make_float2(__uint_as_float(r[4 * m + 2]), __uint_as_float(r[4 * m + 3]))};
  }
}

// This thread's place in a block that takes W columns of each of SL slabs: columns w K .. of the
// strip, transform thread t, slab number sub; strips of the exchange buffer slab after slab.
template <int N, int W, int SL, class V, class C>
struct ColsThread {
  static constexpr int K = lanes_of<V>(), WT = W / K, T = C::T, NT = T * WT * SL;
  int w, t, sub;
  V* S;
  __device__ __forceinline__ explicit ColsThread(float2* smem) {
    const int i = threadIdx.x;
    w = i % WT;
    t = i / WT % T;
    sub = SL == 1 ? 0 : i / (WT * T);
    S = reinterpret_cast<V*>(smem) + (SL == 1 ? 0 : sub * (N * WT));
  }
  __device__ __forceinline__ V& operator()(int n) const { return S[n * WT + w]; }
};

// block (bx, slab0): W columns of SL slabs of the in-place strided FFT (T(N) * W / lanes * SL
// threads); smem: SL N W float2.  Element (n, col) at data[slab * slab_stride + n * row_stride + col].
// (tw: the base twiddle table or an SmemTw stage table)
template <int N, int W, int SL, bool INV, class V, class C = FFTConf<N>, class TW>
__device__ __forceinline__ void cols_body(float2* __restrict__ data, int64_t slab_stride, int64_t row_stride,
                                          int ncols, const TW& tw, int bx, int slab0, float2* smem) {
  const ColsThread<N, W, SL, V, C> mem(smem);
  const int col = bx * W + mem.w * mem.K;
  const bool valid = col < ncols;
  float2* base = data + (int64_t)(slab0 + mem.sub) * slab_stride + (valid ? col : 0);
  auto load = [&](int n) -> V { return valid ? c_load<V>(base + (int64_t)n * row_stride) : c_zero<V>(); };
  auto store = [&](int n, V x) {
    if (valid) c_store(base + (int64_t)n * row_stride, x);
  };
  fft_1d<N, 1, INV, C>(mem.t, tw, load, mem, store);
}

// ---- 1. deposit + x r2c -----------------------------------------------------------------------
// block: one tile of TY x TZ rows (T(N/2) * TY * TZ threads); acc: max(TY TZ N, TY TZ LD) x 8
// bytes of shared memory (the cells' low 32-bit words, then their high words; afterwards the
// rows' transform buffers); ints: 28 ints of shared memory
// rec: the bin-ordered particle records (fixed-point CIC coordinates; offsets index them directly)
// (stw: the row transform's stage twiddles, the base table tw or an SmemTw table)
template <int N, int TY, int TZ, class CM = FFTConf<N / 2>, class STW>
__device__ __forceinline__ void deposit_fftx_body(const Geometry& g, const Tiles& tl, const uint4* __restrict__ rec,
                                                  const int* __restrict__ offsets, float2* __restrict__ out, int P,
                                                  const float2* __restrict__ tw, const STW& stw, float dscale,
                                                  int* __restrict__ err, int tile, unsigned long long* acc,
                                                  int* ints) {
  constexpr int M = N / 2, T = CM::T, ROWS = TY * TZ, LD = xrow_ld<M>(), NT = T * ROWS, R0 = first_radix<CM>();
  int* rbeg = ints;
  int* rpre = ints + 9;
  int* rlen = ints + 19;
  int tyi, tzi;
  tile_of_bin(tl, tile, tyi, tzi);
  const int y0 = tyi * TY, z0 = tzi * TZ;
  for (int i = threadIdx.x; i < ROWS * N; i += NT) acc[i] = 0ull;
  // the tile's own 4 bins and the boundary bins of its 3 lower neighbours, loaded in parallel
  // (a loop: at N = 32 and 48 a block has only 8 threads)
  for (int k = threadIdx.x; k < 9; k += NT) {
    const int tym = tyi == 0 ? tl.nty - 1 : tyi - 1;
    const int tzm = tzi == 0 ? tl.ntz - 1 : tzi - 1;
    const int ty_ = (k == 4 || k == 5 || k == 8) ? tym : tyi;
    const int tz_ = k >= 6 ? tzm : tzi;
    const int reg = k < 4 ? k : ((k == 4 || k == 5) ? (k == 4 ? 1 : 3) : (k == 6 ? 2 : 3));
    const int b = tile_bin(tl, ty_, tz_) * 4 + reg;
    const int o0 = offsets[b];
    rbeg[k] = o0;
    rlen[k] = offsets[b + 1] - o0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = 0;
    for (int k = 0; k < 9; ++k) {
      rpre[k] = run;
      run += rlen[k];
    }
    rpre[9] = run;
  }
  __syncthreads();
  const int total = rpre[9];
  const unsigned long long one = 1ull << g.fbits;
  unsigned* lo = reinterpret_cast<unsigned*>(acc);
  unsigned* hi = lo + ROWS * N;
  constexpr int U = 4;  // particles in flight per thread
  const uint32_t fmask = (uint32_t)one - 1u;
  for (int base = threadIdx.x; base < total; base += NT * U) {
    uint32_t f[U][3];
    bool ok[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + u * NT;
      ok[u] = i < total;
      if (ok[u]) {
        int r = 0;
#pragma unroll
        for (int k = 1; k < 9; ++k) r += (i >= rpre[k]) ? 1 : 0;
        const uint4 q = __ldg(rec + rbeg[r] + (i - rpre[r]));
        f[u][0] = q.x;
        f[u][1] = q.y;
        f[u][2] = q.z;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!ok[u]) continue;
      const int cx = (int)(f[u][0] >> g.fbits), tx = (int)(f[u][0] & fmask);
      const int cy = (int)(f[u][1] >> g.fbits), ty = (int)(f[u][1] & fmask);
      const int cz = (int)(f[u][2] >> g.fbits), tz = (int)(f[u][2] & fmask);
      const int cx1 = wrap_inc(cx, N);
      const unsigned long long wx0 = one - tx, wx1 = tx;
#pragma unroll
      for (int dz = 0; dz < 2; ++dz) {
        const int lz = (dz ? wrap_inc(cz, N) : cz) - z0;
        if (lz < 0 || lz >= TZ) continue;
        const unsigned long long wz = dz ? (unsigned long long)tz : one - tz;
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
          const int ly = (dy ? wrap_inc(cy, N) : cy) - y0;
          if (ly < 0 || ly >= TY) continue;
          const unsigned long long wzy = wz * (dy ? (unsigned long long)ty : one - ty);
          const int row = (lz * TY + ly) * N;
          acc_add64(lo, hi, row + cx, wzy * wx0);
          acc_add64(lo, hi, row + cx1, wzy * wx1);
        }
      }
    }
  }
  __syncthreads();
  // real-to-complex FFT of each tile row; z[n] = (delta[2n], delta[2n+1]).  The transform
  // buffers overlay the accumulators: fft_1d reads all its inputs before a block barrier
  // that precedes its first shared-memory write.
  const int t = threadIdx.x % T, w = threadIdx.x / T;
  const uint2* lrow = reinterpret_cast<const uint2*>(lo + w * N);
  const uint2* hrow = reinterpret_cast<const uint2*>(hi + w * N);
  float2* buf = reinterpret_cast<float2*>(acc) + w * LD;
  bool overflow = false;
  auto load = [&](int n) -> float2 {
    const uint2 l = lrow[n], h = hrow[n];
    overflow |= ((h.x | h.y) >> 30) != 0u;
    const unsigned long long a = ((unsigned long long)h.x << 32) | l.x;
    const unsigned long long b = ((unsigned long long)h.y << 32) | l.y;
    return make_float2(fmaf(u64_to_f32_rn(a), dscale, -1.0f), fmaf(u64_to_f32_rn(b), dscale, -1.0f));
  };
  auto mem = [&](int n) -> float2& { return buf[xpad<R0>(n)]; };
  auto store = [&](int n, float2 x) { buf[xpad<R0>(n)] = x; };
  fft_1d<M, 2, false, CM>(t, stw, load, mem, store);
  if (overflow) atomicOr(err, kErrOverflow);
  __syncthreads();
  const int lz = w / TY, ly = w - lz * TY;
  float2* dst = out + ((int64_t)(z0 + lz) * N + (y0 + ly)) * P;
  // X[k] and X[M - k] from one pair Z[k], Z[M - k]: with e = (Z[k] + conj Z[M - k]) / 2,
  // d = (Z[k] - conj Z[M - k]) / 2 and p = W^k (-i d), X[k] = e + p and X[M - k] = conj(e - p)
  // (as W^(M - k) = -conj W^k); k = 0 gives X[0] and X[M] from Z[0]
  for (int k = t; k <= M / 2; k += T) {
    const float2 a = buf[xpad<R0>(k)];
    const float2 b = c_conj(buf[xpad<R0>(k == 0 ? 0 : M - k)]);
    const float2 e = c_scale(c_add(a, b), 0.5f);
    const float2 d = c_scale(c_sub(a, b), 0.5f);
    const float2 p = c_mul(__ldg(tw + k), make_float2(d.y, -d.x));
    dst[k] = c_add(e, p);
    if (2 * k != M) dst[M - k] = c_conj(c_sub(e, p));
  }
}

// ---- 3. z pass with the Green's function ------------------------------------------------------------
// Forward transform of the strip, phi = delta_k norm / (k^2 W(k)^p), then the inverse transforms
// of i k_z phi (-> Gz) and of phi (-> A, in place): one load and two stores of the strip.  A
// thread ends a transform with the elements the next one starts from, so phi stays in its
// registers and its second use is parked in tensor memory.
//
// shared-memory layout: SL strips (N W float2 each), sinc^2 tables (N + W floats, rounded up to
// 16 bytes), stage twiddle table
template <int N, int W, int SL>
__host__ __device__ constexpr int z_table_offset() {
  return SL * N * W + (N + W + 3) / 4 * 2;
}

// norm / (kf2 m2 W^p): the Green's function of one mode (wk = W(k))
__device__ __forceinline__ float green_of(int m2, float kf2, float wk, int deconv, float norm) {
  float gk = 0.0f;
  if (m2 != 0) {
    float den = kf2 * (float)m2;
    if (deconv) den *= deconv == 2 ? wk * wk : wk;
    gk = __fdividef(norm, den);  // fast reciprocal: <= 2 ulp, far below the transforms' rounding
  }
  return gk;
}

// block (bx, ky0): W columns kx of SL slabs ky (T(N) W / lanes SL threads)
template <int N, int W, int SL, class V, class C = FFTConf<N>, class P_>
__device__ __forceinline__ void z_green_body(float2* __restrict__ A, float2* __restrict__ Gz, float kf, int deconv,
                                             float norm, const float2* __restrict__ tw, int bx, int ky0, float2* sm,
                                             const P_& park) {
  constexpr int K = lanes_of<V>(), E = C::E, T = C::T, nh = N / 2 + 1, P = half_pitch<N>();
  const ColsThread<N, W, SL, V, C> mem(sm);
  float* sz2 = reinterpret_cast<float*>(sm + SL * N * W);
  float* sx2 = sz2 + N;
  float2* stab = sm + z_table_offset<N, W, SL>();
  stw_fill<C, 1>(stab, tw, threadIdx.x, mem.NT);
  const SmemTw<C> stw{stab};
  const int t = mem.t, ky = ky0 + mem.sub;
  const int kx = bx * W + mem.w * K;
  const bool valid = kx < nh;
  constexpr int64_t zstride = (int64_t)N * P;
  const int64_t at = (int64_t)ky * P + (valid ? kx : 0) + t * zstride;
  float2* a = A + at;
  float2* gz = Gz + at;
  V u[E];
#pragma unroll
  for (int m = 0; m < E; ++m) u[m] = valid ? c_load<V>(a + m * (T * zstride)) : c_zero<V>();
  for (int n = threadIdx.x; n < N + W; n += mem.NT) {
    const float sv = n < N ? sinc_pi_f(signed_mode(n, N), N) : sinc_pi_f(bx * W + (n - N), N);
    (n < N ? sz2[n] : sx2[n - N]) = sv * sv;
  }
  fft_regs<N, 1, false, C>(u, t, stw, mem);
  {
    const int ny = signed_mode(ky, N);
    const float sy = sinc_pi_f(ny, N);
    const float wy = sy * sy;
    const float kf2 = kf * kf;
    const float wxy0 = sx2[mem.w * K] * wy, wxy1 = sx2[mem.w * K + K - 1] * wy;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int n = t + T * m, nz = signed_mode(n, N);
      const int myz = ny * ny + nz * nz;
      const float s0 = green_of(kx * kx + myz, kf2, wxy0 * sz2[n], deconv, norm);
      if constexpr (K == 1) {
        u[m] = c_scale(u[m], s0);
      } else {
        const float s1 = green_of((kx + 1) * (kx + 1) + myz, kf2, wxy1 * sz2[n], deconv, norm);
        u[m] = c_scale(u[m], make_float2(s0, s1));
      }
    }
  }
  park_store(park, u);
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const int n = t + T * m;
    u[m] = mul_ik(u[m], (n == N / 2) ? 0.0f : kf * (float)signed_mode(n, N));
  }
  fft_regs<N, 1, true, C>(u, t, stw, mem);
  if (valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(gz + m * (T * zstride), u[m]);
  }
  __syncwarp();
  park_load(park, u);
  fft_regs<N, 1, true, C>(u, t, stw, mem);
  if (valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(a + m * (T * zstride), u[m]);
  }
  __syncwarp();
}

// ---- 4. inverse y passes ------------------------------------------------------------------------------------
// Gy = IFFT_y(i k_y B), then B = IFFT_y(B) in place, then Gz = IFFT_y(Gz): the strip of B is read
// once and parked in tensor memory for its second transform.  block (bx, z0): W columns kx of SL
// slabs z (T(N) W / lanes SL threads); sm: SL N W float2, then the stage twiddle table
template <int N, int W, int SL, class V, class C = FFTConf<N>, class P_>
__device__ __forceinline__ void y_inv3_body(float2* __restrict__ B, float2* __restrict__ Gy, float2* __restrict__ Gz,
                                            float kf, const float2* __restrict__ tw, int bx, int z0, float2* sm,
                                            const P_& park) {
  constexpr int K = lanes_of<V>(), E = C::E, T = C::T, nh = N / 2 + 1, P = half_pitch<N>();
  const ColsThread<N, W, SL, V, C> mem(sm);
  float2* stab = sm + SL * N * W;
  stw_fill<C, 1>(stab, tw, threadIdx.x, mem.NT);
  const SmemTw<C> stw{stab};
  const int t = mem.t;
  const int kx = bx * W + mem.w * K;
  const bool valid = kx < nh;
  const int64_t at = (int64_t)(z0 + mem.sub) * N * P + (valid ? kx : 0) + t * P;
  float2* b = B + at;
  float2* gy = Gy + at;
  float2* gz = Gz + at;
  V u[E];
#pragma unroll
  for (int m = 0; m < E; ++m) u[m] = valid ? c_load<V>(b + m * (T * P)) : c_zero<V>();
  // the Gz strip is read only by the third transform: start pulling it into L2 now
  if (mem.w == 0 && valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) prefetch_l2_line(gz + m * (T * P));
  }
  __syncwarp();
  park_store(park, u);
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const int n = t + T * m;
    u[m] = mul_ik(u[m], (n == N / 2) ? 0.0f : kf * (float)signed_mode(n, N));
  }
  fft_regs<N, 1, true, C>(u, t, stw, mem);
  if (valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(gy + m * (T * P), u[m]);
  }
  __syncwarp();
  park_load(park, u);
  fft_regs<N, 1, true, C>(u, t, stw, mem);
  if (valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(b + m * (T * P), u[m]);
#pragma unroll
    for (int m = 0; m < E; ++m) u[m] = c_load<V>(gz + m * (T * P));
  }
  __syncwarp();
  fft_regs<N, 1, true, C>(u, t, stw, mem);
  if (valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(gz + m * (T * P), u[m]);
  }
  __syncwarp();
}

// ---- 5. inverse x passes of the three components -------------------------------------------------------------
// Work item: RB consecutive rows of one component (C, Gy or Gz; P complex per row).  The rows
// arrive in shared memory by bulk copy (TMA) at pitch LD = xrow_ld(N/2) while the block
// computes the previous item; the first FFT stage reads them there, and later stages reuse
// the same rows as their exchange buffer (the first stage has read all its inputs by then).
template <int N>
__host__ __device__ constexpr int c2r3_rows() {
  return FFTConf<N / 2>::T >= 128 ? 1 : 128 / FFTConf<N / 2>::T;
}

// Called by the 32 threads of warp 0: lane 0 registers the bytes on `bar`, lanes < rb copy one
// row each (P complex; P is a multiple of 4, so every row is a multiple of 32 bytes).
__device__ __forceinline__ void c2r3_issue(float2* stage, const float2* src_rows, int rb, int P, int LD,
                                           uint64_t* bar) {
  const int lane = threadIdx.x & 31;
  fence_proxy_async_smem();
  if (lane == 0) mbar_arrive_expect_tx(bar, (uint32_t)rb * (uint32_t)P * 8u);
  __syncwarp();
  for (int w = lane; w < rb; w += 32) bulk_copy_g2s(stage + w * LD, src_rows + (int64_t)w * P, (uint32_t)P * 8u, bar);
}

// Inverse x transform of the staged rows into F rows (pitch N floats); comp 0 applies i k_x.
// tw: the base twiddle table; stw: the stage twiddles (the base table or an SmemTw table)
template <int N, int RB, class CM = FFTConf<N / 2>, class STW>
__device__ __forceinline__ void c2r3_compute(float2* stage, float* __restrict__ Frows, int comp, float kf,
                                             const float2* __restrict__ tw, const STW& stw) {
  constexpr int M = N / 2, T = CM::T, LD = xrow_ld<M>(), R0 = first_radix<CM>();
  static_assert(T * RB <= 1024, "block too large");
  const int t = threadIdx.x % T, w = threadIdx.x / T;
  float2* buf = stage + w * LD;
  auto X = [&](int k) -> float2 {
    const float2 x = buf[k];
    return comp == 0 ? mul_ik(x, k == M ? 0.0f : kf * (float)k) : x;
  };
  auto load = [&](int n) -> float2 {
    const float2 a = X(n), bb = c_conj(X(M - n));
    const float2 e = c_add(a, bb);
    const float2 o = c_mul(c_sub(a, bb), c_conj(__ldg(tw + n)));
    return make_float2(__fsub_rn(e.x, o.y), __fadd_rn(e.y, o.x));
  };
  auto mem = [&](int n) -> float2& { return buf[xpad<R0>(n)]; };
  float2* dst = reinterpret_cast<float2*>(Frows + (int64_t)w * N);
  auto store = [&](int n, float2 x) { dst[n] = x; };
  fft_1d<M, 2, true, CM>(t, stw, load, mem, store);
}
template <int N, int RB, class CM = FFTConf<N / 2>>
__device__ __forceinline__ void c2r3_compute(float2* stage, float* __restrict__ Frows, int comp, float kf,
                                             const float2* __restrict__ tw) {
  c2r3_compute<N, RB, CM>(stage, Frows, comp, kf, tw, tw);
}

}  // namespace cola
