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
__device__ __forceinline__ V c_zero() {
  return V{};
}
__device__ __forceinline__ void c_store(float2* p, float2 v) { *p = v; }
__device__ __forceinline__ void c_store(float2* p, cpair v) { *reinterpret_cast<float4*>(p) = c_deinterleave(v); }
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

// Shapes of the single-box column passes.  A block holds G groups of threads, each with an
// exchange buffer and a barrier of its own, which transform strips of W columns independently of
// one another (one group's loads and stores overlap another's transforms) and share the stage
// twiddle table.
//
// What bounds them: shared-memory wavefronts (each exchange writes and reads every element) and
// how many bytes they keep in flight.  Loads go through the asynchronous copies of copy_async16
// into the exchange buffer itself: through the L1 cache each 64-byte row segment held a 128-byte
// line until it returned, and a kernel that takes 200 KB of shared memory has few lines left.
// More strips in flight than the shapes below have were slower (768: forward y 659 us with two
// strips of 8 columns per SM, 716 with three, 1046 with four), as were the E complex pairs of a
// thread squeezed into fewer registers; wider strips move more of a DRAM page at once (1024: z
// 4987 us with strips of 8, 4190 with 16).  Event times in us per launch, one column per thread
// with two-pass or re-read strips -> these shapes (GB300):
//   mesh   forward y       z with Green's function   inverse y
//    256    24 ->   26        68 ->    57               68 ->    64
//    384    95 ->   84       271 ->   195              303 ->   220
//    512   246 ->  198       953 ->   448             1172 ->   550
//    768   734 ->  655      2222 ->  1660             2133 ->  1880
//   1024  1922 -> 1714      8445 ->  4190             9090 ->  4710
//   1536  7657 -> 6030     29898 -> 19700            24573 -> 18600
// (Forward y of the force at 256 is the one that lost; one column per thread on four, five or six
// blocks per SM takes 25.5, 25 and 29 and no call is faster for it.)
enum ColsKind { kColsPlain, kColsZ, kColsY };
template <int N, int W, class V, class C>
struct ColsGroup;
template <int N, int KIND>
struct ColsCfg {
  using C = FFTConf<N>;
  static constexpr int N_ = N;
  // two columns per thread from 256 up; below, one, on twice the threads (256: z 57 us, 70 with
  // one; 192: z 33, 35-39 with two)
  using V = std::conditional_t<(N >= 256), cpair, float2>;
  // 16 columns are 128-byte row segments; 8 where buffers of 16 do not fit
  static constexpr int W = (N >= 1536 || (N == 768 && KIND == kColsY)) ? 8 : 16;
  // groups per block
  static constexpr int G = N == 1536 && KIND == kColsPlain ? 2
                           : N == 768                      ? (KIND == kColsPlain ? 1 : 2)
                           : N == 512                      ? 2
                           : N == 384                      ? (KIND == kColsPlain ? 2 : 3)
                                                           : 1;
  // threads per SM the kernel is compiled for (its registers)
  static constexpr int PER_SM = N == 2048   ? 512
                                : N == 1536 ? (KIND == kColsPlain ? 512 : 256)
                                : N == 1024 ? 512
                                : N == 768  ? (KIND == kColsZ ? 512 : 256)
                                : N == 512  ? 1024
                                : N == 384  ? (KIND == kColsPlain ? 256 : 384)
                                : N == 256  ? 512
                                            : 256;
  // persistent blocks, one wave of them, from 384 up
  static constexpr bool RESIDENT = N >= 384;
  static constexpr int K = lanes_of<V>(), GROUP = C::T * W / K, THREADS = GROUP * G;
  static constexpr int WORDS = (2 * C::E * K + 15) / 16 * 16;  // parked words per thread
  // (no more blocks than have their parked words in the tensor memory at once)
  static constexpr int PARKED = KIND == kColsPlain ? 64 : 512 / tmem_columns(THREADS, WORDS);
  static constexpr int WANT = PER_SM / THREADS < 1 ? 1 : PER_SM / THREADS;
  static constexpr int MIN_BLOCKS = WANT < PARKED ? WANT : PARKED;
  static constexpr int STRIPS = (N / 2 + W) / W;  // per slab
  static constexpr int TABLE = G * N * W;         // float2 offset of the stage twiddle table
  using Group = ColsGroup<N, W, V, C>;
};
// one thread's E elements, parked (tmem.cuh)
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

// u += what is parked, 16 words at a time (both at once would not fit in the registers)
template <class P, int E, class V>
__device__ __forceinline__ void park_add(const P& park, V (&u)[E]) {
  constexpr int M = 16 / (2 * lanes_of<V>());  // values in 16 words
#pragma unroll
  for (int m0 = 0; m0 < E; m0 += M) {
    uint32_t r[16];
    park.load16(m0 / M * 16, r);
#pragma unroll
    for (int m = 0; m < M && m0 + m < E; ++m) {
      if constexpr (lanes_of<V>() == 1)
        u[m0 + m] = c_add(u[m0 + m], make_float2(__uint_as_float(r[2 * m]), __uint_as_float(r[2 * m + 1])));
      else
        u[m0 + m] = c_add(u[m0 + m], V{make_float2(__uint_as_float(r[4 * m]), __uint_as_float(r[4 * m + 1])),
                                       make_float2(__uint_as_float(r[4 * m + 2]), __uint_as_float(r[4 * m + 3]))});
    }
  }
}

// A thread's place in a group that transforms a strip of W columns, and the group's exchange
// buffer: columns w K .. of the strip, transform thread t.  Rows of 64 bytes (W = 8) are swapped
// in pairs according to the parity of n / R0, so that the first stage's stores, which are R0 rows
// apart in consecutive threads, do not all fall on the same half of the banks.
template <int N, int W, class V, class C>
struct ColsGroup {
  static constexpr int K = lanes_of<V>(), WT = W / K, T = C::T, NT = T * WT;
  // (the exponent of R0; 0 = rows in place, also where T would not keep the loads' parity constant)
  static constexpr int SHIFT = first_radix<C>() >= 16 ? 4 : 3;
  static constexpr int SWAP = W * (int)sizeof(float2) == 64 && T % (2 << SHIFT) == 0 ? SHIFT : 0;
  int w, t, bar;
  V* S;
  // thread i of the group, its buffer of N W float2 and its hardware barrier
  __device__ __forceinline__ ColsGroup(float2* buf, int i, int barrier)
      : w(i % WT), t(i / WT), bar(barrier), S(reinterpret_cast<V*>(buf)) {}
  // row n = base + off (see mem_at): n ^ ((n >> SWAP) & 1), of which base gives two values (in
  // registers) and off the choice between them and a constant offset
  __device__ __forceinline__ V& at(int base, int off) const {
    if constexpr (SWAP > 0) {
      const int x = base ^ ((base >> SWAP) & 1);
      return (((off ^ (off >> SWAP)) & 1) ? S + ((x ^ 1) * WT + w) : S + (x * WT + w))[(off & ~1) * WT];
    } else {
      return (S + (base * WT + w))[off * WT];
    }
  }
  // The same place with its indices recomputed from here on: keeps a persistent loop from holding
  // every address of the exchange in a register (at 128 registers those would be spilled).
  __device__ __forceinline__ ColsGroup fresh() const {
    ColsGroup g = *this;
    asm volatile("" : "+r"(g.w), "+r"(g.t));
    return g;
  }
  __device__ __forceinline__ void sync() const {
    if constexpr (NT == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(NT) : "memory");
  }
  // Start the copies of this thread's elements n = t + T m (at p + m step) into their slots of the
  // buffer; collect() waits for them.  No other thread touches those slots before the first
  // exchange, and the caller sees to it that the group has read the buffer's last contents.
  // (Scalar columns are 8 bytes wide: they are loaded by collect() itself.)
  __device__ __forceinline__ void fetch(const float2* p, int64_t step, bool valid) const {
    if constexpr (K == 2) {
#pragma unroll
      for (int m = 0; m < C::E; ++m, p += step) copy_async16(&at(t, T * m), p, valid);
    }
  }
  __device__ __forceinline__ void collect(V (&u)[C::E], const float2* p, int64_t step, bool valid) const {
    if constexpr (K == 2) {
      copy_wait_all();
#pragma unroll
      for (int m = 0; m < C::E; ++m) {
        const V& slot = at(t, T * m);
        u[m] = c_interleave(*reinterpret_cast<const float4*>(&slot));
      }
    } else {
#pragma unroll
      for (int m = 0; m < C::E; ++m, p += step) u[m] = valid ? c_load<V>(p) : c_zero<V>();
    }
  }
};

// The strips of one column pass: strip i covers W columns from bx W of one slab (i = slab NB + bx,
// NB strips per slab); element (n, col) of it at data[slab * slab_stride + n * row_stride + col].
// A thread's first element of strip i, and whether its columns exist:
template <int N, int W, class V, class C>
struct StripWalk {
  int64_t slab_stride, row_stride;
  int kx, slab;
  bool valid;
  int64_t first;
  __device__ __forceinline__ StripWalk(int64_t slab_stride_, int64_t row_stride_, int bx, int slab_,
                                       const ColsGroup<N, W, V, C>& g)
      : slab_stride(slab_stride_), row_stride(row_stride_), kx(bx * W + g.w * g.K), slab(slab_), valid(kx < N / 2 + 1),
        first(slab * slab_stride + g.t * row_stride + (valid ? kx : 0)) {}
  __device__ __forceinline__ int64_t step() const { return C::T * row_stride; }
};

// In-place FFT of a strip whose copies are under way; next() starts those of the group's next
// strip, once the group is done with the buffer and before the last stage and the stores.
template <bool INV, int N, int W, class V, class C, class TW, class Next>
__device__ __forceinline__ void cols_strip(float2* __restrict__ data, const StripWalk<N, W, V, C>& s, const TW& tw,
                                           const ColsGroup<N, W, V, C>& mem, Next&& next) {
  constexpr int E = C::E;
  float2* p = data + s.first;
  V u[E];
  mem.collect(u, p, s.step(), s.valid);
  auto after_reads = [&] {
    mem.sync();
    next();
  };
  fft_regs<N, 1, INV, C>(u, mem.t, tw, mem, after_reads);
  if (s.valid) {
#pragma unroll
    for (int m = 0; m < E; ++m, p += s.step()) c_store(p, u[m]);
  }
}

// The walk of a group over the strips of nslabs slabs (the blocks' first groups take the first
// strips, then the second groups, ...): one(walk, mem, next) transforms a strip whose copies from
// src are under way and calls next() where its buffer is free for the following strip's.
template <class Cfg, class One>
__device__ __forceinline__ void cols_walk(const float2* src, int64_t slab_stride, int64_t row_stride, int nslabs,
                                          float2* smem, One&& one) {
  constexpr int G = Cfg::G, NB = Cfg::STRIPS, N = Cfg::N_;
  static_assert(G <= 15, "hardware barriers: 0 is the block's, 1 to 15 the groups'");
  using Group = typename Cfg::Group;
  using Walk = StripWalk<N, Cfg::W, typename Cfg::V, typename Cfg::C>;
  const int group = threadIdx.x / Cfg::GROUP;
  const Group place(smem + group * (N * Cfg::W), threadIdx.x % Cfg::GROUP, group + 1);
  const int total = NB * nslabs, stride = gridDim.x * G;
  int i = blockIdx.x + gridDim.x * group;
  if (i < total) {
    const Walk s(slab_stride, row_stride, i % NB, i / NB, place);
    place.fetch(src + s.first, s.step(), s.valid);
  }
  for (; i < total; i += stride) {
    const Group mem = place.fresh();
    const Walk s(slab_stride, row_stride, i % NB, i / NB, mem);
    auto next = [&] {
      const int j = i + stride;
      if (j < total) {
        const Walk n(slab_stride, row_stride, j % NB, j / NB, mem);
        mem.fetch(src + n.first, n.step(), n.valid);
      }
    };
    one(s, mem, next);
  }
}

// ---- 1. deposit + x r2c -----------------------------------------------------------------------
// block: one tile of TY x TZ rows (T(N/2) * TY * TZ threads); acc: max(TY TZ N, TY TZ LD) x 8
// bytes of shared memory (the cells' low 32-bit words, then their high words; afterwards the
// rows' transform buffers); ints: 28 ints of shared memory
// rec: the bin-ordered particle records (fixed-point CIC coordinates; offsets index them directly)
// (stw: the row transform's stage twiddles, the base table tw or an SmemTw table)
// The block has D >= T(N/2) TY TZ threads: all of them deposit, the first T(N/2) TY TZ transform.
// Row buffers of a tile, with a barrier of their own for the threads that transform:
template <int R0, int NT, int D>
struct RowBuffer {
  float2* buf;
  __device__ __forceinline__ float2& operator()(int n) const { return buf[xpad<R0>(n)]; }
  __device__ __forceinline__ void sync() const {
    if constexpr (NT == D) __syncthreads();
    else if constexpr (NT < 32) __syncwarp((1u << NT) - 1u);
    else if constexpr (NT == 32) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
  }
};
template <int N, int TY, int TZ, class CM = FFTConf<N / 2>, int D = CM::T * TY * TZ, class STW>
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
  for (int i = threadIdx.x; i < ROWS * N; i += D) acc[i] = 0ull;
  // the tile's own 4 bins and the boundary bins of its 3 lower neighbours, loaded in parallel
  // (a loop: a block may have fewer than 9 threads)
  for (int k = threadIdx.x; k < 9; k += D) {
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
  unsigned* lo = reinterpret_cast<unsigned*>(acc);
  unsigned* hi = lo + ROWS * N;
  constexpr int U = 4;  // particles in flight per thread
  for (int base = threadIdx.x; base < total; base += D * U) {
    uint32_t f[U][3];
    bool ok[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + u * D;
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
    for (int u = 0; u < U; ++u)
      if (ok[u]) acc_cloud<TY, TZ, (N <= 384)>(lo, hi, f[u], g.fbits, N, y0, z0);
  }
  __syncthreads();
  // real-to-complex FFT of each tile row; z[n] = (delta[2n], delta[2n+1]).  The transform
  // buffers overlay the accumulators: fft_1d reads all its inputs before a block barrier
  // that precedes its first shared-memory write.
  if (NT < D && (int)threadIdx.x >= NT) return;
  const int t = threadIdx.x % T, w = threadIdx.x / T;
  const uint2* lrow = reinterpret_cast<const uint2*>(lo + w * N);
  const uint2* hrow = reinterpret_cast<const uint2*>(hi + w * N);
  float2* buf = reinterpret_cast<float2*>(acc) + w * LD;
  RowBuffer<R0, NT, D> mem{buf};
  bool overflow = false;
  auto load = [&](int n) -> float2 {
    const uint2 l = lrow[n], h = hrow[n];
    overflow |= ((h.x | h.y) >> 30) != 0u;
    const unsigned long long a = ((unsigned long long)h.x << 32) | l.x;
    const unsigned long long b = ((unsigned long long)h.y << 32) | l.y;
    return make_float2(fmaf(u64_to_f32_rn(a), dscale, -1.0f), fmaf(u64_to_f32_rn(b), dscale, -1.0f));
  };
  auto store = [&](int n, float2 x) { buf[xpad<R0>(n)] = x; };
  fft_1d<M, 2, false, CM>(t, stw, load, mem, store);
  if (overflow) atomicOr(err, kErrOverflow);
  mem.sync();
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

// sinc^2 of the N mode numbers of a mesh side, into shared memory by threads tid of nth
template <int N>
__device__ __forceinline__ void sinc2_fill(float* dst, int tid, int nth) {
  for (int n = tid; n < N; n += nth) {
    const float sv = sinc_pi_f(signed_mode(n, N), N);
    dst[n] = sv * sv;
  }
}

// one strip (slab = ky) whose copies are under way (sinc2: the table above; next: see cols_strip)
template <int N, int W, class V, class C, class TW, class P_, class Next>
__device__ __forceinline__ void z_green_strip(float2* __restrict__ A, float2* __restrict__ Gz, float kf, int deconv,
                                              float norm, const TW& stw, const float* sinc2,
                                              const StripWalk<N, W, V, C>& s, const ColsGroup<N, W, V, C>& mem,
                                              const P_& park, Next&& next) {
  constexpr int K = lanes_of<V>(), E = C::E, T = C::T;
  constexpr int64_t zstep = (int64_t)T * N * half_pitch<N>();
  const int t = mem.t, kx = s.kx;
  float2* a = A + s.first;
  float2* gz = Gz + s.first;
  V u[E];
  mem.collect(u, a, zstep, s.valid);
  fft_regs<N, 1, false, C>(u, t, stw, mem);
  {
    // (sinc is even: sinc2[k] is that of the mode numbers k and -k; the columns beyond N/2 are padding)
    const int ny = signed_mode(s.slab, N);
    const float wy = sinc2[s.slab];
    const float kf2 = kf * kf;
    const float wxy0 = sinc2[s.valid ? kx : 0] * wy, wxy1 = sinc2[s.valid ? kx + K - 1 : 0] * wy;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int n = t + T * m, nz = signed_mode(n, N);
      const int myz = ny * ny + nz * nz;
      const float s0 = green_of(kx * kx + myz, kf2, wxy0 * sinc2[n], deconv, norm);
      if constexpr (K == 1) {
        u[m] = c_scale(u[m], s0);
      } else {
        const float s1 = green_of((kx + 1) * (kx + 1) + myz, kf2, wxy1 * sinc2[n], deconv, norm);
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
  if (s.valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(gz + m * zstep, u[m]);
  }
  park_load(park, u);
  auto after_reads = [&] {
    mem.sync();
    next();
  };
  fft_regs<N, 1, true, C>(u, t, stw, mem, after_reads);
  if (s.valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(a + m * zstep, u[m]);
  }
  __syncwarp();
}

// ---- 3a. the z pass of the force's transpose --------------------------------------------------
// Phi_k = sum_i conj(i k_i / (k^2 W^p)) Lam_i,k / N^3 of the three deposited adjoints' spectra after
// their x and y transforms, back along z into lx.  k_x and k_y do not change along z, so k_x Lam_x
// + k_y Lam_y is one transform; its result is parked while Lam_z is transformed.  One strip
// (slab = ky) whose copies of lx are under way (next: see cols_strip).
template <int N, int W, class V, class C, class TW, class P_, class Next>
__device__ __forceinline__ void z_adjoint_strip(float2* __restrict__ lx, const float2* __restrict__ ly,
                                                const float2* __restrict__ lz, float kf, int deconv, float norm,
                                                const TW& stw, const float* sinc2, const StripWalk<N, W, V, C>& s,
                                                const ColsGroup<N, W, V, C>& mem, const P_& park, Next&& next) {
  constexpr int K = lanes_of<V>(), E = C::E, T = C::T;
  constexpr int64_t zstep = (int64_t)T * N * half_pitch<N>();
  const int t = mem.t, kx = s.kx, ny = signed_mode(s.slab, N);
  auto k_of = [&](int n) { return n == N / 2 || n == -N / 2 ? 0.0f : kf * (float)n; };
  V u[E];
  mem.collect(u, lx + s.first, zstep, s.valid);
  {
    const float ky = k_of(ny), kx0 = k_of(kx), kx1 = k_of(kx + K - 1);
    const float2* p = ly + s.first;
#pragma unroll
    for (int m = 0; m < E; ++m, p += zstep) {
      const V b = s.valid ? c_load<V>(p) : c_zero<V>();
      if constexpr (K == 1) u[m] = c_fma(ky, b, c_scale(u[m], kx0));
      else u[m] = c_fma(ky, b, c_scale(u[m], make_float2(kx0, kx1)));
    }
  }
  auto fetch_lz = [&] {
    mem.sync();
    mem.fetch(lz + s.first, zstep, s.valid);
  };
  fft_regs<N, 1, false, C>(u, t, stw, mem, fetch_lz);
  park_store(park, u);
  mem.collect(u, lz + s.first, zstep, s.valid);
  fft_regs<N, 1, false, C>(u, t, stw, mem);
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const float kz = k_of(signed_mode(t + T * m, N));
    if constexpr (K == 1) u[m] = c_scale(u[m], kz);
    else u[m] = c_scale(u[m], make_float2(kz, kz));
  }
  park_add(park, u);
  {
    const float kf2 = kf * kf, wy = sinc2[s.slab];
    const float wxy0 = sinc2[s.valid ? kx : 0] * wy, wxy1 = sinc2[s.valid ? kx + K - 1 : 0] * wy;
    auto green = [&](int nx, int nz, float wk) {
      const int m2 = nx * nx + ny * ny + nz * nz;
      if (m2 == 0) return 0.0f;
      float den = kf2 * (float)m2;
      if (deconv) den *= deconv == 2 ? wk * wk : wk;
      return norm / den;
    };
#pragma unroll
    for (int m = 0; m < E; ++m) {  // -i times the sum
      const int n = t + T * m, nz = signed_mode(n, N);
      const float g0 = green(kx, nz, wxy0 * sinc2[n]);
      if constexpr (K == 1) {
        u[m] = make_float2(u[m].y * g0, -u[m].x * g0);
      } else {
        const float g1 = green(kx + 1, nz, wxy1 * sinc2[n]);
        u[m] = V{make_float2(u[m].im.x * g0, u[m].im.y * g1), make_float2(-u[m].re.x * g0, -u[m].re.y * g1)};
      }
    }
  }
  auto after_reads = [&] {
    mem.sync();
    next();
  };
  fft_regs<N, 1, true, C>(u, t, stw, mem, after_reads);
  if (s.valid) {
    float2* p = lx + s.first;
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(p + m * zstep, u[m]);
  }
  __syncwarp();
}

// ---- 4. inverse y passes ------------------------------------------------------------------------------------
// Gy = IFFT_y(i k_y B), then B = IFFT_y(B) in place, then Gz = IFFT_y(Gz): the strip of B is read
// once and parked in tensor memory for its second transform, after whose last exchange the copies
// of the Gz strip start.  One strip (slab = z) whose copies of B are under way (next: see
// cols_strip).
template <int N, int W, class V, class C, class TW, class P_, class Next>
__device__ __forceinline__ void y_inv3_strip(float2* __restrict__ B, float2* __restrict__ Gy, float2* __restrict__ Gz,
                                             float kf, const TW& stw, const StripWalk<N, W, V, C>& s,
                                             const ColsGroup<N, W, V, C>& mem, const P_& park, Next&& next) {
  constexpr int E = C::E, T = C::T, step = T * half_pitch<N>();
  const int t = mem.t;
  float2* b = B + s.first;
  float2* gy = Gy + s.first;
  float2* gz = Gz + s.first;
  V u[E];
  mem.collect(u, b, step, s.valid);
  park_store(park, u);
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const int n = t + T * m;
    u[m] = mul_ik(u[m], (n == N / 2) ? 0.0f : kf * (float)signed_mode(n, N));
  }
  fft_regs<N, 1, true, C>(u, t, stw, mem);
  if (s.valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(gy + m * step, u[m]);
  }
  park_load(park, u);
  auto fetch_gz = [&] {
    mem.sync();
    mem.fetch(gz, step, s.valid);
  };
  fft_regs<N, 1, true, C>(u, t, stw, mem, fetch_gz);
  if (s.valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(b + m * step, u[m]);
  }
  mem.collect(u, gz, step, s.valid);
  auto after_reads = [&] {
    mem.sync();
    next();
  };
  fft_regs<N, 1, true, C>(u, t, stw, mem, after_reads);
  if (s.valid) {
#pragma unroll
    for (int m = 0; m < E; ++m) c_store(gz + m * step, u[m]);
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
// (put(w, n, x): element n of row w, two real values)
template <int N, int RB, class CM = FFTConf<N / 2>, class STW, class Put>
__device__ __forceinline__ void c2r_rows(float2* stage, int comp, float kf, const float2* __restrict__ tw,
                                         const STW& stw, Put&& put) {
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
  auto store = [&](int n, float2 x) { put(w, n, x); };
  fft_1d<M, 2, true, CM>(t, stw, load, mem, store);
}
template <int N, int RB, class CM = FFTConf<N / 2>, class STW>
__device__ __forceinline__ void c2r3_compute(float2* stage, float* __restrict__ Frows, int comp, float kf,
                                             const float2* __restrict__ tw, const STW& stw) {
  c2r_rows<N, RB, CM>(stage, comp, kf, tw, stw,
                      [&](int w, int n, float2 x) { reinterpret_cast<float2*>(Frows + (int64_t)w * N)[n] = x; });
}

// The persistent inverse-x loop over `total` items of RB rows: the rows of item i at src_of(i),
// its transform done by one(item, staged rows).  Each block walks items blockIdx.x, blockIdx.x +
// gridDim.x, ... with the bulk copy of its next item in flight (two buffers at `stages`).
template <int N, int RB, class Src, class One>
__device__ __forceinline__ void c2r_walk(float2* stages, uint64_t (&bars)[2], int64_t total, int P,
                                         int* __restrict__ err, Src&& src_of, One&& one) {
  constexpr int LD = xrow_ld<N / 2>();
  if (threadIdx.x == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    mbar_fence_init();
  }
  __syncthreads();
  int64_t item = blockIdx.x;
  if (item < total && threadIdx.x < 32) c2r3_issue(stages, src_of(item), RB, P, LD, &bars[0]);
  for (int it = 0; item < total; ++it, item += gridDim.x) {
    const int b = it & 1;
    const int64_t ahead = item + gridDim.x;
    // (the other buffer was consumed at iteration it - 1, free after its closing barrier)
    if (ahead < total && threadIdx.x < 32) c2r3_issue(stages + (b ^ 1) * RB * LD, src_of(ahead), RB, P, LD, &bars[b ^ 1]);
    const bool ok = mbar_wait(&bars[b], (it >> 1) & 1);
    if (__syncthreads_or(!ok)) {
      // leave no bulk copy in flight into shared memory the block releases: wait again (bounded)
      // for the copy that timed out and for the later one if it was issued
      if (threadIdx.x == 0) atomicOr(err, kErrTimeout);
      mbar_wait(&bars[b], (it >> 1) & 1);
      if (ahead < total) mbar_wait(&bars[b ^ 1], ((it + 1) >> 1) & 1);
      return;
    }
    one(item, stages + b * RB * LD);
    __syncthreads();
  }
}

}  // namespace cola
