// Batched 1-D FFT passes of the 3-D real-to-complex / complex-to-real transforms.
//
// Layout of a half spectrum of an n^3 real mesh: [z][y][kx], kx in [0, n/2], rows padded to
// P >= n/2 + 1 complex entries.  A 3-D r2c is: x pass (real rows -> half rows), y pass and
// z pass (strided complex columns, in place).  The c2r runs the same passes in reverse.
#include "cola_internal.cuh"
#include "fft.cuh"
#include "pm_bodies.cuh"
#include "cols_launch.cuh"

namespace cola {

// rows per block of the contiguous x passes (about 256 threads per block)
template <int N>
__host__ __device__ constexpr int x_rows() {
  return FFTConf<N / 2>::T >= 256 ? 1 : 256 / FFTConf<N / 2>::T;
}

// In-place FFT of the N/2 + 1 columns of the N slabs of a half spectrum, along y (slab = z) or
// along z (slab = y).
template <int N, bool INV, bool ALONG_Z>
__global__ void __launch_bounds__(ColsCfg<N, kColsPlain>::THREADS, ColsCfg<N, kColsPlain>::MIN_BLOCKS)
    k_fft_cols(float2* __restrict__ data, const float2* __restrict__ tw) {
  extern __shared__ __align__(16) float2 smem[];
  using Cfg = ColsCfg<N, kColsPlain>;
  float2* stab = smem + Cfg::TABLE;
  stw_fill<FFTConf<N>, 1>(stab, tw, threadIdx.x, Cfg::THREADS);
  pdl_begin();
  __syncthreads();
  const SmemTw<FFTConf<N>> stw{stab};
  constexpr int64_t P = half_pitch<N>();
  cols_walk<Cfg>(data, ALONG_Z ? P : N * P, ALONG_Z ? N * P : P, N, smem,
                 [&](const auto& s, const auto& mem, auto& next) { cols_strip<INV>(data, s, stw, mem, next); });
}

// Real rows of length N -> half-spectrum rows (N/2 + 1 entries, stride P), via a complex
// FFT of length M = N/2 of z[n] = x[2n] + i x[2n+1] and the split
//   X[k] = (Z[k] + conj Z[M-k]) / 2 - (i/2) exp(-2 pi i k/N) (Z[k] - conj Z[M-k]).
// The x passes read their stage twiddles from a shared-memory table behind the row buffers
// (fft.cuh; filled per block, first read after the transform's first barrier).
template <int N>
__global__ void __launch_bounds__(FFTConf<N / 2>::T * x_rows<N>())
    k_fft_x_r2c(const float* __restrict__ in, float2* __restrict__ out, int P, const float2* __restrict__ tw) {
  constexpr int M = N / 2, T = FFTConf<M>::T, RB = x_rows<N>(), LD = xrow_ld<M>();
  constexpr int R0 = first_radix<FFTConf<M>>();
  extern __shared__ __align__(16) float2 smem[];
  float2* stab = smem + RB * LD;
  stw_fill<FFTConf<M>, 2>(stab, tw, threadIdx.x, T * RB);
  pdl_begin();
  const SmemTw<FFTConf<M>> stw{stab};
  const int t = threadIdx.x % T, w = threadIdx.x / T;
  const int64_t row = (int64_t)blockIdx.x * RB + w;
  const float2* src = reinterpret_cast<const float2*>(in + row * N);
  float2* buf = smem + w * LD;
  auto load = [&](int n) -> float2 { return src[n]; };
  auto mem = [&](int n) -> float2& { return buf[xpad<R0>(n)]; };
  auto store = [&](int n, float2 x) { buf[xpad<R0>(n)] = x; };
  fft_1d<M, 2, false>(t, stw, load, mem, store);
  __syncthreads();
  float2* dst = out + row * P;
  // X[k] = e + p and X[M - k] = conj(e - p) from one pair Z[k], Z[M - k] (p = W^k (-i d))
  for (int k = t; k <= M / 2; k += T) {
    const float2 a = buf[xpad<R0>(k)];
    const float2 b = c_conj(buf[xpad<R0>(k == 0 ? 0 : M - k)]);
    const float2 e = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y + b.y));
    const float2 d = make_float2(0.5f * (a.x - b.x), 0.5f * (a.y - b.y));
    const float2 p = c_mul(__ldg(tw + k), make_float2(d.y, -d.x));
    dst[k] = c_add(e, p);
    if (2 * k != M) dst[M - k] = c_conj(c_sub(e, p));
  }
}

// The same of the first three components of a mesh of float4, into three half spectra: a thread
// reads its cells once and keeps the components that wait in registers.
struct Spectra3 {
  float2* p[3];
};
template <int N>
__global__ void __launch_bounds__(FFTConf<N / 2>::T * x_rows<N>())
    k_fft_x_r2c3(const float4* __restrict__ in, Spectra3 out, int P, const float2* __restrict__ tw) {
  using C = FFTConf<N / 2>;
  constexpr int M = N / 2, T = C::T, E = C::E, RB = x_rows<N>(), LD = xrow_ld<M>();
  constexpr int R0 = first_radix<C>();
  extern __shared__ __align__(16) float2 smem[];
  float2* stab = smem + RB * LD;
  stw_fill<C, 2>(stab, tw, threadIdx.x, T * RB);
  const SmemTw<C> stw{stab};
  const int t = threadIdx.x % T, w = threadIdx.x / T;
  const int64_t row = (int64_t)blockIdx.x * RB + w;
  const float4* src = in + row * N;
  float2* buf = smem + w * LD;
  auto mem = [&](int n) -> float2& { return buf[xpad<R0>(n)]; };
  float2 v[3][E];
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const float4 a = src[2 * (t + T * m)], b = src[2 * (t + T * m) + 1];
    v[0][m] = make_float2(a.x, b.x);
    v[1][m] = make_float2(a.y, b.y);
    v[2][m] = make_float2(a.z, b.z);
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if constexpr (M == R0) {  // one stage: nothing is exchanged
      auto load = [&](int n) -> float2 { return v[j][(n - t) / T]; };
      auto store = [&](int n, float2 x) { mem(n) = x; };
      fft_1d<M, 2, false>(t, stw, load, mem, store);
    } else {
      fft_regs<M, 2, false>(v[j], t, stw, mem);
      __syncthreads();
#pragma unroll
      for (int m = 0; m < E; ++m) mem(t + T * m) = v[j][m];
    }
    __syncthreads();
    float2* dst = out.p[j] + row * P;
    for (int k = t; k <= M / 2; k += T) {
      const float2 a = mem(k), b = c_conj(mem(k == 0 ? 0 : M - k));
      const float2 e = c_scale(c_add(a, b), 0.5f), d = c_scale(c_sub(a, b), 0.5f);
      const float2 p = c_mul(__ldg(tw + k), make_float2(d.y, -d.x));
      dst[k] = c_add(e, p);
      if (2 * k != M) dst[M - k] = c_conj(c_sub(e, p));
    }
  }
}

// Half-spectrum rows -> real rows of length N (unscaled inverse, times `scale`): the persistent
// inverse-x pass of the force with one component.  SUB_SQ: the rows are not stored but their
// squares taken off what out holds (the 2LPT source's cross terms).  256^3: 51 us with one item per
// block read through registers, 25 this way.
template <int N, bool SUB_SQ>
__global__ void __launch_bounds__(FFTConf<N / 2>::T * c2r3_rows<N>(), 3)
    k_fft_x_c2r(const float2* __restrict__ in, float* __restrict__ out, int P, const float2* __restrict__ tw,
                float scale, int* __restrict__ err) {
  constexpr int M = N / 2, RB = c2r3_rows<N>(), LD = xrow_ld<M>();
  extern __shared__ __align__(128) float2 smem[];
  __shared__ __align__(8) uint64_t bars[2];
  float2* stab = smem + 2 * RB * LD;
  stw_fill<FFTConf<M>, 2>(stab, tw, threadIdx.x, blockDim.x);
  const SmemTw<FFTConf<M>> stw{stab};
  pdl_begin();
  c2r_walk<N, RB>(
      smem, bars, (int64_t)N * N / RB, P, err, [&](int64_t item) { return in + item * RB * P; },
      [&](int64_t item, float2* rows) {
        float2* dst = reinterpret_cast<float2*>(out + item * RB * N);
        c2r_rows<N, RB>(rows, 1, 0.0f, tw, stw, [&](int w, int n, float2 x) {
          float2* p = dst + w * M + n;
          const float2 r = c_scale(x, scale);
          if constexpr (SUB_SQ) {
            const float2 acc = *p;
            *p = make_float2(fmaf(-r.x, r.x, acc.x), fmaf(-r.y, r.y, acc.y));
          } else {
            *p = r;
          }
        });
      });
}

// Spectral factor of one mode on its way into the inverse z pass (mode numbers nx, ny, nz):
//   kind 0: scale * (i k_i) / k^2 * a          (s1_i; with scale < 0: s2 from mu2)
//   kind 1: scale * (i k_i)(i k_j) / k^2 * a   (psi1_{i,j})
// first derivatives zero on their Nyquist plane
struct SpectralFactor {
  int kind, i, j;
  float kf, scale;
};
template <int N>
__device__ __forceinline__ float2 spectral_mul(const SpectralFactor& f, int nx, int ny, int nz, float2 a) {
  const int m2 = nx * nx + ny * ny + nz * nz;
  if (m2 == 0) return make_float2(0.f, 0.f);
  const float inv_k2 = f.scale / (f.kf * f.kf * (float)m2);
  auto k_of = [&](int c) {
    const int m = c == 0 ? nx : (c == 1 ? ny : nz);
    return (m == N / 2 || m == -N / 2) ? 0.0f : f.kf * (float)m;
  };
  const float ki = k_of(f.i);
  if (f.kind == 0) return make_float2(__fmul_rn(__fmul_rn(-ki, a.y), inv_k2), __fmul_rn(__fmul_rn(ki, a.x), inv_k2));
  const float kk = __fmul_rn(__fmul_rn(-ki, k_of(f.j)), inv_k2);
  return make_float2(__fmul_rn(kk, a.x), __fmul_rn(kk, a.y));
}

// The inverse z pass of `factor` times the half spectrum `in`, into `out` (a launch of the factor
// alone reads and writes the spectrum once more: 42 us at 256^3).
template <int N>
__global__ void __launch_bounds__(ColsCfg<N, kColsPlain>::THREADS, ColsCfg<N, kColsPlain>::MIN_BLOCKS)
    k_fft_z_factor(const float2* __restrict__ in, float2* __restrict__ out, SpectralFactor factor,
                   const float2* __restrict__ tw) {
  extern __shared__ __align__(16) float2 smem[];
  using Cfg = ColsCfg<N, kColsPlain>;
  using V = typename Cfg::V;
  float2* stab = smem + Cfg::TABLE;
  stw_fill<FFTConf<N>, 1>(stab, tw, threadIdx.x, Cfg::THREADS);
  pdl_begin();
  __syncthreads();
  const SmemTw<FFTConf<N>> stw{stab};
  constexpr int64_t P = half_pitch<N>();
  constexpr int E = Cfg::C::E, T = Cfg::C::T;
  cols_walk<Cfg>(in, P, N * P, N, smem, [&](const auto& s, const auto& mem, auto& next) {
    V u[E];
    mem.collect(u, in + s.first, s.step(), s.valid);
    const int ny = signed_mode(s.slab, N);
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int nz = signed_mode(mem.t + T * m, N);
      if constexpr (Cfg::K == 1) {
        u[m] = spectral_mul<N>(factor, s.kx, ny, nz, u[m]);
      } else {
        const float2 a = spectral_mul<N>(factor, s.kx, ny, nz, make_float2(u[m].re.x, u[m].im.x));
        const float2 b = spectral_mul<N>(factor, s.kx + 1, ny, nz, make_float2(u[m].re.y, u[m].im.y));
        u[m] = V{make_float2(a.x, b.x), make_float2(a.y, b.y)};
      }
    }
    auto after_reads = [&] {
      mem.sync();
      next();
    };
    fft_regs<N, 1, true>(u, mem.t, stw, mem, after_reads);
    if (s.valid) {
      float2* p = out + s.first;
#pragma unroll
      for (int m = 0; m < E; ++m, p += s.step()) c_store(p, u[m]);
    }
  });
}

// persistent per-size kernel labels for the profiler
template <int N>
static const char* label(const char* kind) {
  static const std::string names[4] = {std::string("fft_x_r2c_") + std::to_string(N),
                                       std::string("fft_x_c2r_") + std::to_string(N),
                                       std::string("fft_cols_fwd_") + std::to_string(N),
                                       std::string("fft_cols_inv_") + std::to_string(N)};
  const int i = kind[0] == 'r' ? 0 : kind[0] == 'c' ? 1 : kind[0] == 'f' ? 2 : 3;
  return names[i].c_str();
}

template <class K>
static void allow_smem(K kernel, size_t bytes) {
  if (bytes > 32 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int N>
static int x_r2c(const float* in, float2* out, int64_t nrows, int P, const float2* tw, cudaStream_t st) {
  constexpr int M = N / 2, RB = x_rows<N>();
  const size_t smem = (size_t)(RB * xrow_ld<M>() + stw_size<FFTConf<M>>()) * sizeof(float2);
  if (nrows % RB) return fail(COLA_EINVAL, "fft x pass: row count not a multiple of the block rows");
  allow_smem(k_fft_x_r2c<N>, smem);
  { LaunchScope ls_(label<N>("r2c"), st);
  launch(k_fft_x_r2c<N>, (unsigned)(nrows / RB), FFTConf<M>::T * RB, smem, st, in, out, P, tw); }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

template <int N>
static int x_r2c3(const float4* in, const Spectra3& out, int P, const float2* tw, cudaStream_t st) {
  constexpr int M = N / 2, RB = x_rows<N>();
  constexpr size_t smem = (size_t)(RB * xrow_ld<M>() + stw_size<FFTConf<M>>()) * sizeof(float2);
  static_assert((N * N) % RB == 0, "whole blocks of rows");
  allow_smem(k_fft_x_r2c3<N>, smem);
  LaunchScope ls_(label<N>("r2c"), st);
  k_fft_x_r2c3<N><<<N * N / RB, FFTConf<M>::T * RB, smem, st>>>(in, out, P, tw);
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

template <int N, bool SUB_SQ>
static int x_c2r_t(const float2* in, float* out, int P, const float2* tw, float scale, int* err, cudaStream_t st) {
  constexpr int M = N / 2, RB = c2r3_rows<N>(), NT = FFTConf<M>::T * RB;
  constexpr size_t smem = (size_t)(2 * RB * xrow_ld<M>() + stw_size<FFTConf<M>>()) * sizeof(float2);
  static_assert((N * N) % RB == 0, "whole items");
  if (P % 4) return fail(COLA_EINVAL, "fft x pass: row pitch must be a multiple of 4 complex");
  static std::atomic<int> resident[64] = {};
  int dev = 0;
  COLA_CUDA_CHECK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(COLA_EUNSUPPORTED, "device index above 63");
  int cap = resident[dev].load(std::memory_order_acquire);
  if (!cap) {
    int occ = 0, sms = 0;
    allow_smem(k_fft_x_c2r<N, SUB_SQ>, smem);
    COLA_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_fft_x_c2r<N, SUB_SQ>, NT, smem));
    COLA_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (occ < 1) return fail(COLA_EUNSUPPORTED, "inverse x pass does not fit on an SM");
    cap = occ * sms;
    resident[dev].store(cap, std::memory_order_release);
  }
  const unsigned grid = (unsigned)std::min<int64_t>((int64_t)N * N / RB, cap);
  LaunchScope ls_(label<N>("c2r"), st);
  launch(k_fft_x_c2r<N, SUB_SQ>, grid, NT, smem, st, in, out, P, tw, scale, err);
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}
template <int N>
static int x_c2r(const float2* in, float* out, int P, const float2* tw, float scale, bool sub_sq, int* err,
                 cudaStream_t st) {
  return sub_sq ? x_c2r_t<N, true>(in, out, P, tw, scale, err, st) : x_c2r_t<N, false>(in, out, P, tw, scale, err, st);
}

template <int N>
static int z_factor(const float2* in, float2* out, int P, const SpectralFactor& factor, const float2* tw,
                    cudaStream_t st) {
  if (P != half_pitch<N>()) return fail(COLA_EINVAL, "fft column pass: unexpected row pitch");
  using Cfg = ColsCfg<N, kColsPlain>;
  constexpr size_t smem = cols_smem<Cfg>(0);
  unsigned grid = 0;
  if (const int rc = cols_grid<Cfg, k_fft_z_factor<N>>(smem, Cfg::STRIPS * N, &grid)) return rc;
  LaunchScope ls_(label<N>("inv"), st);
  launch(k_fft_z_factor<N>, grid, Cfg::THREADS, smem, st, in, out, factor, tw);
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

template <int N, bool INV, bool ALONG_Z>
static int cols_t(float2* data, const float2* tw, cudaStream_t st) {
  using Cfg = ColsCfg<N, kColsPlain>;
  constexpr size_t smem = cols_smem<Cfg>(0);
  unsigned grid = 0;
  if (const int rc = cols_grid<Cfg, k_fft_cols<N, INV, ALONG_Z>>(smem, Cfg::STRIPS * N, &grid)) return rc;
  LaunchScope ls_(label<N>(INV ? "inv" : "fwd"), st);
  launch(k_fft_cols<N, INV, ALONG_Z>, grid, Cfg::THREADS, smem, st, data, tw);
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}
template <int N>
static int cols(bool inverse, bool along_z, float2* data, int P, const float2* tw, cudaStream_t st) {
  if (P != half_pitch<N>()) return fail(COLA_EINVAL, "fft column pass: unexpected row pitch");
  if (inverse) return along_z ? cols_t<N, true, true>(data, tw, st) : cols_t<N, true, false>(data, tw, st);
  return along_z ? cols_t<N, false, true>(data, tw, st) : cols_t<N, false, false>(data, tw, st);
}

#define COLA_FOR_SIZES(X) \
  X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512) X(768) X(1024) X(1536) X(2048)

bool fft_size_supported(int n) {
  switch (n) {
#define X(N) case N:
    COLA_FOR_SIZES(X)
#undef X
    return true;
    default:
      return false;
  }
}

int launch_fft_x_r2c(int n, const float* in, float2* out, int64_t nrows, int P, const float2* tw, cudaStream_t st) {
  switch (n) {
#define X(N) \
  case N:    \
    return x_r2c<N>(in, out, nrows, P, tw, st);
    COLA_FOR_SIZES(X)
#undef X
    default:
      return fail(COLA_EUNSUPPORTED, "fft: unsupported length " + std::to_string(n));
  }
}

int launch_fft_x_r2c3(int n, const float4* in, float2* x, float2* y, float2* z, int P, const float2* tw,
                      cudaStream_t st) {
  const Spectra3 out{{x, y, z}};
  switch (n) {
#define X(N) \
  case N:    \
    return x_r2c3<N>(in, out, P, tw, st);
    COLA_FOR_SIZES(X)
#undef X
    default:
      return fail(COLA_EUNSUPPORTED, "fft: unsupported length " + std::to_string(n));
  }
}

int launch_fft_x_c2r(int n, const float2* in, float* out, int P, const float2* tw, float scale, bool sub_sq, int* err,
                     cudaStream_t st) {
  switch (n) {
#define X(N) \
  case N:    \
    return x_c2r<N>(in, out, P, tw, scale, sub_sq, err, st);
    COLA_FOR_SIZES(X)
#undef X
    default:
      return fail(COLA_EUNSUPPORTED, "fft: unsupported length " + std::to_string(n));
  }
}

int launch_fft_z_factor(int n, int P, double box, int kind, int i, int j, float scale, const float2* in, float2* out,
                        const float2* tw, cudaStream_t st) {
  const SpectralFactor factor{kind, i, j, (float)(2.0 * 3.14159265358979323846 / box), scale};
  switch (n) {
#define X(N) \
  case N:    \
    return z_factor<N>(in, out, P, factor, tw, st);
    COLA_FOR_SIZES(X)
#undef X
    default:
      return fail(COLA_EUNSUPPORTED, "fft: unsupported length " + std::to_string(n));
  }
}

int launch_fft_cols(int n, bool inverse, bool along_z, float2* data, int P, const float2* tw, cudaStream_t st) {
  switch (n) {
#define X(N) \
  case N:    \
    return cols<N>(inverse, along_z, data, P, tw, st);
    COLA_FOR_SIZES(X)
#undef X
    default:
      return fail(COLA_EUNSUPPORTED, "fft: unsupported length " + std::to_string(n));
  }
}

int fft3d_r2c(int n, int P, const float* in, float2* out, const float2* tw, cudaStream_t st) {
  const int64_t nn = n;
  int rc = launch_fft_x_r2c(n, in, out, nn * nn, P, tw, st);
  if (rc) return rc;
  rc = launch_fft_cols(n, false, false, out, P, tw, st);
  if (rc) return rc;
  return launch_fft_cols(n, false, true, out, P, tw, st);
}

int fft3d_c2r(int n, int P, float2* in, float* out, const float2* tw, float scale, int* err, cudaStream_t st) {
  int rc = launch_fft_cols(n, true, true, in, P, tw, st);
  if (rc) return rc;
  rc = launch_fft_cols(n, true, false, in, P, tw, st);
  if (rc) return rc;
  return launch_fft_x_c2r(n, in, out, P, tw, scale, false, err, st);
}

int fft3d_c2r_factor(int n, int P, double box, int kind, int i, int j, float factor_scale, const float2* in,
                     float2* tmp, float* out, bool sub_sq, const float2* tw, int* err, cudaStream_t st) {
  int rc = launch_fft_z_factor(n, P, box, kind, i, j, factor_scale, in, tmp, tw, st);
  if (rc) return rc;
  rc = launch_fft_cols(n, true, false, tmp, P, tw, st);
  if (rc) return rc;
  return launch_fft_x_c2r(n, tmp, out, P, tw, 1.0f, sub_sq, err, st);
}

}  // namespace cola
