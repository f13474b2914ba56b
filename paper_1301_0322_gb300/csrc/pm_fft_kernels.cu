// Fused mesh passes of one PM force evaluation (App. A.1 eq. eom: the force
// -(3/2) Om a d_x d_x^-2 delta; readings: CIC, spectral gradient, 1/W^p deconvolution).
//
// With A the half spectrum [z][y][kx] (rows of P complex), one force evaluation runs
//   1. k_deposit_fftx   CIC deposit of a tile of TY x TZ rows (int64 in shared memory), the
//                       overdensity, and the real-to-complex FFT of those rows -> A
//   2. k_fft_cols       forward y pass on A (fft_kernels.cu)
//   3. k_fft_z_green    forward z pass, then two inverse z passes of
//                       phi_k = delta_k / (k^2 W^p N^3) and of i k_z phi_k   -> B (in A), Gz
//   4. k_fft_y_inv3     inverse y passes: C = IFFT_y(B), Gy = IFFT_y(i k_y B), Gz' = IFFT_y(Gz)
//   5. k_fft_x_c2r3     inverse x passes of (i k_x C, Gy, Gz') -> the three real force meshes
// Steps 3-5 use linearity: i k_x and i k_y are constant along z, so the x and y components
// share the inverse z transform of phi_k, and the x component shares the inverse y transform.
#include "cols_launch.cuh"
#include "pm_bodies.cuh"

namespace cola {

// ---- single-box kernels ------------------------------------------------------------------------
// Threads of the fused deposit: those of the row transforms (8 to 128 for 8 rows), and up to 256
// cells per side more to deposit with: there a tile with a clump in it keeps the few threads of its
// transforms busy long after the other tiles are done.  us per launch with the transforms' threads
// alone -> these: 32^3 mesh and particles 117 -> 11, 64: 16 -> 8, 192 with clumps 78 -> 39, 256 with
// clumps 272 -> 219 (without 76 either way); at 384 128 threads lose (250 -> 263).
template <int N, int TY, int TZ>
__host__ __device__ constexpr int deposit_threads() {
  constexpr int rows = FFTConf<N / 2>::T * TY * TZ, least = N <= 96 ? 256 : (N <= 256 ? 128 : 0);
  return rows < least ? least : rows;
}
// resident blocks per SM it is compiled for, by threads per SM (1024: three blocks of 512 threads at
// 42 registers, 6.9 ms with one -> 5.0; 512: six of 128, 534 -> 509 us; more at 384 or 768 lose);
// three blocks of 2 x 2 tiles at N = 2048 (64 KB of cell sums each; 80 registers, no spills)
template <int N, int TY, int TZ>
__host__ __device__ constexpr int deposit_min_blocks() {
  constexpr int threads = N <= 96 ? 1024 : N <= 256 || N == 512 ? 768 : N == 1024 ? 1536 : 512;
  constexpr int per_sm = threads / deposit_threads<N, TY, TZ>();
  return N == 2048 && TY * TZ == 4 ? 3 : (per_sm > 0 ? per_sm : 1);
}

// cell sums (8 bytes per cell) of a TY x TZ tile, which later hold the rows' transform buffers
template <int N, int TY, int TZ>
__host__ __device__ constexpr int deposit_acc_cells() {
  return TY * TZ * (N > xrow_ld<N / 2>() ? N : xrow_ld<N / 2>());
}
// A tight stage twiddle table (fft.cuh) behind the cell sums at N = 2048 (10.3 KB: three blocks
// of 2 x 2 tiles per SM still fit); below 2048 the table costs more in resident blocks than the
// twiddle loads it saves.
template <int N>
__host__ __device__ constexpr int deposit_table_size() {
  return N == 2048 ? stw_size<FFTConf<N / 2>, true>() : 0;
}

template <int N, int TY, int TZ>
__global__ void __launch_bounds__(deposit_threads<N, TY, TZ>(), deposit_min_blocks<N, TY, TZ>())
    k_deposit_fftx(Geometry g, Tiles tl, const uint4* __restrict__ rec, const int* __restrict__ offsets,
                   float2* __restrict__ out, int P, const float2* __restrict__ tw, float dscale,
                   int* __restrict__ err) {
  extern __shared__ __align__(16) unsigned long long acc[];
  __shared__ int ints[28];
  if constexpr (deposit_table_size<N>() > 0) {
    float2* stab = reinterpret_cast<float2*>(acc + deposit_acc_cells<N, TY, TZ>());
    stw_fill<FFTConf<N / 2>, 2, true>(stab, tw, threadIdx.x, blockDim.x);
    pdl_begin();
    deposit_fftx_body<N, TY, TZ, FFTConf<N / 2>, deposit_threads<N, TY, TZ>()>(
        g, tl, rec, offsets, out, P, tw, SmemTw<FFTConf<N / 2>, true>{stab}, dscale, err, blockIdx.x, acc, ints);
  } else {
    pdl_begin();
    deposit_fftx_body<N, TY, TZ, FFTConf<N / 2>, deposit_threads<N, TY, TZ>()>(g, tl, rec, offsets, out, P, tw, tw,
                                                                               dscale, err, blockIdx.x, acc, ints);
  }
}

template <class Cfg>
using ColsPark = std::conditional_t<Cfg::K == 1, RegPark<Cfg::WORDS>, TmemPark<Cfg::THREADS, Cfg::WORDS>>;

template <int N>
__global__ void __launch_bounds__(ColsCfg<N, kColsZ>::THREADS, ColsCfg<N, kColsZ>::MIN_BLOCKS)
    k_fft_z_green(float2* __restrict__ A, float2* __restrict__ Gz, float kf, int deconv, float norm,
                  const float2* __restrict__ tw) {
  extern __shared__ __align__(16) float2 sm[];
  __shared__ uint32_t slot;
  using Cfg = ColsCfg<N, kColsZ>;
  constexpr int P = half_pitch<N>();
  float2* stab = sm + Cfg::TABLE;
  float* sinc2 = reinterpret_cast<float*>(stab + stw_size<FFTConf<N>>());
  stw_fill<FFTConf<N>, 1>(stab, tw, threadIdx.x, Cfg::THREADS);
  sinc2_fill<N>(sinc2, threadIdx.x, Cfg::THREADS);
  pdl_begin();
  // (after the wait: a predecessor's blocks must not wait for this kernel's tensor memory; its block
  // barrier publishes the tables as well)
  const ColsPark<Cfg> park(&slot);
  const SmemTw<FFTConf<N>> stw{stab};
  cols_walk<Cfg>(A, P, (int64_t)N * P, N, sm, [&](const auto& s, const auto& mem, auto& next) {
    z_green_strip(A, Gz, kf, deconv, norm, stw, sinc2, s, mem, park, next);
  });
  park.close();
}

// the transpose's z pass (z_adjoint_strip): 256^3 74 us, against 77 for three forward passes, 82 for
// the factors in a launch of their own and 26 for the inverse pass
template <int N>
__global__ void __launch_bounds__(ColsCfg<N, kColsZ>::THREADS, ColsCfg<N, kColsZ>::MIN_BLOCKS)
    k_fft_z_adjoint(float2* __restrict__ lx, const float2* __restrict__ ly, const float2* __restrict__ lz, float kf,
                    int deconv, float norm, const float2* __restrict__ tw) {
  extern __shared__ __align__(16) float2 sm[];
  __shared__ uint32_t slot;
  using Cfg = ColsCfg<N, kColsZ>;
  constexpr int P = half_pitch<N>();
  float2* stab = sm + Cfg::TABLE;
  float* sinc2 = reinterpret_cast<float*>(stab + stw_size<FFTConf<N>>());
  stw_fill<FFTConf<N>, 1>(stab, tw, threadIdx.x, Cfg::THREADS);
  sinc2_fill<N>(sinc2, threadIdx.x, Cfg::THREADS);
  pdl_begin();
  const ColsPark<Cfg> park(&slot);
  const SmemTw<FFTConf<N>> stw{stab};
  cols_walk<Cfg>(lx, P, (int64_t)N * P, N, sm, [&](const auto& s, const auto& mem, auto& next) {
    z_adjoint_strip(lx, ly, lz, kf, deconv, norm, stw, sinc2, s, mem, park, next);
  });
  park.close();
}

template <int N>
__global__ void __launch_bounds__(ColsCfg<N, kColsY>::THREADS, ColsCfg<N, kColsY>::MIN_BLOCKS)
    k_fft_y_inv3(float2* __restrict__ B, float2* __restrict__ Gy, float2* __restrict__ Gz, float kf,
                 const float2* __restrict__ tw) {
  extern __shared__ __align__(16) float2 sm[];
  __shared__ uint32_t slot;
  using Cfg = ColsCfg<N, kColsY>;
  constexpr int P = half_pitch<N>();
  float2* stab = sm + Cfg::TABLE;
  stw_fill<FFTConf<N>, 1>(stab, tw, threadIdx.x, Cfg::THREADS);
  pdl_begin();
  const ColsPark<Cfg> park(&slot);
  const SmemTw<FFTConf<N>> stw{stab};
  cols_walk<Cfg>(B, (int64_t)N * P, P, N, sm, [&](const auto& s, const auto& mem, auto& next) {
    y_inv3_strip(B, Gy, Gz, kf, stw, s, mem, park, next);
  });
  park.close();
}

// resident blocks per SM of the inverse-x pass: four at N = 2048 (128 registers, no spills;
// 16 warps to cover the shared-memory latency of the staged rows), three otherwise
template <int N>
__host__ __device__ constexpr int c2r3_min_blocks() {
  return N == 2048 ? 4 : 3;
}

template <int N>
__global__ void __launch_bounds__(FFTConf<N / 2>::T * c2r3_rows<N>(), c2r3_min_blocks<N>())
    k_fft_x_c2r3(const float2* __restrict__ C, const float2* __restrict__ Gy, const float2* __restrict__ Gz,
                 float* __restrict__ F, int P, float kf, const float2* __restrict__ tw, int* __restrict__ err) {
  constexpr int M = N / 2, RB = c2r3_rows<N>(), LD = xrow_ld<M>();
  extern __shared__ __align__(128) float2 c2r_stage[];
  __shared__ __align__(8) uint64_t bars[2];
  const int64_t nrb = (int64_t)N * N / RB;
  // stage twiddles, copied once per block (persistent) behind the staging buffers
  float2* stab = c2r_stage + 2 * RB * LD;
  stw_fill<FFTConf<M>, 2>(stab, tw, threadIdx.x, blockDim.x);
  const SmemTw<FFTConf<M>> stw{stab};
  pdl_begin();
  c2r_walk<N, RB>(
      c2r_stage, bars, 3 * nrb, P, err,
      [&](int64_t item) -> const float2* {
        const int comp = (int)(item / nrb);
        const float2* m = comp == 0 ? C : (comp == 1 ? Gy : Gz);
        return m + (item - comp * nrb) * RB * P;
      },
      [&](int64_t item, float2* rows) {
        const int comp = (int)(item / nrb);
        const int64_t row0 = (item - comp * nrb) * RB;
        c2r3_compute<N, RB>(rows, F + (int64_t)comp * N * N * N + row0 * N, comp, kf, tw, stw);
      });
}

// ---- launchers ---------------------------------------------------------------------------------------------------
template <class K>
static int set_smem(K kernel, size_t bytes) {
  if (bytes > 227 * 1024) return fail(COLA_EUNSUPPORTED, "fused FFT kernel: shared memory request too large");
  if (bytes > 32 * 1024)
    COLA_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  return COLA_OK;
}

template <int N>
static const char* flabel(int kind) {
  static const std::string names[4] = {std::string("deposit_fftx_") + std::to_string(N),
                                       std::string("fft_z_green_") + std::to_string(N),
                                       std::string("fft_y_inv3_") + std::to_string(N),
                                       std::string("fft_x_c2r3_") + std::to_string(N)};
  return names[kind].c_str();
}

// 1. deposit + x r2c of every tile into the half spectrum A
template <int N>
static int deposit_fftx_t(const Geometry& g, const Tiles& tl, const uint4* rec, const int* offsets, float2* A, int P,
                          const float2* tw, int* err, cudaStream_t st) {
  int rc;
  const double n3 = (double)N * N * N;
  const float dscale = (float)(n3 / ((double)g.np3 * std::ldexp(1.0, 3 * g.fbits)));
  if (tl.ty == 4 && tl.tz == 2) {
    const size_t smem = sizeof(unsigned long long) * (deposit_acc_cells<N, 4, 2>() + deposit_table_size<N>());
    if ((rc = set_smem(k_deposit_fftx<N, 4, 2>, smem))) return rc;
    LaunchScope ls_(flabel<N>(0), st);
    launch(k_deposit_fftx<N, 4, 2>, tl.nty * tl.ntz, deposit_threads<N, 4, 2>(), smem, st, g, tl, rec, offsets, A, P, tw, dscale, err);
  } else if (tl.ty == 2 && tl.tz == 2) {
    const size_t smem = sizeof(unsigned long long) * (deposit_acc_cells<N, 2, 2>() + deposit_table_size<N>());
    if ((rc = set_smem(k_deposit_fftx<N, 2, 2>, smem))) return rc;
    LaunchScope ls_(flabel<N>(0), st);
    launch(k_deposit_fftx<N, 2, 2>, tl.nty * tl.ntz, deposit_threads<N, 2, 2>(), smem, st, g, tl, rec, offsets, A, P, tw, dscale, err);
  } else {
    return fail(COLA_EUNSUPPORTED, "fused deposit: unsupported tile shape");
  }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

template <int N>
static int force_passes_t(const Geometry& g, const Tiles& tl, const uint4* rec, const int* offsets,
                          float2* A, float2* Gy, float2* Gz, float* F, int P, double box, int deconv,
                          const float2* tw, int* err, cudaStream_t st) {
  constexpr int M = N / 2;
  const float kf = (float)(2.0 * 3.14159265358979323846 / box);
  const float norm = (float)(1.0 / ((double)N * N * N));
  if (P != half_pitch<N>()) return fail(COLA_EINVAL, "force passes: unexpected half-spectrum pitch");
  int rc;
  if ((rc = deposit_fftx_t<N>(g, tl, rec, offsets, A, P, tw, err, st))) return rc;
  // 2. forward y pass
  if ((rc = launch_fft_cols(N, false, false, A, P, tw, st))) return rc;
  unsigned grid = 0;
  // 3. z pass with the Green's function
  {
    using Cfg = ColsCfg<N, kColsZ>;
    constexpr size_t smem = cols_smem<Cfg>(N);
    if ((rc = cols_grid<Cfg, k_fft_z_green<N>>(smem, Cfg::STRIPS * N, &grid))) return rc;
    LaunchScope ls_(flabel<N>(1), st);
    launch(k_fft_z_green<N>, grid, Cfg::THREADS, smem, st, A, Gz, kf, deconv, norm, tw);
    COLA_LAUNCH_CHECK();
  }
  // 4. inverse y passes
  {
    using Cfg = ColsCfg<N, kColsY>;
    constexpr size_t smem = cols_smem<Cfg>(0);
    if ((rc = cols_grid<Cfg, k_fft_y_inv3<N>>(smem, Cfg::STRIPS * N, &grid))) return rc;
    LaunchScope ls_(flabel<N>(2), st);
    launch(k_fft_y_inv3<N>, grid, Cfg::THREADS, smem, st, A, Gy, Gz, kf, tw);
    COLA_LAUNCH_CHECK();
  }
  // 5. inverse x passes (persistent, bulk-copy pipelined)
  {
    constexpr int RB = c2r3_rows<N>(), T = FFTConf<M>::T;
    const size_t smem = sizeof(float2) * (2 * RB * xrow_ld<M>() + stw_size<FFTConf<M>>());
    if ((rc = set_smem(k_fft_x_c2r3<N>, smem))) return rc;
    const int64_t nrows = (int64_t)N * N;
    if (nrows % RB) return fail(COLA_EINVAL, "fused c2r: row count not a multiple of the block rows");
    if (P % 4) return fail(COLA_EINVAL, "fused c2r: row pitch must be a multiple of 4 complex");
    // resident blocks x SMs of the current device (cached per device)
    static int grid_cap[64] = {};
    int dev = 0;
    COLA_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(COLA_EUNSUPPORTED, "device index above 63");
    if (!grid_cap[dev]) {
      int occ = 0, sms = 0;
      COLA_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_fft_x_c2r3<N>, T * RB, smem));
      COLA_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
      if (occ < 1) return fail(COLA_EUNSUPPORTED, "fused c2r does not fit on an SM");
      grid_cap[dev] = occ * sms;
    }
    const int64_t items = 3 * nrows / RB;
    const unsigned grid = (unsigned)std::min<int64_t>(items, grid_cap[dev]);
    LaunchScope ls_(flabel<N>(3), st);
    launch(k_fft_x_c2r3<N>, grid, T * RB, smem, st, A, Gy, Gz, F, P, kf, tw, err);
    COLA_LAUNCH_CHECK();
  }
  return COLA_OK;
}

template <int N>
static int z_adjoint_t(int P, double box, int deconv, float2* lx, const float2* ly, const float2* lz, const float2* tw,
                       cudaStream_t st) {
  using Cfg = ColsCfg<N, kColsZ>;
  if (P != half_pitch<N>()) return fail(COLA_EINVAL, "adjoint z pass: unexpected half-spectrum pitch");
  const float kf = (float)(2.0 * 3.14159265358979323846 / box);
  const float norm = (float)(1.0 / ((double)N * N * N));
  constexpr size_t smem = cols_smem<Cfg>(N);
  unsigned grid = 0;
  if (const int rc = cols_grid<Cfg, k_fft_z_adjoint<N>>(smem, Cfg::STRIPS * N, &grid)) return rc;
  LaunchScope ls_("fft_z_adjoint", st);
  launch(k_fft_z_adjoint<N>, grid, Cfg::THREADS, smem, st, lx, ly, lz, kf, deconv, norm, tw);
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

int launch_z_adjoint(int ng, int P, double box, int deconv, float2* lx, const float2* ly, const float2* lz,
                     const float2* tw, cudaStream_t st) {
  switch (ng) {
#define X(N) \
  case N:    \
    return z_adjoint_t<N>(P, box, deconv, lx, ly, lz, tw, st);
    X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512) X(768) X(1024) X(1536) X(2048)
#undef X
    default:
      return fail(COLA_EUNSUPPORTED, "adjoint z pass: unsupported mesh size");
  }
}

int launch_density_spectrum(const Geometry& g, const Tiles& tl, const uint4* rec, const int* offsets, float2* A,
                            int P, const float2* tw, int* err, cudaStream_t st) {
  switch (g.ng) {
#define X(N)                                                                                          \
  case N: {                                                                                           \
    int rc;                                                                                           \
    if ((rc = deposit_fftx_t<N>(g, tl, rec, offsets, A, P, tw, err, st))) return rc;                  \
    if ((rc = launch_fft_cols(N, false, false, A, P, tw, st))) return rc;                                       \
    return launch_fft_cols(N, false, true, A, P, tw, st);                                              \
  }
    X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512) X(768) X(1024) X(1536) X(2048)
#undef X
    default:
      return fail(COLA_EUNSUPPORTED, "density spectrum: unsupported mesh size");
  }
}

int launch_force_passes(const Geometry& g, const Tiles& tl, const uint4* rec, const int* offsets,
                        float2* A, float2* Gy, float2* Gz, float* F, int P, double box, int deconv, const float2* tw,
                        int* err, cudaStream_t st) {
  switch (g.ng) {
#define X(N) \
  case N:    \
    return force_passes_t<N>(g, tl, rec, offsets, A, Gy, Gz, F, P, box, deconv, tw, err, st);
    X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512) X(768) X(1024) X(1536) X(2048)
#undef X
    default:
      return fail(COLA_EUNSUPPORTED, "force passes: unsupported mesh size");
  }
}

}  // namespace cola
