// Particle-mesh kernels of a COLA force evaluation (Sec. 2 PM code; App. A.1 eq. eom;
// App. A.3 eq. KDKALC):
//   binning  : particles -> (y, z) row tiles of the mesh (counting sort, integer atomics)
//   deposit  : CIC mass of every particle touching a tile, int64 fixed point in shared memory
//              (integer sums: the result does not depend on the order of the atomics)
//   k-space  : g_j = i k_j delta_k / (k^2 W^p) / ng^3 (Nyquist plane of j and k = 0 set to 0)
//   gather   : CIC interpolation of g with the deposit's weights, fused with the COLA Kick and
//              Drift (or the final L+ of eq. Lops)
#include "cola_internal.cuh"
#include "pm_common.cuh"
#include "particle_bodies.cuh"

namespace cola {

// ---- binning -------------------------------------------------------------------------------
// four particles per thread (ranks_x4_body or count_x4_body)
template <bool RANK>
__global__ void __launch_bounds__(256) k_keys_x4(Geometry g, Tiles tl, const float* __restrict__ s,
                                                 int* __restrict__ ranks, int* __restrict__ counts,
                                                 int* __restrict__ err) {
  pdl_begin();
  const int64_t q0 = (int64_t)blockIdx.x * blockDim.x * kPartPerThread;
  if constexpr (RANK) ranks_x4_body(g, tl, s, q0, 0, ranks, counts, err);
  else count_x4_body(g, tl, s, q0, counts, err);
}

// Exclusive scan of the bin counts in three launches (block sums, scan of the block sums,
// per-block scan); resets the counts for the next use.  kScanTile bins per block.
constexpr int kScanTile = 1024;

// inclusive block scan of one int per thread (blockDim.x == 1024)
__device__ __forceinline__ int block_inclusive_scan(int x, int* warp_sums) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int ws = warp_sums[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, ws, o);
      if (lane >= o) ws += y;
    }
    warp_sums[lane] = ws;
  }
  __syncthreads();
  return x + (wid > 0 ? warp_sums[wid - 1] : 0);
}

__global__ void __launch_bounds__(1024) k_scan_reduce(int n, const int* __restrict__ counts, int* __restrict__ block_sums) {
  pdl_begin();
  __shared__ int warp_sums[32];
  const int i = blockIdx.x * kScanTile + threadIdx.x;
  const int x = i < n ? counts[i] : 0;
  const int incl = block_inclusive_scan(x, warp_sums);
  if (threadIdx.x == kScanTile - 1) block_sums[blockIdx.x] = incl;
}

// exclusive scan of nb block sums in place (single block; nb <= 1024 * per)
__global__ void __launch_bounds__(1024) k_scan_blocks(int nb, int* __restrict__ block_sums) {
  pdl_begin();
  __shared__ int warp_sums[32];
  const int per = (nb + 1023) / 1024;
  const int b0 = min(nb, (int)threadIdx.x * per), b1 = min(nb, b0 + per);
  int local = 0;
  for (int b = b0; b < b1; ++b) local += block_sums[b];
  int run = block_inclusive_scan(local, warp_sums) - local;
  for (int b = b0; b < b1; ++b) {
    const int c = block_sums[b];
    block_sums[b] = run;
    run += c;
  }
}

// (shift 1: bin i's offset goes to offsets[i + 1], where the scatter takes it as a running cursor and
// leaves the bin's end, the next one's offset)
__global__ void __launch_bounds__(1024) k_scan_apply(int n, int* __restrict__ counts, const int* __restrict__ block_sums,
                                                    int* __restrict__ offsets, int shift) {
  pdl_begin();
  __shared__ int warp_sums[32];
  const int i = blockIdx.x * kScanTile + threadIdx.x;
  const int x = i < n ? counts[i] : 0;
  const int excl = block_inclusive_scan(x, warp_sums) - x + block_sums[blockIdx.x];
  if (i < n) {
    offsets[i + shift] = excl;
    counts[i] = 0;
  }
  if (shift && i == 0) offsets[0] = 0;
  if (!shift && i == n - 1) offsets[n] = excl + x;
}

// The three launches as one block for up to kScanOne bins (meshes up to 256): every count is loaded
// before the first is needed, so the block waits for memory once (6 us in all against 3 x 6).
constexpr int kScanOne = 32768;
__global__ void __launch_bounds__(1024) k_scan_one(int n, int* __restrict__ counts, int* __restrict__ offsets) {
  pdl_begin();
  constexpr int R = kScanOne / 4096;
  __shared__ int warp_sums[32];
  int4 v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = r * 4096 + 4 * threadIdx.x;
    v[r] = i < n ? *reinterpret_cast<const int4*>(counts + i) : make_int4(0, 0, 0, 0);  // (n is a multiple of 4)
  }
  int run = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r * 4096 >= n) break;
    const int x = v[r].x + v[r].y + v[r].z + v[r].w;
    const int incl = block_inclusive_scan(x, warp_sums);
    const int total = warp_sums[31], e = run + incl - x, i = r * 4096 + 4 * threadIdx.x;
    if (i < n) {
      const int4 o = make_int4(e, e + v[r].x, e + v[r].x + v[r].y, e + v[r].x + v[r].y + v[r].z);
      *reinterpret_cast<int4*>(offsets + i) = o;
      *reinterpret_cast<int4*>(counts + i) = make_int4(0, 0, 0, 0);
    }
    run += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) offsets[n] = run;
}

// four particles per thread (scatter_x4_body or place_x4_body, whose cursors are the words from
// offsets[1], see k_scan_apply)
template <bool RANK>
__global__ void __launch_bounds__(256) k_scatter_x4(Geometry g, Tiles tl, const float* __restrict__ s,
                                                    const int* __restrict__ ranks, int* __restrict__ offsets,
                                                    uint4* __restrict__ rec) {
  pdl_begin();
  const int64_t q0 = (int64_t)blockIdx.x * blockDim.x * kPartPerThread;
  if constexpr (RANK) scatter_x4_body(g, tl, s, q0, 0, ranks, offsets, rec);
  else place_x4_body(g, tl, s, q0, offsets + 1, rec);
}

// ---- deposit ----------------------------------------------------------------------------------
// One block per tile of TY x TZ mesh rows (whole x extent).  It reads the bin-ordered records
// (fixed-point CIC coordinates, stored by the scatter) of the particles binned to the tile and to
// the boundary regions of its three lower neighbours, accumulates exact int64 CIC weights in
// shared memory and writes the rows once (int64 and/or float overdensity).  The outputs are the
// caller's: PAIRS stores two cells per access, which takes a rho of 16 and a delta of 8 bytes
// alignment; other buffers (slices of larger ones) get one cell per access.
template <int TY, int TZ, bool PAIRS>
__global__ void __launch_bounds__(256) k_deposit(Geometry g, Tiles tl, const uint4* __restrict__ rec,
                                                 const int* __restrict__ offsets, int64_t* __restrict__ rho,
                                                 float* __restrict__ delta, float dscale, int* __restrict__ err) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned long long acc[];
  __shared__ int rbeg[9], rpre[10];
  const int ng = g.ng;
  int tyi, tzi;
  tile_of_bin(tl, blockIdx.x, tyi, tzi);
  const int y0 = tyi * TY, z0 = tzi * TZ;
  const int ncell = TZ * TY * ng;
  for (int i = threadIdx.x; i < ncell / 2; i += blockDim.x)
    reinterpret_cast<ulonglong2*>(acc)[i] = make_ulonglong2(0ull, 0ull);
  if (threadIdx.x == 0) {
    const int tym = tyi == 0 ? tl.nty - 1 : tyi - 1;
    const int tzm = tzi == 0 ? tl.ntz - 1 : tzi - 1;
    const int tys[9] = {tyi, tyi, tyi, tyi, tym, tym, tyi, tyi, tym};
    const int tzs[9] = {tzi, tzi, tzi, tzi, tzi, tzi, tzm, tzm, tzm};
    const int reg[9] = {0, 1, 2, 3, 1, 3, 2, 3, 3};
    int run = 0;
    for (int k = 0; k < 9; ++k) {
      const int b = tile_bin(tl, tys[k], tzs[k]) * 4 + reg[k];
      rbeg[k] = offsets[b];
      rpre[k] = run;
      run += offsets[b + 1] - offsets[b];
    }
    rpre[9] = run;
  }
  __syncthreads();
  const int total = rpre[9];
  unsigned* lo = reinterpret_cast<unsigned*>(acc);
  unsigned* hi = lo + ncell;
  constexpr int U = 4;  // particles in flight per thread
  for (int base = threadIdx.x; base < total; base += U * blockDim.x) {
    uint32_t f[U][3];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + u * blockDim.x;
      if (i < total) {
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
      if (base + u * (int)blockDim.x < total) acc_cloud<TY, TZ, false>(lo, hi, f[u], g.fbits, ng, y0, z0);
  }
  __syncthreads();
  // two cells per thread, row by row (no division per cell; ng is a multiple of 4)
  bool overflow = false;
  for (int r = 0; r < TY * TZ; ++r) {
    const int64_t row = ((int64_t)(z0 + r / TY) * ng + (y0 + r % TY)) * ng;
    const uint2* l2 = reinterpret_cast<const uint2*>(lo + r * ng);
    const uint2* h2 = reinterpret_cast<const uint2*>(hi + r * ng);
    for (int x = threadIdx.x; x < ng / 2; x += blockDim.x) {
      const uint2 l = l2[x], h = h2[x];
      const unsigned long long a = ((unsigned long long)h.x << 32) | l.x, b = ((unsigned long long)h.y << 32) | l.y;
      overflow |= ((h.x | h.y) >> 30) != 0u;
      if (rho) {
        if constexpr (PAIRS) {
          longlong2 v;
          v.x = (int64_t)a;
          v.y = (int64_t)b;
          reinterpret_cast<longlong2*>(rho + row)[x] = v;
        } else {
          rho[row + 2 * x] = (int64_t)a;
          rho[row + 2 * x + 1] = (int64_t)b;
        }
      }
      if (delta) {
        const float2 d = make_float2(fmaf(__ull2float_rn(a), dscale, -1.0f), fmaf(__ull2float_rn(b), dscale, -1.0f));
        if constexpr (PAIRS) {
          reinterpret_cast<float2*>(delta + row)[x] = d;
        } else {
          delta[row + 2 * x] = d.x;
          delta[row + 2 * x + 1] = d.y;
        }
      }
    }
  }
  if (overflow) atomicOr(err, kErrOverflow);
}

// ---- gather + kick + drift -------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_gather_kick_drift(Geometry g, const float* __restrict__ fmesh,
                                                            float* __restrict__ s, float* __restrict__ v,
                                                            const float* __restrict__ s1, const float* __restrict__ s2,
                                                            const float* __restrict__ coef, int mode,
                                                            float* __restrict__ gout) {
  pdl_begin();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < g.np3) gather_kick_drift_body(g, fmesh, s, v, s1, s2, coef, mode, gout, p);
}

// Gather in bin order: thread i takes the particle of bin position i from its record (lattice
// index p and the fixed-point coordinates, which equal fixed_axis of the current s), so the
// threads of a block read neighbouring mesh rows however clustered the particles are; the
// force goes to fj[p].
__global__ void __launch_bounds__(256) k_gather_binned(Geometry g, const float* __restrict__ fmesh,
                                                        const uint4* __restrict__ rec, float* __restrict__ f0,
                                                        float* __restrict__ f1, float* __restrict__ f2) {
  pdl_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.np3) return;
  const uint4 q = __ldg(rec + i);
  const int64_t p = q.w;
  const uint32_t fmask = (1u << g.fbits) - 1u;
  const uint32_t fq[3] = {q.x, q.y, q.z};
  int c[3], t[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    c[d] = (int)(fq[d] >> g.fbits);
    t[d] = (int)(fq[d] & fmask);
  }
  float f[3];
  gather_force(g, fmesh, c, t, f);
  f0[p] = f[0];
  f1[p] = f[1];
  f2[p] = f[2];
}

// As k_gather_binned, with the three components written as one 16-byte float4 at the particle's
// lattice index: once the particles cluster, consecutive bin positions belong to scattered
// lattice indices, and one 16-byte write touches one 32-byte sector where three 4-byte writes
// to three arrays touch three.
__global__ void __launch_bounds__(256) k_gather_binned4(Geometry g, const float* __restrict__ fmesh,
                                                         const uint4* __restrict__ rec, float4* __restrict__ f4) {
  pdl_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.np3) return;
  const uint4 q = __ldg(rec + i);
  const uint32_t fmask = (1u << g.fbits) - 1u;
  const uint32_t fq[3] = {q.x, q.y, q.z};
  int c[3], t[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    c[d] = (int)(fq[d] >> g.fbits);
    t[d] = (int)(fq[d] & fmask);
  }
  float f[3];
  gather_force(g, fmesh, c, t, f);
  f4[q.w] = make_float4(f[0], f[1], f[2], 0.0f);
}

// Kick/drift in lattice order with the forces of k_gather_binned4.
__global__ void __launch_bounds__(256) k_kick_drift4(Geometry g, const float4* __restrict__ f4,
                                                      float* __restrict__ s, float* __restrict__ v,
                                                      const float* __restrict__ s1, const float* __restrict__ s2,
                                                      const float* __restrict__ coef, int mode) {
  pdl_begin();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= g.np3) return;
  const float4 q = __ldg(f4 + p);
  const float f[3] = {q.x, q.y, q.z};
  kick_drift_update(g, s, v, s1, s2, coef, mode, p, f);
}

// Kick/drift in lattice order with the gathered force fj[p].
__global__ void __launch_bounds__(256) k_kick_drift(Geometry g, const float* __restrict__ f0,
                                                     const float* __restrict__ f1, const float* __restrict__ f2,
                                                     float* __restrict__ s, float* __restrict__ v,
                                                     const float* __restrict__ s1, const float* __restrict__ s2,
                                                     const float* __restrict__ coef, int mode) {
  pdl_begin();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= g.np3) return;
  const float f[3] = {f0[p], f1[p], f2[p]};
  kick_drift_update(g, s, v, s1, s2, coef, mode, p, f);
}

// ---- launchers ------------------------------------------------------------------------------------
static unsigned blocks_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// Ranks pay where the lanes of a warp share bins: meshes no finer than the lattice.  On finer ones, and
// at the largest lattices, the count waits for more atomics to return than the scatter saves.  us,
// count + scatter of an evolved state, particles on mesh, ranked / counted: 512^3 on 512^3 1905 /
// 2012, 768 on 768 6258 / 6394 | 1024 on 1024 14395 / 13928, 256 on 768 314 / 299, 384 on 768 954 /
// 908, 512 on 1024 2195 / 1996, 768 on 1536 7562 / 6936, 1024 on 2048 20319 / 18184.  At 384 and
// below they are as good (192 on 384 129 / 128, 128 on 384 45 / 47): ranked, as are the ensembles' bins.
bool bins_ranked(const Geometry& g) { return g.ng <= 384 || (g.ng <= g.np && g.np <= 768); }

int launch_keys(const Geometry& g, const Tiles& t, const float* s, int* ranks, int* counts, int* err, cudaStream_t st) {
  const unsigned blocks = blocks_for(g.np3, 256 * kPartPerThread);
  { LaunchScope ls_(bins_ranked(g) ? "keys" : "count", st);
  if (bins_ranked(g)) launch(k_keys_x4<true>, blocks, 256, 0, st, g, t, s, ranks, counts, err);
  else launch(k_keys_x4<false>, blocks, 256, 0, st, g, t, s, ranks, counts, err); }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

int scan_block_count(const Tiles& t) { return (t.nbins + kScanTile - 1) / kScanTile; }

int launch_scan(const Tiles& t, int* counts, int* offsets, int* block_sums, bool one_block, bool cursors,
                cudaStream_t st) {
  if (one_block && !cursors && t.nbins <= kScanOne && t.nbins % 4 == 0) {
    LaunchScope ls_("scan_one", st);
    launch(k_scan_one, 1, 1024, 0, st, t.nbins, counts, offsets);
    COLA_LAUNCH_CHECK();
    return COLA_OK;
  }
  const int nb = scan_block_count(t);
  {
    LaunchScope ls_("scan_reduce", st);
    launch(k_scan_reduce, nb, kScanTile, 0, st, t.nbins, counts, block_sums);
  }
  COLA_LAUNCH_CHECK();
  {
    LaunchScope ls_("scan_blocks", st);
    launch(k_scan_blocks, 1, 1024, 0, st, nb, block_sums);
  }
  COLA_LAUNCH_CHECK();
  {
    LaunchScope ls_("scan_apply", st);
    launch(k_scan_apply, nb, kScanTile, 0, st, t.nbins, counts, block_sums, offsets, cursors ? 1 : 0);
  }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

int launch_scatter(const Geometry& g, const Tiles& t, const float* s, const int* ranks, int* offsets, uint4* rec,
                   cudaStream_t st) {
  const unsigned blocks = blocks_for(g.np3, 256 * kPartPerThread);
  { LaunchScope ls_(bins_ranked(g) ? "scatter" : "place", st);
  if (bins_ranked(g)) launch(k_scatter_x4<true>, blocks, 256, 0, st, g, t, s, ranks, offsets, rec);
  else launch(k_scatter_x4<false>, blocks, 256, 0, st, g, t, s, ranks, offsets, rec); }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

template <int TY, int TZ, bool PAIRS>
static int deposit_t(const Geometry& g, const Tiles& t, const uint4* rec, const int* offsets, int64_t* rho,
                     float* delta, int* err, cudaStream_t st) {
  const size_t smem = (size_t)TY * TZ * g.ng * sizeof(unsigned long long);
  if (smem > 227 * 1024) return fail(COLA_EUNSUPPORTED, "deposit tile does not fit in shared memory");
  if (smem > 32 * 1024)
    COLA_CUDA_CHECK(cudaFuncSetAttribute(k_deposit<TY, TZ, PAIRS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const double ng3 = (double)g.ng * g.ng * g.ng;
  const float dscale = (float)(ng3 / ((double)g.np3 * std::ldexp(1.0, 3 * g.fbits)));
  { LaunchScope ls_(TY == 2 ? "deposit_2x2" : (TZ == 2 ? "deposit_4x2" : "deposit_4x4"), st);
  launch(k_deposit<TY, TZ, PAIRS>, t.nty * t.ntz, 256, smem, st, g, t, rec, offsets, rho, delta, dscale, err); }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

template <int TY, int TZ>
static int deposit_any(const Geometry& g, const Tiles& t, const uint4* rec, const int* offsets, int64_t* rho,
                       float* delta, int* err, cudaStream_t st) {
  // (a null output is aligned; rows are multiples of 16 cells)
  const bool pairs = reinterpret_cast<uintptr_t>(rho) % 16 == 0 && reinterpret_cast<uintptr_t>(delta) % 8 == 0;
  return pairs ? deposit_t<TY, TZ, true>(g, t, rec, offsets, rho, delta, err, st)
               : deposit_t<TY, TZ, false>(g, t, rec, offsets, rho, delta, err, st);
}

int launch_deposit(const Geometry& g, const Tiles& t, const uint4* rec, const int* offsets, int64_t* rho,
                   float* delta, int* err, cudaStream_t st) {
  if (t.ty == 4 && t.tz == 4) return deposit_any<4, 4>(g, t, rec, offsets, rho, delta, err, st);
  if (t.ty == 4 && t.tz == 2) return deposit_any<4, 2>(g, t, rec, offsets, rho, delta, err, st);
  if (t.ty == 2 && t.tz == 2) return deposit_any<2, 2>(g, t, rec, offsets, rho, delta, err, st);
  return fail(COLA_EUNSUPPORTED, "deposit: unsupported tile shape");
}

int launch_gather_kick_drift(const Geometry& g, const float* fmesh, float* s, float* v, const float* s1,
                             const float* s2, const float* coef_row, int mode, float* gout, cudaStream_t st) {
  { LaunchScope ls_("gather_kick_drift", st);
  launch(k_gather_kick_drift, blocks_for(g.np3, 256), 256, 0, st, g, fmesh, s, v, s1, s2, coef_row, mode, gout); }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

int launch_gather_binned(const Geometry& g, const float* fmesh, const uint4* rec,
                         float* f0, float* f1, float* f2, cudaStream_t st) {
  { LaunchScope ls_("gather_binned", st);
  launch(k_gather_binned, blocks_for(g.np3, 256), 256, 0, st, g, fmesh, rec, f0, f1, f2); }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

int launch_gather_binned4(const Geometry& g, const float* fmesh, const uint4* rec, float4* f4, cudaStream_t st) {
  { LaunchScope ls_("gather_binned4", st);
  launch(k_gather_binned4, blocks_for(g.np3, 256), 256, 0, st, g, fmesh, rec, f4); }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

int launch_kick_drift4(const Geometry& g, const float4* f4, float* s, float* v, const float* s1, const float* s2,
                       const float* coef_row, int mode, cudaStream_t st) {
  { LaunchScope ls_("kick_drift4", st);
  launch(k_kick_drift4, blocks_for(g.np3, 256), 256, 0, st, g, f4, s, v, s1, s2, coef_row, mode); }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

int launch_kick_drift(const Geometry& g, const float* f0, const float* f1, const float* f2, float* s, float* v,
                      const float* s1, const float* s2, const float* coef_row, int mode, cudaStream_t st) {
  { LaunchScope ls_("kick_drift", st);
  launch(k_kick_drift, blocks_for(g.np3, 256), 256, 0, st, g, f0, f1, f2, s, v, s1, s2, coef_row, mode); }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

}  // namespace cola
