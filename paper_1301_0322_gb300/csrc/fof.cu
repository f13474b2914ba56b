// Friends-of-friends halo groups (Sec. 3.2) on the GPU.
//
// Positions are the particles' fixed-point CIC coordinates f (mesh cells x 2^F, the PM
// force's own quantised positions).  Two particles are friends iff den^2 |d|^2 < num^2 s^2
// with d the periodic minimum-image separation and s = (ng/np) 2^F the mean separation
// (b = num/den, 1/5 in the paper): an exact integer test, so the groups do not depend on
// rounding or on the order of the atomics.
//
//   1. cells of `csize` mesh cells (>= the linking length): per particle its cell and its rank
//      among the cell's particles (the value its count atomic returns); an in-place scan of the
//      counts; records (f and the lattice index) into cell order, offset + rank
//   2. link: sixteen lanes per particle (cell order) take the rest of its cell and the 13 cells
//      ahead of it, five runs of neighbouring cells along x, and unite it with every friend there:
//      lock-free union-find whose roots always point to smaller positions (compare-and-swap,
//      bounded retries)
//   3. compress every path to its root, count group sizes, smallest original index per group
//   4. per particle: group label (smallest particle index of its group, -1 below nmin) and
//      group size; per threshold: number of halos with at least that many particles
#include <climits>
#include <cstring>

#include "cola_internal.cuh"
#include "particle_bodies.cuh"

namespace cola {
namespace {

constexpr int kMaxThresholds = 32;

struct Thresholds {
  int n;
  int v[kMaxThresholds];
};

// cell of particle p (-1 past the last one): the fixed-point coordinates' mesh cells / csize
__device__ __forceinline__ int fof_cell(const Geometry& g, int64_t p, float sx, float sy, float sz, int csize, int nc) {
  int ix, iy, iz;
  lattice_index(g, p, ix, iy, iz);
  int cx, cy, cz, t;
  fixed_axis(g, ix, sx, cx, t);
  fixed_axis(g, iy, sy, cy, t);
  fixed_axis(g, iz, sz, cz, t);
  if (csize > 1) {
    cx /= csize;
    cy /= csize;
    cz /= csize;
  }
  return (cz * nc + cy) * nc + cx;
}

// key and rank of each particle, four per thread (their loads and atomics in flight together)
__global__ void __launch_bounds__(256) k_fof_keys(Geometry g, const float* __restrict__ s, int csize, int nc,
                                                  int* __restrict__ keys, int* __restrict__ ranks,
                                                  int* __restrict__ counts, int* __restrict__ err) {
  constexpr int U = kPartPerThread;
  const int64_t p0 = x4_first((int64_t)blockIdx.x * blockDim.x * U);
  float sx[U], sy[U], sz[U];
  int key[U], rank[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t p = p0 + 32 * u;
    if (p < g.np3) {
      sx[u] = __ldg(s + p);
      sy[u] = __ldg(s + g.np3 + p);
      sz[u] = __ldg(s + 2 * g.np3 + p);
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t p = p0 + 32 * u;
    if (p < g.np3) {
      if (!isfinite(sx[u]) || !isfinite(sy[u]) || !isfinite(sz[u])) atomicOr(err, kErrNonFinite);
      key[u] = fof_cell(g, p, sx[u], sy[u], sz[u], csize, nc);
      rank[u] = atomicAdd(counts + key[u], 1);
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t p = p0 + 32 * u;
    if (p < g.np3) {
      keys[p] = key[u];
      ranks[p] = rank[u];
    }
  }
}

// ---- scan of the cell counts, in place ------------------------------------------------------
// At cells of one mesh cell the 768^3 counts are 1.8 GB: block sums (one read), a scan of them,
// and one read and one write of the counts, 16 bytes per thread and access (1.1 ms; the general
// scan, which keeps the counts, a cursor and an offset per bin in three arrays, took 4.7).
constexpr int kFofRound = 4096, kFofTile = 4 * kFofRound;  // counts per round of a block, per block

__device__ __forceinline__ int warp_inclusive(int x) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) >= o) x += y;
  }
  return x;
}
// exclusive scan of one int per thread of a block of 1024 and the total (sums: 33 ints)
__device__ __forceinline__ int block_exclusive(int x, int* sums, int& total) {
  const int incl = warp_inclusive(x), wid = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 31) sums[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const int w = warp_inclusive(sums[threadIdx.x]);
    sums[threadIdx.x] = w;
  }
  __syncthreads();
  total = sums[31];
  return incl - x + (wid > 0 ? sums[wid - 1] : 0);
}

// four counts from i (i a multiple of 4), zeros beyond n
__device__ __forceinline__ int4 load4(const int* p, int i, int n) {
  if (i + 4 <= n) return *reinterpret_cast<const int4*>(p + i);
  int4 v = make_int4(0, 0, 0, 0);
  if (i < n) v.x = p[i];
  if (i + 1 < n) v.y = p[i + 1];
  if (i + 2 < n) v.z = p[i + 2];
  return v;
}

__global__ void __launch_bounds__(1024) k_fof_scan_sums(int n, const int* __restrict__ counts, int* __restrict__ sums) {
  __shared__ int ws[32];
  const int64_t base = (int64_t)blockIdx.x * kFofTile + 4 * threadIdx.x;
  int4 v[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int64_t i = base + r * kFofRound;
    v[r] = i < n ? load4(counts, (int)i, n) : make_int4(0, 0, 0, 0);
  }
  int x = 0;
#pragma unroll
  for (int r = 0; r < 4; ++r) x += v[r].x + v[r].y + v[r].z + v[r].w;
  int total;
  block_exclusive(x, ws, total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// exclusive scan of nb block sums in place, one block
__global__ void __launch_bounds__(1024) k_fof_scan_blocks(int nb, int* __restrict__ sums) {
  __shared__ int ws[32];
  int run = 0;
  for (int b = 0; b < nb; b += 1024) {
    const int i = b + threadIdx.x;
    const int x = i < nb ? sums[i] : 0;
    int total;
    const int e = block_exclusive(x, ws, total);
    if (i < nb) sums[i] = run + e;
    run += total;
    __syncthreads();
  }
}

// counts -> exclusive offsets, and offsets[n] = the number of particles
__global__ void __launch_bounds__(1024) k_fof_scan_apply(int n, int* __restrict__ counts, const int* __restrict__ sums,
                                                         int particles) {
  __shared__ int ws[32];
  const int64_t base = (int64_t)blockIdx.x * kFofTile + 4 * threadIdx.x;
  int4 v[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int64_t i = base + r * kFofRound;
    v[r] = i < n ? load4(counts, (int)i, n) : make_int4(0, 0, 0, 0);
  }
  int run = sums[blockIdx.x];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int64_t i = base + r * kFofRound;
    int total;
    const int e = run + block_exclusive(v[r].x + v[r].y + v[r].z + v[r].w, ws, total);
    const int4 o = make_int4(e, e + v[r].x, e + v[r].x + v[r].y, e + v[r].x + v[r].y + v[r].z);
    if (i + 4 <= n) {
      *reinterpret_cast<int4*>(counts + i) = o;
    } else if (i < n) {
      counts[i] = o.x;
      if (i + 1 < n) counts[i + 1] = o.y;
      if (i + 2 < n) counts[i + 2] = o.z;
    }
    run += total;
    __syncthreads();
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) counts[n] = particles;
}

// records into cell order; every particle starts as its own group
__global__ void __launch_bounds__(256) k_fof_scatter(Geometry g, const float* __restrict__ s,
                                                     const int* __restrict__ keys, const int* __restrict__ ranks,
                                                     const int* __restrict__ offsets, uint4* __restrict__ rec,
                                                     int* __restrict__ parent, int* __restrict__ gsize,
                                                     int* __restrict__ minp) {
  constexpr int U = kPartPerThread;
  const int64_t p0 = x4_first((int64_t)blockIdx.x * blockDim.x * U);
  int at[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t p = p0 + 32 * u;
    at[u] = p < g.np3 ? __ldg(offsets + __ldg(keys + p)) + __ldg(ranks + p) : -1;
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t p = p0 + 32 * u;
    if (at[u] < 0) continue;
    rec[at[u]] = particle_record(g, p, __ldg(s + p), __ldg(s + g.np3 + p), __ldg(s + 2 * g.np3 + p));
    parent[p] = (int)p;  // (positions: any order will do)
    gsize[p] = 0;
    minp[p] = INT_MAX;
  }
}

// Root of x: parents only ever point to smaller positions, so the walk ends within x steps.  It
// halves the path it walks: a position that is not a root never becomes one again, so any of its
// ancestors may replace its parent at any time, whatever other threads write there meanwhile.
__device__ __forceinline__ int fof_find(int* parent, int x) {
  int p = __ldcg(parent + x);
  while (p != x) {
    const int q = __ldcg(parent + p);
    if (q == p) return p;
    __stcg(parent + x, q);
    x = q;
    p = __ldcg(parent + x);
  }
  return x;
}

// the same without writing (k_fof_groups leaves every position's root in parent, which a halved
// path written by another thread must not replace)
__device__ __forceinline__ int fof_find_only(const int* parent, int x) {
  int p = __ldcg(parent + x);
  while (p != x) {
    x = p;
    p = __ldcg(parent + x);
  }
  return x;
}

// link the larger of the two roots under the smaller one; false if the `tries` attempts ran out
__device__ __forceinline__ bool fof_union(int* parent, int a, int b, int tries) {
  for (int it = 0; it < tries; ++it) {
    a = fof_find(parent, a);
    b = fof_find(parent, b);
    if (a == b) return true;
    if (a < b) {
      const int t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(parent + a, a, b) == a) return true;
  }
  return false;
}

// shortest periodic difference of two coordinates in [0, period), period <= 2^31 (in 32 bits: the
// difference itself lies within +-2^31)
__device__ __forceinline__ int min_image(unsigned a, unsigned b, unsigned period) {
  int d = (int)(a - b);
  const int half = (int)(period >> 1);
  if (d > half) d = (int)((unsigned)d - period);
  else if (d < -half) d = (int)((unsigned)d + period);
  return d;
}

// the linking rule den^2 d^2 < lim: in float32 except within 1e-5 of the limit (the float's own
// error is below 1e-6), where it is decided in integers
struct LinkRule {
  int64_t den2, lim;
  float below, above;  // (lim / den2) (1 -+ 1e-5)
  unsigned period;
};
__device__ __forceinline__ bool is_friend(const LinkRule& r, const uint4& a, const uint4& b) {
  const int dx = min_image(b.x, a.x, r.period), dy = min_image(b.y, a.y, r.period), dz = min_image(b.z, a.z, r.period);
  const float fx = (float)dx, fy = (float)dy, fz = (float)dz;
  const float d2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
  if (d2 >= r.above) return false;
  if (d2 <= r.below) return true;
  return r.den2 * ((int64_t)dx * dx + (int64_t)dy * dy + (int64_t)dz * dz) < r.lim;
}

// Sixteen lanes per particle, a lane taking every sixteenth candidate, so a warp's lanes stay busy
// in dense cells (where one thread per particle left most of them waiting for the one in the
// densest cell).  Candidates lie in five runs of sorted positions: run 0, the rest of this cell and
// the next one along x; runs 1-4, the cells x - 1 .. x + 1 of the rows (z, y + 1), (z + 1, y - 1),
// (z + 1, y), (z + 1, y + 1).  Lanes 0-4 look up one run each, so a particle waits for its offsets
// once.  A friend whose parent is this particle's root needs no union: in a dense cell most do
// after the first.  256^3 particles, 40% of them in clumps: 136 ms with one thread per particle,
// 27 cells, 64-bit distances and two walks per friend; 45 with lanes, 7.7 with halved paths as
// well, and with one look-up and shared roots 7.8 (8 lanes), 6.3 (16), 7.2 (32).
constexpr int kLinkLanes = 16;
__global__ void __launch_bounds__(256) k_fof_link(Geometry g, const uint4* __restrict__ rec,
                                                  const int* __restrict__ offsets, int csize, int nc, LinkRule rule,
                                                  int tries, int* __restrict__ parent, int* __restrict__ err) {
  const int64_t n = g.np3;
  const int lane = threadIdx.x % kLinkLanes;
  const unsigned lanes = 0xffffu << (threadIdx.x & 16);  // this particle's lanes of the warp
  const int64_t ngroups = (int64_t)gridDim.x * (blockDim.x / kLinkLanes);
  for (int64_t i = (int64_t)blockIdx.x * (blockDim.x / kLinkLanes) + threadIdx.x / kLinkLanes; i < n; i += ngroups) {
    const uint4 qi = __ldg(rec + i);
    int cx = (int)(qi.x >> g.fbits), cy = (int)(qi.y >> g.fbits), cz = (int)(qi.z >> g.fbits);
    if (csize > 1) {
      cx /= csize;
      cy /= csize;
      cz /= csize;
    }
    int root = fof_find(parent, (int)i);
    bool ok = true;
    auto visit = [&](int j) {
      if (!is_friend(rule, qi, __ldg(rec + j))) return;
      const int pj = __ldcg(parent + j);
      if (pj == root) return;
      const bool joined = fof_union(parent, root, pj, tries);
      ok = ok && joined;
      root = fof_find(parent, root);
      // (only a position that had a parent of its own: a root's word belongs to the unions)
      if (joined && pj != j) __stcg(parent + j, root);
    };
    // first cell of the row of run r
    auto row_of = [&](int r) {
      const int dz = r >= 2 ? 1 : 0, dy = r == 0 ? 0 : r == 1 ? 1 : r - 3;
      const int zz = cz + dz == nc ? 0 : cz + dz;
      int yy = cy + dy;
      yy = yy == nc ? 0 : (yy < 0 ? nc - 1 : yy);
      return (zz * nc + yy) * nc;
    };
    if (cx > 0 && cx < nc - 1) {  // (the same for all lanes of the particle)
      int b = 0, c = 0;
      if (lane < 5) {
        const int* o = offsets + row_of(lane) + cx;
        const int e = __ldg(o + 2);
        b = lane == 0 ? (int)i + 1 : __ldg(o - 1);
        c = e - b;
      }
      // candidate k of the particle is position start + k, start that of the run k falls in
      int start[5], upto[5], total = 0;
#pragma unroll
      for (int r = 0; r < 5; ++r) {
        start[r] = __shfl_sync(lanes, b, r, kLinkLanes) - total;
        total += __shfl_sync(lanes, c, r, kLinkLanes);
        upto[r] = total;
      }
      for (int k0 = 0; k0 < total; k0 += kLinkLanes) {
        const int k = k0 + lane;
        if (k0) root = __reduce_min_sync(lanes, root);  // the lanes share what they have walked to
        if (k >= total) continue;
        const int s = k < upto[0] ? start[0] : k < upto[1] ? start[1] : k < upto[2] ? start[2] : k < upto[3] ? start[3] : start[4];
        visit(s + k);
      }
    } else {  // at the faces of the box along x the cells of a run are apart: one at a time
      for (int r = 0; r < 5; ++r) {
        const int row = row_of(r);
        for (int dx = r == 0 ? 0 : -1; dx <= 1; ++dx) {
          const int xx = cx + dx < 0 ? nc - 1 : (cx + dx == nc ? 0 : cx + dx);
          const int b = r == 0 && dx == 0 ? (int)i + 1 : __ldg(offsets + row + xx);
          const int e = __ldg(offsets + row + xx + 1);
          for (int j = b + lane; j < e; j += kLinkLanes) visit(j);
        }
      }
    }
    if (!ok) atomicOr(err, kErrUnion);
    __syncwarp(lanes);
  }
}

// roots, group sizes and labels; the lanes of a warp that share a root (neighbours in cell order
// mostly do) add their particles with one pair of atomics
__global__ void __launch_bounds__(256) k_fof_groups(int64_t n, const uint4* __restrict__ rec, int* __restrict__ parent,
                                                    int* __restrict__ gsize, int* __restrict__ minp) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int r = -1;
  unsigned p = 0;
  if (i < n) {
    r = fof_find_only(parent, (int)i);
    parent[i] = r;
    p = rec[i].w;
  }
  const unsigned peers = __match_any_sync(0xffffffffu, r);
  const unsigned least = __reduce_min_sync(peers, p);
  if (i < n && (int)(threadIdx.x & 31) == __ffs(peers) - 1) {
    atomicAdd(gsize + r, __popc(peers));
    atomicMin(minp + r, (int)least);
  }
}

__global__ void k_fof_output(int64_t n, const uint4* __restrict__ rec, const int* __restrict__ parent,
                             const int* __restrict__ gsize, const int* __restrict__ minp, int nmin, Thresholds thr,
                             int* __restrict__ group, int* __restrict__ size, unsigned long long* __restrict__ n_ge) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int r = parent[i];
    const int gs = gsize[r];
    const unsigned p = rec[i].w;
    if (size) size[p] = gs;
    if (group) group[p] = gs >= nmin ? minp[r] : -1;
    if (r == (int)i && gs >= nmin)
      for (int k = 0; k < thr.n; ++k)
        if (gs >= thr.v[k]) atomicAdd(n_ge + k, 1ULL);
  }
}

unsigned grid_of(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 64); }

}  // namespace
}  // namespace cola

using namespace cola;

extern "C" int cola_fof(cola_plan* plan, const float* s, int32_t b_num, int32_t b_den, int32_t nmin, int32_t* group,
                        int32_t* size, int32_t nthr, const int32_t* thresholds, int64_t* n_ge, cola_stream stream) {
  if (!plan) return fail(COLA_EINVAL, "null plan");
  if (!plan->ws_base) return fail(COLA_ENOWORKSPACE, "cola_set_workspace has not been called");
  ProfilerGuard pg(&plan->prof);
  if (!s || (!group && !size)) return fail(COLA_EINVAL, "null array");
  if (b_num < 1 || b_den < 1 || b_den > 50 || b_num > b_den)
    return fail(COLA_EINVAL, "linking length b = b_num / b_den needs 1 <= b_num <= b_den <= 50");
  if (nmin < 1) return fail(COLA_EINVAL, "nmin must be >= 1");
  if (nthr < 0 || nthr > kMaxThresholds || (nthr > 0 && (!thresholds || !n_ge)))
    return fail(COLA_EINVAL, "0..32 thresholds with host thresholds and a device n_ge array");
  const Geometry& g = plan->geo;
  if (g.ratio < 1) return fail(COLA_EUNSUPPORTED, "FOF needs ng to be a multiple of np");
  if (g.np3 >= 0x7fffffffLL) return fail(COLA_EUNSUPPORTED, "FOF supports fewer than 2^31 particles");
  // cells of csize mesh cells: at least the linking length b * (ng/np), a divisor of ng, and few
  // enough cells for int32 bin offsets
  int csize = (b_num * g.ratio + b_den - 1) / b_den;
  while (csize <= g.ng && (g.ng % csize != 0 || (int64_t)(g.ng / csize) * (g.ng / csize) * (g.ng / csize) >= (1LL << 30)))
    ++csize;
  const int nc = csize <= g.ng ? g.ng / csize : 0;
  if (nc < 3) return fail(COLA_EUNSUPPORTED, "FOF needs at least 3 linking cells per side");
  // exact int64 tests: den^2 d^2 with |d| < 2 csize 2^F per axis, and num^2 s^2
  if (((int64_t)csize << g.fbits) >= (1LL << 24) || (((int64_t)g.ratio << g.fbits) >= (1LL << 24)))
    return fail(COLA_EUNSUPPORTED, "FOF: linking cells or mean separation too large for exact int64 distances");
  Thresholds thr{};
  thr.n = nthr;
  for (int k = 0; k < nthr; ++k) thr.v[k] = thresholds[k];
  cudaStream_t st = (cudaStream_t)stream;
  Workspace& w = plan->ws;
  // scratch: the cells' counts (then offsets), the ranks and the scan's block sums in the
  // force-mesh region (3 ng^3 words for at most ng^3 + 1, np^3 and ng^3 / 16384 + 1 of them; ng >= np
  // as ng is a multiple of np), the union-find arrays in the half spectra
  const int ncells = nc * nc * nc;
  int* offsets = reinterpret_cast<int*>(w.freal);
  int* ranks = offsets + ((int64_t)ncells + 64) / 64 * 64;
  int* sums = ranks + g.np3;
  int* parent = reinterpret_cast<int*>(w.meshA);
  int* gsize = reinterpret_cast<int*>(w.meshG[1]);
  int* minp = reinterpret_cast<int*>(w.meshG[2]);
  const int64_t n = g.np3;
  const unsigned per_block4 = 256 * kPartPerThread, nb4 = (unsigned)((n + per_block4 - 1) / per_block4);
  COLA_CUDA_CHECK(cudaMemsetAsync(offsets, 0, sizeof(int) * ncells, st));
  if (nthr > 0) COLA_CUDA_CHECK(cudaMemsetAsync(n_ge, 0, sizeof(int64_t) * nthr, st));
  {
    LaunchScope ls_("fof_keys", st);
    k_fof_keys<<<nb4, 256, 0, st>>>(g, s, csize, nc, w.keys, ranks, offsets, w.err);
  }
  COLA_LAUNCH_CHECK();
  const int nsums = (ncells + kFofTile - 1) / kFofTile;
  {
    LaunchScope ls_("fof_scan_sums", st);
    k_fof_scan_sums<<<nsums, 1024, 0, st>>>(ncells, offsets, sums);
  }
  COLA_LAUNCH_CHECK();
  {
    LaunchScope ls_("fof_scan_blocks", st);
    k_fof_scan_blocks<<<1, 1024, 0, st>>>(nsums, sums);
  }
  COLA_LAUNCH_CHECK();
  {
    LaunchScope ls_("fof_scan_apply", st);
    k_fof_scan_apply<<<nsums, 1024, 0, st>>>(ncells, offsets, sums, (int)n);
  }
  COLA_LAUNCH_CHECK();
  {
    LaunchScope ls_("fof_scatter", st);
    k_fof_scatter<<<nb4, 256, 0, st>>>(g, s, w.keys, ranks, offsets, w.rec, parent, gsize, minp);
  }
  COLA_LAUNCH_CHECK();
  const int64_t sfix = (int64_t)g.ratio << g.fbits;
  LinkRule rule;
  rule.den2 = (int64_t)b_den * b_den;
  rule.lim = (int64_t)b_num * b_num * sfix * sfix;
  const double limit = (double)rule.lim / (double)rule.den2;
  rule.below = (float)(limit * (1.0 - 1e-5));
  rule.above = (float)(limit * (1.0 + 1e-5));
  rule.period = (unsigned)g.ng << g.fbits;
  {
    LaunchScope ls_("fof_link", st);
    k_fof_link<<<grid_of(n * kLinkLanes), 256, 0, st>>>(g, w.rec, offsets, csize, nc, rule, plan->fof_union_tries,
                                                        parent, w.err);
  }
  COLA_LAUNCH_CHECK();
  {
    LaunchScope ls_("fof_groups", st);
    k_fof_groups<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, w.rec, parent, gsize, minp);
  }
  COLA_LAUNCH_CHECK();
  {
    LaunchScope ls_("fof_output", st);
    k_fof_output<<<grid_of(n), 256, 0, st>>>(n, w.rec, parent, gsize, minp, nmin, thr, group, size,
                                             reinterpret_cast<unsigned long long*>(n_ge));
  }
  COLA_LAUNCH_CHECK();
  return COLA_OK;
}

extern "C" int cola_set_fof_union_tries(cola_plan* plan, int32_t tries) {
  if (!plan) return fail(COLA_EINVAL, "null plan");
  if (tries < 0 || tries > (1 << 30)) return fail(COLA_EINVAL, "tries must be in [0, 2^30]");
  plan->fof_union_tries = tries;
  return COLA_OK;
}
