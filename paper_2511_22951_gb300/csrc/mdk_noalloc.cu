// mdk_noalloc.cu -- mdk_lj_compute_noalloc: LJ energy and forces with no
// device allocation and no workspace (declared in include/mdk.h).
//
// Some callers cannot allocate device memory: their device memory belongs to
// another allocator (a framework's caching pool, an arena reserved at
// start-up), or their host loop cannot afford an allocation and the device
// synchronisation that freeing implies.  For them this variant of the force
// kernel keeps its scratch -- cell histogram, cell starts, atoms and wrapped
// positions sorted by cell, partial energies -- in one fixed-size file-scope
// __device__ array instead of a caller-supplied workspace, and walks the
// 27-cell stencil directly (no Verlet list, pairs with r < rc).
//
// Two launches: k_na_cells sorts the atoms into cells (one cluster of 8
// blocks, its phases separated by cluster barriers), k_na_force takes a warp
// per slice of at most 4 atoms of a cell.  4000 argon atoms: 1056 -> 63 us a
// call (256: 961 -> 39, 32,000: 1078 -> 224); the version before took seven
// launches and gave each atom one thread that tested all ~500 candidates in
// FP64 (4000 atoms: 16 blocks of 256 threads, 1028 us).
//
// The array lives in every GPU that loads the library until the process
// exits.  Host code cannot use its name as a device address (there it is a
// host-side shadow), so the first call on each device looks its address up
// with cudaGetSymbolAddress while that device is current, and passes the
// pointer to the kernels.  Every call shares the array: each call zeroes the
// histogram it accumulates into, and calls whose work overlaps on a GPU race.
//
// An atom with a non-finite coordinate goes to a bucket past the real cells:
// no pair includes it, and its force row and the energy come out NaN (the
// call does not synchronise, so the results are its only status channel).
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>
#include <mutex>

#include "mdk.h"
#include "lj_pair.cuh"

namespace mdk {
namespace {

constexpr int kMaxAtoms = MDK_NOALLOC_MAX_ATOMS;
constexpr int kMaxCells = MDK_NOALLOC_MAX_CELLS;
constexpr int kMaxDevices = 64;
constexpr int kCta = 8;          // blocks of the sorting cluster
constexpr int kCtaThreads = 1024;
constexpr int kSlice = 4;        // atoms of one warp at most
constexpr int kFWarps = 4;       // warps per block of the force kernel
constexpr int kList = 192;       // entries per atom between two evaluations

// scratch layout (bytes), every part 256-byte aligned; the cell arrays hold
// n_cells + 1 buckets (the last one for atoms with a non-finite coordinate)
constexpr size_t kBuckets = (size_t)kMaxCells + 64;
constexpr size_t kOffCount = 0;
constexpr size_t kOffStart = kOffCount + 4 * kBuckets;
constexpr size_t kOffOrder = kOffStart + 4 * kBuckets;
constexpr size_t kOffAtom = kOffOrder + 4 * (size_t)kMaxAtoms;
constexpr size_t kOffCell = kOffAtom + 4 * (size_t)kMaxAtoms;
constexpr size_t kOffX = kOffCell + 4 * (size_t)kMaxAtoms;
constexpr size_t kOffP = kOffX + 24 * (size_t)kMaxAtoms;
constexpr size_t kOffE = kOffP + 16 * (size_t)kMaxAtoms;
constexpr size_t kMaxBlocks = kMaxAtoms / (kSlice * kFWarps);  // of the force kernel
constexpr size_t kOffMisc = kOffE + 8 * kMaxBlocks;
constexpr size_t kScratchBytes = kOffMisc + 256;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

struct NaScratch {
  int *count, *start, *order;
  int *atom, *cell;  // by place in the cell order: caller's index, cell
  double *x;         // wrapped positions in cell order [3][kMaxAtoms]
  float4 *p;         // offsets from the cell centre (NaN beyond 2 cells)
  double *e;         // energy of each block of the force kernel
  int *part;         // bucket totals of the sorting blocks
  unsigned *done;    // force blocks that have finished
};

struct NaParams {
  int N;
  int nc[3], per[3];
  int n_cells;
  double lo[3], hi[3], L[3], inv_h[3], h[3];
  float hi_f;  // FP32 pre-filter: candidates with a larger r^2 are outside rc
  pair::LJc<double> lj;
};

__host__ __device__ inline NaScratch carve(unsigned char *base) {
  NaScratch s;
  s.count = reinterpret_cast<int *>(base + kOffCount);
  s.start = reinterpret_cast<int *>(base + kOffStart);
  s.order = reinterpret_cast<int *>(base + kOffOrder);
  s.atom = reinterpret_cast<int *>(base + kOffAtom);
  s.cell = reinterpret_cast<int *>(base + kOffCell);
  s.x = reinterpret_cast<double *>(base + kOffX);
  s.p = reinterpret_cast<float4 *>(base + kOffP);
  s.e = reinterpret_cast<double *>(base + kOffE);
  s.part = reinterpret_cast<int *>(base + kOffMisc);
  s.done = reinterpret_cast<unsigned *>(base + kOffMisc + 128);
  return s;
}

// a coordinate wrapped by whole box lengths, as in the list build
__device__ __forceinline__ double na_wrap(const NaParams &p, int d, double v) {
  if (p.per[d] && (v >= p.hi[d] || v < p.lo[d])) {
    if (fabs(v - p.lo[d]) > 4.0 * p.L[d]) v = v - p.L[d] * floor((v - p.lo[d]) / p.L[d]);
    for (int it = 0; it < 8 && v >= p.hi[d]; ++it) v = v - p.L[d];
    for (int it = 0; it < 8 && v < p.lo[d]; ++it) v = v + p.L[d];
    if (v >= p.hi[d] || v < p.lo[d]) v = p.lo[d];
  }
  return v;
}

// block-wide exclusive scan of one value per thread (kCtaThreads threads)
__device__ __forceinline__ int na_exscan(int v, int *total) {
  __shared__ int warp_tot[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_tot[w] = incl;
  __syncthreads();
  if (w == 0) {
    const int v0 = warp_tot[lane];
    int vi = v0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, vi, o);
      if (lane >= o) vi += t;
    }
    warp_tot[lane] = vi - v0;
    if (lane == 31) *total = vi;
  }
  __syncthreads();
  return warp_tot[w] + incl - v;
}

// cell coordinate along d of a wrapped coordinate
__device__ __forceinline__ int na_coord(const NaParams &p, double v, int d) {
  return min(max((int)floor((v - p.lo[d]) * p.inv_h[d]), 0), p.nc[d] - 1);
}
// atom i's wrapped position and cell (n_cells for a non-finite coordinate)
__device__ __forceinline__ int na_cell(const NaParams &p, const double *x, int i, double (&v)[3]) {
  bool fin = true;
  for (int d = 0; d < 3; ++d) {
    v[d] = x[3 * (size_t)i + d];
    fin = fin && isfinite(v[d]);
  }
  if (!fin) return p.n_cells;
  int c[3];
  for (int d = 0; d < 3; ++d) {
    v[d] = na_wrap(p, d, v[d]);
    c[d] = na_coord(p, v[d], d);
  }
  return c[0] + p.nc[0] * (c[1] + p.nc[1] * c[2]);
}
// Atoms into cells: histogram, scan, scatter, order inside each cell by index
// (so results do not depend on the order of the atomics).  A non-finite
// coordinate sends the atom to bucket n_cells.  At these sizes the phases are
// latencies, not throughput, so they share one launch: a cluster of 8 blocks
// (scheduled together by the hardware) with a cluster barrier between phases;
// a thread keeps its atoms' wrapped positions, cells and slots in registers.
// 4000 atoms: 19 us.  One block with everything in shared memory took 71:
// the ~35 FP64 operations of an atom are more than one SM's FP64 pipe (2 lanes
// a clock) can do in that time.
constexpr int kPer = kMaxAtoms / (kCta * kCtaThreads);
__global__ void __cluster_dims__(kCta, 1, 1) __launch_bounds__(kCtaThreads, 1)
    k_na_cells(NaParams p, const double *x, unsigned char *base) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const NaScratch s = carve(base);
  const int t = blockIdx.x * kCtaThreads + threadIdx.x;
  constexpr int nt = kCta * kCtaThreads;
  const int nb = p.n_cells + 1;
  for (int c = t; c < nb; c += nt) s.count[c] = 0;
  if (t == 0) *s.done = 0u;
  cluster.sync();
  double v[kPer][3];
  int cell[kPer], slot[kPer];
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int i = t + q * nt;
    if (i < p.N) {
      cell[q] = na_cell(p, x, i, v[q]);
      slot[q] = atomicAdd(&s.count[cell[q]], 1);
    }
  }
  cluster.sync();
  // scan: every block takes one run of buckets, then adds the blocks before it
  const int seg = (nb + kCta - 1) / kCta, per = (seg + kCtaThreads - 1) / kCtaThreads;
  const int c0 = blockIdx.x * seg + threadIdx.x * per;
  const int c1 = min(min(c0 + per, (int)(blockIdx.x + 1) * seg), nb);
  int sum = 0;
  for (int c = c0; c < c1; ++c) sum += s.count[c];
  __shared__ int tot;
  int pre = na_exscan(sum, &tot);
  if (threadIdx.x == 0) s.part[blockIdx.x] = tot;
  cluster.sync();
  for (int b = 0; b < (int)blockIdx.x; ++b) pre += s.part[b];
  for (int c = c0; c < c1; ++c) {
    s.start[c] = pre;
    pre += s.count[c];
  }
  if (t == 0) s.start[nb] = p.N;
  cluster.sync();
#pragma unroll
  for (int q = 0; q < kPer; ++q)
    if (t + q * nt < p.N) s.order[s.start[cell[q]] + slot[q]] = t + q * nt;
  cluster.sync();
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int i = t + q * nt;
    if (i >= p.N) continue;
    const int a = s.start[cell[q]], e = s.start[cell[q] + 1];
    int at = a;
    for (int k = a; k < e; ++k) at += s.order[k] < i ? 1 : 0;
    s.atom[at] = i;
    s.cell[at] = cell[q];
    if (cell[q] == p.n_cells) continue;
    const int c[3] = {cell[q] % p.nc[0], (cell[q] / p.nc[0]) % p.nc[1],
                      cell[q] / (p.nc[0] * p.nc[1])};
    float f[3];
    bool far = false;
    for (int d = 0; d < 3; ++d) {
      s.x[(size_t)d * kMaxAtoms + at] = v[q][d];
      const double o = v[q][d] - (p.lo[d] + ((double)c[d] + 0.5) * p.h[d]);
      f[d] = (float)o;
      far = far || !(fabsf(f[d]) <= 2.0f * (float)p.h[d]);
    }
    s.p[at] = make_float4(far ? __int_as_float(0x7fc00000) : f[0], f[1], f[2], 0.f);
  }
}

struct NaWarp {
  uint32_t list[kSlice][kList];  // candidate (place in the cell order) | template cell << 16
  float4 sh[27];                 // template cell: shift s h
  int img[27];                   // its periodic image: 2-bit codes n + 1 per dimension
  int end[28], off[28];          // flattened candidates: end, place = candidate + off
  int cnt[kSlice];
};

// The force kernel's variant: 27-cell stencil, each stencil position one
// periodic image, d = x_j - (x_i - n L), pairs with r^2 < rc^2, FP64; decided on
// (x_j - x_i) + n L, whose mirror image is exact, within 2^-20 of rc^2 (see
// Vec<Fp64>::inside).
// One warp per slice of a cell's atoms.  Lanes hold candidates (the 27 cells
// flattened) and an FP32 test on cell-centre offsets drops those clearly
// outside rc (~85%): GB300's FP64 pipe (2 lanes per clock and SM) is what
// binds here, so only pairs inside rc and its 1e-4 margin reach it.  Those
// collect in per-atom lists in shared memory, which 32 / n lanes per atom
// then evaluate side by side (32 lanes busy instead of the ~5 that a
// candidate-per-lane evaluation would keep busy).
template <int SHIFT>
__global__ void __launch_bounds__(32 * kFWarps) k_na_force(NaParams p, unsigned char *base,
                                                          double *F, double *E) {
  using namespace pair;
  __shared__ NaWarp sm_[kFWarps];
  __shared__ double e_warp[kFWarps];
  __shared__ bool last;
  const NaScratch s = carve(base);
  NaWarp &sm = sm_[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned full = 0xffffffffu, lower = (1u << lane) - 1u;
  const int tile = kSlice * (blockIdx.x * kFWarps + (threadIdx.x >> 5));
  // slices that start in this warp's kSlice places (equal parts of a cell)
  int n_sl = 0;
  bool lead = false;
  double e_sum = 0.0;
  if (lane < kSlice && tile + lane < p.N) {
    const int cell = s.cell[tile + lane];
    if (cell == p.n_cells) {  // non-finite input: in no pair, NaN results
      const size_t i = (size_t)s.atom[tile + lane];
      F[3 * i] = F[3 * i + 1] = F[3 * i + 2] = NAN;
      e_sum = NAN;
    } else {
      const int a = s.start[cell], n = s.start[cell + 1] - a;
      const int parts = (n + kSlice - 1) / kSlice, sz = (n + parts - 1) / parts;
      const int k = tile + lane - a;
      lead = k % sz == 0;
      n_sl = min(sz, n - k);
    }
  }
  for (unsigned leads = __ballot_sync(full, lead); leads; leads &= leads - 1) {
    const int l0 = __ffs(leads) - 1;
    const int a0 = tile + l0, n = __shfl_sync(full, n_sl, l0);
    const int cell = s.cell[a0];
    const int c0 = cell % p.nc[0], c1 = (cell / p.nc[0]) % p.nc[1],
              c2 = cell / (p.nc[0] * p.nc[1]);
    int len = 0, first = 0;
    if (lane < 27) {
      const int sd[3] = {lane % 3 - 1, (lane / 3) % 3 - 1, lane / 9 - 1};
      int c[3] = {c0 + sd[0], c1 + sd[1], c2 + sd[2]};
      bool in = true;
      int code = 0;
      for (int d = 0; d < 3; ++d) {
        int img = 0;
        if (p.per[d]) {
          img = c[d] < 0 ? -1 : (c[d] >= p.nc[d] ? 1 : 0);
          c[d] -= img * p.nc[d];
        } else {
          in = in && c[d] >= 0 && c[d] < p.nc[d];
        }
        code |= (img + 1) << (2 * d);
      }
      sm.img[lane] = code;
      if (in) {
        const int cj = c[0] + p.nc[0] * (c[1] + p.nc[1] * c[2]);
        first = s.start[cj];
        len = s.start[cj + 1] - first;
      }
      sm.sh[lane] = make_float4((float)(sd[0] * p.h[0]), (float)(sd[1] * p.h[1]),
                                (float)(sd[2] * p.h[2]), 0.f);
    }
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(full, incl, o);
      if (lane >= o) incl += t;
    }
    const int total = __shfl_sync(full, incl, 31);
    if (lane < 28) {
      sm.end[lane] = incl;  // lane 27: the total
      sm.off[lane] = first - (incl - len);
    }
    float4 pa[kSlice];
#pragma unroll
    for (int k = 0; k < kSlice; ++k) pa[k] = s.p[a0 + min(k, n - 1)];
    // this lane's atom and its share of that atom's entries
    const int T = 32 / n, ka = lane / T, la = lane % T;
    const bool on = ka < n;
    Shift3 gx, gy, gz;  // x_i - n L
    if (on) {
      gx = Shift3(s.x[a0 + ka], p.L[0]);
      gy = Shift3(s.x[kMaxAtoms + a0 + ka], p.L[1]);
      gz = Shift3(s.x[2 * kMaxAtoms + a0 + ka], p.L[2]);
    }
    double fx = 0, fy = 0, fz = 0, e = 0;
    int cnt[kSlice];
#pragma unroll
    for (int k = 0; k < kSlice; ++k) cnt[k] = 0;
    __syncwarp();
    int t = 0;
    uint32_t next_ent = 0;
    float4 next_p = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](int q) {  // candidate q, a chunk ahead of its tests
      if (q >= total) return;
      while (q >= sm.end[t]) ++t;
      const int j = q + sm.off[t];
      next_p = s.p[j];
      next_ent = (uint32_t)j | ((uint32_t)t << 16);
    };
    fetch(lane);
    for (int c = 0; c < total; c += 32) {
      const int q = c + lane;
      const uint32_t ent = next_ent;
      const float4 d = sm.sh[ent >> 16];
      const float4 v = make_float4(next_p.x + d.x, next_p.y + d.y, next_p.z + d.z, 0.f);
      fetch(q + 32);
      int most = 0;
#pragma unroll
      for (int k = 0; k < kSlice; ++k) {
        if (k >= n) break;
        const float dx = v.x - pa[k].x, dy = v.y - pa[k].y, dz = v.z - pa[k].z;
        const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
        // NaN (far atoms) passes; the atom itself is template cell 13
        const bool ok = q < total && !(r2 > p.hi_f) && ent != ((uint32_t)(a0 + k) | (13u << 16));
        const unsigned b = __ballot_sync(full, ok);
        if (ok) sm.list[k][cnt[k] + __popc(b & lower)] = ent;
        cnt[k] += __popc(b);
        most = max(most, cnt[k]);
      }
      if (most <= kList - 32 && c + 32 < total) continue;
      // evaluate what the lists hold
      if (lane == 0)
#pragma unroll
        for (int k = 0; k < kSlice; ++k) sm.cnt[k] = cnt[k];
      __syncwarp();
      const int m = on ? sm.cnt[ka] : 0;
#pragma unroll 2
      for (int w = la; w < m; w += T) {
        const uint32_t en = sm.list[ka][w];
        const int j = (int)(en & 0xffffu), tc = (int)(en >> 16);
        const int im = sm.img[tc];
        const double dx = s.x[j] - gx.at(im);
        const double dy = s.x[kMaxAtoms + j] - gy.at(im >> 2);
        const double dz = s.x[2 * kMaxAtoms + j] - gz.at(im >> 4);
        const double r2 = r2_of(dx, dy, dz);
        bool in = below(r2, p.lj.rc2);
        if ((unsigned)(__double2hiint(r2) - __double2hiint(p.lj.rc2) + 1) <= 2u) {
          const double ex = __fma_rn((double)nbr_s(im, 0), p.L[0], __dsub_rn(s.x[j], gx.b));
          const double ey =
              __fma_rn((double)nbr_s(im, 1), p.L[1], __dsub_rn(s.x[kMaxAtoms + j], gy.b));
          const double ez =
              __fma_rn((double)nbr_s(im, 2), p.L[2], __dsub_rn(s.x[2 * kMaxAtoms + j], gz.b));
          in = r2_of(ex, ey, ez) < p.lj.rc2;
        }
        double fr, u;
        lj_pair<G<Fp64>, SHIFT, true>(p.lj, r2, fr, u);
        fr = in ? fr : 0.0;
        fx += fr * dx;
        fy += fr * dy;
        fz += fr * dz;
        e += in ? 0.5 * u : 0.0;
      }
#pragma unroll
      for (int k = 0; k < kSlice; ++k) cnt[k] = 0;
      __syncwarp();
    }
    // the T lanes of an atom, in a fixed order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double gx = __shfl_down_sync(full, fx, o), gy = __shfl_down_sync(full, fy, o),
                   gz = __shfl_down_sync(full, fz, o), ge = __shfl_down_sync(full, e, o);
      if (la < o && la + o < T) {
        fx += gx;
        fy += gy;
        fz += gz;
        e += ge;
      }
    }
    if (on && la == 0) {
      const size_t i = (size_t)s.atom[a0 + ka];
      F[3 * i] = fx;
      F[3 * i + 1] = fy;
      F[3 * i + 2] = fz;
      e_sum += e;
    }
    __syncwarp();
  }
  // energies: lanes, warps, blocks in a fixed order; the last block adds up
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e_sum += __shfl_xor_sync(full, e_sum, o);
  if (lane == 0) e_warp[threadIdx.x >> 5] = e_sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kFWarps; ++w) t += e_warp[w];
    s.e[blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(s.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last || threadIdx.x >= 32) return;
  __threadfence();
  double t = 0.0;
  for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(s.e + b);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(full, t, o);
  if (lane == 0) E[0] = t;
}

std::mutex g_mu;
unsigned char *g_addr[kMaxDevices] = {};

// device address of the scratch array on the current device (looked up once)
int scratch_address(unsigned char **out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MDK_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_addr[dev]) {
    void *ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return MDK_ERR_CUDA;
    g_addr[dev] = static_cast<unsigned char *>(ptr);
  }
  *out = g_addr[dev];
  return MDK_OK;
}

}  // namespace
}  // namespace mdk

using namespace mdk;

extern "C" int mdk_lj_compute_noalloc(const double *x, int64_t N, const double box_lo[3],
                                      const double box_hi[3], const int periodic[3], double eps,
                                      double sigma, double rc, int shift_mode, double *F,
                                      double *E, void *cuda_stream) {
  if (N < 0 || !box_lo || !box_hi || !periodic || !E || (N > 0 && (!x || !F)))
    return MDK_ERR_BAD_ARG;
  if (!(eps > 0.0) || !(sigma > 0.0) || !(rc > 0.0) || shift_mode < 0 || shift_mode > 2)
    return MDK_ERR_BAD_ARG;
  if (N > kMaxAtoms) return MDK_ERR_TOO_LARGE;
  NaParams p{};
  p.N = (int)N;
  long long cells = 1;
  for (int d = 0; d < 3; ++d) {
    const double L = box_hi[d] - box_lo[d];
    if (!(L > 0.0)) return MDK_ERR_BAD_ARG;
    if (periodic[d] && L < rc) return MDK_ERR_BOX_TOO_SMALL;
    int nc = (int)floor(L / (rc * (1.0 + 1e-10)));
    if (nc < 1) nc = 1;
    if (nc > kMaxCells) return MDK_ERR_TOO_LARGE;
    p.nc[d] = nc;
    p.per[d] = periodic[d] ? 1 : 0;
    p.lo[d] = box_lo[d];
    p.hi[d] = box_hi[d];
    p.L[d] = L;
    p.h[d] = L / nc;
    p.inv_h[d] = 1.0 / p.h[d];
    cells *= nc;
  }
  if (cells > kMaxCells) return MDK_ERR_TOO_LARGE;
  p.n_cells = (int)cells;
  LJParams q{};
  lj_fill(q, eps, sigma, rc, shift_mode);
  p.lj = pair::LJc<double>(q);
  // the FP32 r^2 of offsets up to 2 h per dimension is off by less than 2.5e-5 h^2
  const double hm = fmax(p.h[0], fmax(p.h[1], p.h[2]));
  p.hi_f = (float)(p.lj.rc2 + 1e-4 * hm * hm);
  unsigned char *base = nullptr;
  int r = scratch_address(&base);
  if (r) return r;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  k_na_cells<<<kCta, kCtaThreads, 0, st>>>(p, x, base);
  const int grid = (int)std::max<int64_t>(1, (N + kSlice * kFWarps - 1) / (kSlice * kFWarps));
  if (shift_mode == 2)
    k_na_force<2><<<grid, 32 * kFWarps, 0, st>>>(p, base, F, E);
  else
    k_na_force<1><<<grid, 32 * kFWarps, 0, st>>>(p, base, F, E);
  return cudaPeekAtLastError() == cudaSuccess ? MDK_OK : MDK_ERR_CUDA;
}
