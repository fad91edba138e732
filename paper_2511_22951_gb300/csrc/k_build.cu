// k_build.cu -- Verlet-list rebuild on the GPU (Sec. "Neighbor lists
// construction" of the paper: a virtual Cartesian grid of cells of size
// >= R = r_ns, one bucket-sort pass of the atoms into the cells, then a
// 3x3x3 cell stencil search; Eq. rhrz gives r_ns = (1 + beta) r_cut, here
// rc + skin).
//
// The chain runs every step and every kernel returns at once unless the
// device flag st->rebuild is set, so the whole step stays on the device
// (no host round trip to decide whether to rebuild):
//   k_pre       count steps since the last build; fixed-interval trigger
//   k_bin       wrap periodic coordinates, cell id per atom, cell histogram
//   k_scan_*    exclusive scan of the histogram (3 phases; one at small sizes)
//   k_scatter   counting-sort scatter into cell order (atomic slots)
//   k_cell_sort order each cell's atoms by their permanent id (determinism)
//   k_permute   gather every per-atom array into the new order (scratch)
//   k_copyback  scratch -> primary arrays
//   k_build     Verlet lists (full, or half: each pair once): FP32
//               pre-filter on cell-relative offsets,
//               exact FP64 test for the few candidates near r_ns
//   k_finish    clear the flag, count the build
#include <math.h>

#include <algorithm>

#include <climits>

#include "mdk_internal.cuh"

namespace mdk {

namespace {

constexpr int kBlk = 256;
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ bool flag_on(const Sys &s) {
  return *(volatile int *)&s.st->rebuild != 0;
}
// a full build: re-bin, re-sort and rebuild the (outer) list from the cells;
// with the outer list off every build is full
__device__ __forceinline__ bool full_on(const Sys &s) {
  return flag_on(s) && *(volatile int *)&s.st->full != 0;
}

// Window and build kind of the build that st->rebuild asks for (one thread).
__device__ __forceinline__ void plan_build(const Sys &s, int count_step) {
  DevStatus *st = s.st;
  st->step_build = count_step;
  st->build_ovf = 0;
  if (s.rebuild_every > 0 && st->since_build >= s.rebuild_every) st->rebuild = 1;
  // the window acts at builds that stepping triggers, not at explicit builds
  st->win_active = (s.win_on && count_step && st->rebuild) ? 1 : 0;
  // explicit builds, window builds, list-free forces and a missing outer
  // list take a full build; otherwise k_outer_decide checks the budget
  st->full = (st->rebuild && (!s.outer_on || !count_step || st->win_active ||
                              !st->outer_valid || s.half == 2))
                 ? 1
                 : 0;
  st->win_cut = -INFINITY;
  if (st->win_active) {
    st->key_xmax = dkey(-INFINITY);
    st->key_xmin = dkey(INFINITY);
    st->win_insert = 0;
  }
}

__global__ void k_pre(Sys s, int count_step, int use_cond, cudaGraphConditionalHandle h) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  DevStatus *st = s.st;
  if (st->abort) {  // stepping stopped at an overflowing build: nothing more
    if (use_cond) cudaGraphSetConditional(h, 0u);
    return;
  }
  if (count_step) {
    st->since_build += 1;
    st->n_steps += 1;  // index of the force evaluation that follows (Langevin noise)
  }
  plan_build(s, count_step);
  if (use_cond) cudaGraphSetConditional(h, st->rebuild ? 1u : 0u);
}

// The end of a captured loop body of `places` steps.  The steps up to the first
// that triggered a build (or to the end of the body, of the loop or of the
// fixed interval) are done, the places after it did nothing (run_n).  The
// check and the conditional nodes cost once per body instead of once per step:
// a step without a build 19.4 -> 11.3 us on 256 FP64 LJ atoms (its force pass
// alone: 11.1), 21.2 -> 14.4 us on 32,000 mixed.  The next body reads the copy
// that this one started from: after an odd e it is written again (by the
// build, or by k_regather).
__global__ void k_loop_head(Sys s, int places, int kernels, cudaGraphConditionalHandle h,
                            cudaGraphConditionalHandle loop) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  DevStatus *st = s.st;
  st->n_graph_kernels += kernels;
  const unsigned trig = st->trig;
  st->trig = 0u;
  if (st->abort) {
    st->left = 0;
    cudaGraphSetConditional(h, 0u);
    cudaGraphSetConditional(loop, 0u);
    return;
  }
  int e = min(places, st->left);
  if (s.rebuild_every > 0) e = min(e, max(1, s.rebuild_every - st->since_build));
  const unsigned m = trig & ((1u << e) - 1u);
  if (m) {
    e = __ffs(m);
    st->rebuild = 1;
  }
  st->left -= e;
  st->since_build += e;
  st->n_steps += e;  // index of the force evaluation that follows
  st->regather = e & 1;
  plan_build(s, 1);
  cudaGraphSetConditional(h, st->rebuild || st->regather ? 1u : 0u);
  cudaGraphSetConditional(loop, st->left > 0 ? 1u : 0u);
}

__global__ void k_set_left(Sys s, int left) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  s.st->left = left;
  s.st->trig = 0u;
}

// ---- moving window (Sec. "Moving window simulation"; rules in mdk.h) ----
// Front: bins of width front_bin along x; a bin is shocked when its mean v_x
// exceeds u_p / 2, decided exactly on velocities rounded to multiples of
// 2^-40 Angstrom/fs (integer sums, so the order of the atomics is irrelevant).
// Leading edge = max x.
constexpr double kTwo40 = 1099511627776.0;
constexpr int kFbinSmem = 2048;  // bins privatised in shared memory up to this count

__device__ __forceinline__ int front_bin_of(const Sys &s, double x) {
  const double u = floor(__ddiv_rn(__dsub_rn(x, s.win_xlo), s.front_bin));
  return u < 0.0 ? 0 : (u > (double)(s.n_fbins - 1) ? s.n_fbins - 1 : (int)u);
}

__global__ void __launch_bounds__(kBlk) k_win_stats(Sys s) {
  __shared__ long long sh[2 * kFbinSmem];
  if (!full_on(s) || !s.st->win_active) return;
  const bool priv = s.n_fbins <= kFbinSmem;
  if (priv)
    for (int q = threadIdx.x; q < 2 * s.n_fbins; q += blockDim.x) sh[q] = 0;
  __syncthreads();
  long long *hist = priv ? sh : s.fbin;
  const int N = s.st->N;
  long long xmax = dkey(-INFINITY);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    const double x = s.x[i], vx = s.v[i];
    const long long k = dkey(x);
    if (k > xmax) xmax = k;
    if (!isfinite(x) || !isfinite(vx)) continue;
    const int b = front_bin_of(s, x);
    atomicAdd((unsigned long long *)&hist[2 * b], (unsigned long long)__double2ll_rn(vx * kTwo40));
    atomicAdd((unsigned long long *)&hist[2 * b + 1], 1ull);
  }
  for (int o = 16; o > 0; o >>= 1) xmax = max(xmax, __shfl_xor_sync(0xffffffffu, xmax, o));
  if ((threadIdx.x & 31) == 0) atomicMax(&s.st->key_xmax, xmax);
  if (priv) {
    __syncthreads();
    for (int q = threadIdx.x; q < 2 * s.n_fbins; q += blockDim.x)
      if (sh[q] != 0) atomicAdd((unsigned long long *)&s.fbin[q], (unsigned long long)sh[q]);
  }
}

// Front, cut and the number of fresh-slab copies to append (capped by the
// box along x and by the capacity).  One block; the bin sums are cleared
// for the next build.
__global__ void __launch_bounds__(kBlk) k_win_plan(Sys s) {
  __shared__ int best;
  if (!full_on(s) || !s.st->win_active) return;
  if (threadIdx.x == 0) best = -1;
  __syncthreads();
  const long long q_up = __double2ll_rn(s.u_p * kTwo40);
  int mine = -1;
  for (int b = threadIdx.x; b < s.n_fbins; b += blockDim.x) {
    const long long sum = s.fbin[2 * b], cnt = s.fbin[2 * b + 1];
    if (cnt > 0 && 2 * sum > cnt * q_up) mine = b;
  }
  if (mine >= 0) atomicMax(&best, mine);
  __syncthreads();
  for (int q = threadIdx.x; q < 2 * s.n_fbins; q += blockDim.x) s.fbin[q] = 0;
  if (threadIdx.x != 0) return;
  DevStatus *st = s.st;
  const double xmax = dkey_inv(st->key_xmax);
  st->win_n_old = st->N;
  st->win_insert = 0;
  st->win_cut = -INFINITY;
  const bool fixed = isfinite(s.fixed_front);
  if (best < 0 && !fixed) return;
  const double front =
      fixed ? s.fixed_front : __dadd_rn(s.win_xlo, __dmul_rn((double)(best + 1), s.front_bin));
  st->win_cut = front - s.L_behind;
  const double need = front + s.L_ahead - xmax;
  long long copies = need > 0.0 ? (long long)ceil(need / s.slab_lx) : 0;
  const double fit = floor(__ddiv_rn(__dsub_rn(__dsub_rn(s.win_xhi, xmax), s.slab_gap), s.slab_lx));
  const long long fit_n = fit > 0.0 ? (long long)fit : 0;
  if (copies > fit_n) copies = fit_n;
  long long add = copies * (long long)s.n_slab;
  const long long room = (long long)s.N_cap - st->N;
  if (add > room) {
    add = room;
    atomicOr(&st->bits, kStCapacity);
  }
  st->win_insert = (int)add;
  st->win_x0 = xmax;
  st->win_id0 = st->next_id;
  st->next_id += (int)add;
  st->N += (int)add;
  st->n_inserted += add;
}

__global__ void __launch_bounds__(kBlk) k_win_insert(Sys s) {
  if (!full_on(s) || !s.st->win_active) return;
  const DevStatus *st = s.st;
  const int add = st->win_insert, n0 = st->win_n_old, id0 = st->win_id0;
  const size_t Nc = s.N_cap;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < add; q += gridDim.x * blockDim.x) {
    const int c = q / s.n_slab, k = q % s.n_slab;
    const double *a = s.slab + 6 * (size_t)k;
    const int i = n0 + q;
    // copy c sits at x offset (x_max + gap) + c * slab_lx, rounded in that order
    const double x0 = __dadd_rn(__dadd_rn(st->win_x0, s.slab_gap), __dmul_rn((double)c, s.slab_lx));
    s.x[i] = __dadd_rn(a[0], x0);
    s.x[Nc + i] = a[1];
    s.x[2 * Nc + i] = a[2];
    for (int d = 0; d < 3; ++d) {
      s.v[d * Nc + i] = a[3 + d];
      s.f[d * Nc + i] = 0.0;
    }
    s.id[i] = id0 + q;
    s.info[i] = s.slab_info;
  }
}

// atoms a window deleted sit in the last bucket, past the kept ones: drop them
__global__ void k_win_trim(Sys s) {
  if (threadIdx.x != 0 || blockIdx.x != 0 || !full_on(s)) return;
  DevStatus *st = s.st;
  const int kept = s.cell_start[s.n_cells];
  st->n_deleted += st->N - kept;
  st->N = kept;
}


__global__ void k_set_flag(Sys s) {
  if (threadIdx.x == 0 && blockIdx.x == 0) s.st->rebuild = 1;
}

__global__ void __launch_bounds__(kBlk) k_bin(Sys s) {
  if (!full_on(s)) return;
  const int N = s.st->N;
  const bool win = s.win_on && s.st->win_active;
  long long xmin = dkey(INFINITY);  // smallest x kept (window: new rear layer)
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
  const Grid &g = s.grid[s.info[i] >> 8];
  if (win) {
    const double x = s.x[i];
    if (x < s.st->win_cut) {  // behind the window: to the deletion bucket
      s.cell_of[i] = s.n_cells;
      s.tmpu[i] = 0;
      atomicAdd(&s.cell_cnt[s.n_cells], 1);
      continue;
    }
    xmin = min(xmin, dkey(x));
  }
  int c[3];
  for (int d = 0; d < 3; ++d) {
    double xv = s.x[(size_t)d * s.N_cap + i];
    if (!isfinite(xv)) {
      atomicOr(&s.st->bits, kStNonfinite);
      xv = g.lo[d];
      s.x[(size_t)d * s.N_cap + i] = xv;
    }
    if (g.per[d]) {
      const double lo = g.lo[d], hi = g.hi[d], L = g.L[d];
      if (xv >= hi || xv < lo) {
        // whole box lengths, one at a time (as the definition states);
        // atoms more than 4 boxes away jump by a floor first
        if (fabs(xv - lo) > 4.0 * L) xv = xv - L * floor((xv - lo) / L);
        for (int it = 0; it < 8 && xv >= hi; ++it) xv = xv - L;
        for (int it = 0; it < 8 && xv < lo; ++it) xv = xv + L;
        if (xv >= hi || xv < lo) xv = lo;
        s.x[(size_t)d * s.N_cap + i] = xv;
      }
    }
    int ck = (int)floor((xv - g.lo[d]) * g.inv_h[d]);
    ck = min(max(ck, 0), g.nc[d] - 1);
    c[d] = ck;
  }
  const int cell = g.cell_off + c[0] + g.nc[0] * (c[1] + g.nc[1] * c[2]);
  s.cell_of[i] = cell;
  s.tmpu[i] = pack_cell(c[0], c[1], c[2]);
  atomicAdd(&s.cell_cnt[cell], 1);
  }
  if (win) {  // one atomic per warp, not per atom
    for (int o = 16; o > 0; o >>= 1) xmin = min(xmin, __shfl_xor_sync(0xffffffffu, xmin, o));
    if ((threadIdx.x & 31) == 0) atomicMin(&s.st->key_xmin, xmin);
  }
}

// block-wide exclusive scan of one value per thread; returns the prefix and
// writes the block total to *total
__device__ __forceinline__ int block_exscan(int v, int *total) {
  __shared__ int warp_sums[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_sums[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    int w = (lane < nw) ? warp_sums[lane] : 0;
    int wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += t;
    }
    if (lane < nw) warp_sums[lane] = wi - w;
    if (lane == nw - 1) *total = wi;
  }
  __syncthreads();
  const int res = warp_sums[warp] + incl - v;
  __syncthreads();
  return res;
}

// ONE: the whole scan in this kernel, where one tile holds all buckets (the
// partials' two launches, ~2.5 us each, are what the scan costs then)
template <bool ONE>
__global__ void __launch_bounds__(kScanThreads) k_scan_apply(Sys s) {
  if (!full_on(s)) return;
  const int base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  int loc[kScanItems];
  int sum = 0;
#pragma unroll
  for (int q = 0; q < kScanItems; ++q) {
    loc[q] = (base + q <= s.n_cells) ? s.cell_cnt[base + q] : 0;
    sum += loc[q];
  }
  __shared__ int tot;
  int pre = block_exscan(sum, &tot) + (ONE ? 0 : s.scan_part[blockIdx.x]);
#pragma unroll
  for (int q = 0; q < kScanItems; ++q) {
    const int c = base + q;
    if (c <= s.n_cells) {
      s.cell_start[c] = pre;
      s.cell_fill[c] = pre;
      s.cell_cnt[c] = 0;  // ready for the next build
    }
    pre += loc[q];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kScanThreads - 1)
    s.cell_start[s.n_cells + 1] = pre;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(Sys s) {
  if (!full_on(s)) return;
  const int base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  int sum = 0;
#pragma unroll
  for (int q = 0; q < kScanItems; ++q)
    if (base + q <= s.n_cells) sum += s.cell_cnt[base + q];
  __shared__ int tot;
  block_exscan(sum, &tot);
  if (threadIdx.x == 0) s.scan_part[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_top(Sys s) {
  if (!full_on(s)) return;
  // n_scan_blocks <= kScanThreads * 8
  constexpr int kPer = 8;
  const int base = threadIdx.x * kPer;
  int loc[kPer];
  int sum = 0;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    loc[q] = (base + q < s.n_scan_blocks) ? s.scan_part[base + q] : 0;
    sum += loc[q];
  }
  __shared__ int tot;
  int pre = block_exscan(sum, &tot);
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    if (base + q < s.n_scan_blocks) s.scan_part[base + q] = pre;
    pre += loc[q];
  }
}

__global__ void __launch_bounds__(kBlk) k_scatter(Sys s) {
  if (!full_on(s)) return;
  const int N = s.st->N;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
  const int pos = atomicAdd(&s.cell_fill[dbg_idx(s, s.cell_of[i], s.n_cells + 1)], 1);
  s.order[dbg_idx(s, pos, s.N_cap)] = i;
  }
}

// Order inside each cell by permanent atom id, so the layout does not depend
// on the order of the scatter's atomics: the atom at slot k of its cell takes
// rank = number of atoms of the cell with a smaller id, and lands at
// cell_start + rank of the final order (kept in tmpi, which k_permute reads
// first and overwrites at the same index).  One thread per atom: the
// comparisons of a cell run in parallel, with independent loads.  Atoms a
// window deletes (the last bucket) keep the scatter's order.
__global__ void __launch_bounds__(kBlk) k_cell_sort(Sys s) {
  if (!full_on(s)) return;
  const int N = s.st->N;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < N; k += gridDim.x * blockDim.x) {
    const int v = s.order[k];
    const int b = s.cell_of[v];
    const int a = s.cell_start[b], e = s.cell_start[b + 1];
    int rank = k - a;
    if (b < s.n_cells) {
      const int key = s.id[v];
      rank = 0;
#pragma unroll 4
      for (int q = a; q < e; ++q) rank += s.id[s.order[q]] < key ? 1 : 0;
    }
    s.tmpi[dbg_idx(s, a + rank, s.N_cap)] = v;
  }
}

template <class P>
__global__ void __launch_bounds__(kBlk) k_permute(Sys s, typename P::vec4 *pg_target) {
  if (!full_on(s)) return;
  const int N = s.st->N;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < N; k += gridDim.x * blockDim.x) {
  const size_t Nc = s.N_cap;
  const int o = dbg_idx(s, s.tmpi[k], s.N_cap);  // the cell-sorted order (k_cell_sort)
  double xv[3];
  for (int d = 0; d < 3; ++d) {
    xv[d] = s.x[d * Nc + o];
    s.tmp[d * Nc + k] = xv[d];
    s.tmp[(3 + d) * Nc + k] = s.v[d * Nc + o];
    s.tmp[(6 + d) * Nc + k] = s.f[d * Nc + o];
    s.xref[d * Nc + k] = xv[d];
  }
  s.tmpi[k] = s.id[o];
  const uint32_t cc = s.tmpu[o];
  s.cellc[k] = cc;
  uint32_t inf = s.info[o] & ~kInfoFar;
  if (s.win_on && s.st->win_active && s.st->win_cut > -INFINITY &&
      xv[0] < dkey_inv(s.st->key_xmin) + s.piston_depth)
    inf |= kInfoPiston;
  const Grid &g = s.grid[inf >> 8];
  double p[3];
  bool far = false;
  for (int d = 0; d < 3; ++d) {
    p[d] = xv[d] - cell_center(g, d, cell_coord(cc, d));
    // the FP32 pre-filter bound assumes |p| <= 2h (true for periodic
    // dimensions after wrapping); atoms clamped into an end cell of a free
    // dimension may lie further out and always take the exact test
    if (!(fabs(p[d]) <= 2.0 * g.h[d])) far = true;
  }
  if (far) inf |= kInfoFar;
  s.tmpu[Nc + k] = inf;
  // a far atom's pre-filter offset is NaN: every float r^2 with it is NaN,
  // fails both band tests and so always takes the exact FP64 test
  s.pf[k] = far ? make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, __uint_as_float(inf))
                : Mixed::make(p[0], p[1], p[2], inf);
  pg_target[k] = P::make(p[0], p[1], p[2], inf);
  }
}

__global__ void __launch_bounds__(kBlk) k_copyback(Sys s) {
  if (!full_on(s)) return;
  const int N = s.st->N;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < N; k += gridDim.x * blockDim.x) {
  const size_t Nc = s.N_cap;
  for (int d = 0; d < 3; ++d) {
    s.x[d * Nc + k] = s.tmp[d * Nc + k];
    s.v[d * Nc + k] = s.tmp[(3 + d) * Nc + k];
    s.f[d * Nc + k] = s.tmp[(6 + d) * Nc + k];
  }
  s.id[k] = s.tmpi[k];
  s.info[k] = s.tmpu[Nc + k];
  }
}

// periodic image crossed when stencil offset sd leaves cell cd of nc cells
__device__ __forceinline__ bool stencil_cell(int cd, int sd, int nc, int per, int *cell,
                                             int *img) {
  int c = cd + sd;
  int n = 0;
  if (per) {
    if (c < 0) {
      c += nc;
      n = -1;
    } else if (c >= nc) {
      c -= nc;
      n = 1;
    }
  } else if (c < 0 || c >= nc) {
    return false;
  }
  *cell = c;
  *img = n;
  return true;
}

__device__ __forceinline__ int image_of(int c, int sd, int nc, int per) {
  if (!per) return 0;
  const int q = c + sd;
  return q < 0 ? -1 : (q >= nc ? 1 : 0);
}

// The definition, rounded step by step without contraction, for a candidate
// inside the pre-filter band or with a far atom:
// d = (x_j - x_i) + n L,  r^2 = (dx^2 + dy^2) + dz^2 < r_ns^2.
__device__ __noinline__ bool exact_pair(const Sys &s, const Grid &g, int i, uint32_t code, int c0,
                                        int c1, int c2, double rns2) {
  const size_t Nc = s.N_cap;
  const int j = nbr_j(code);
  const int nx = image_of(c0, nbr_s(code, 0), g.nc[0], g.per[0]);
  const int ny = image_of(c1, nbr_s(code, 1), g.nc[1], g.per[1]);
  const int nz = image_of(c2, nbr_s(code, 2), g.nc[2], g.per[2]);
  const double ex = __dadd_rn(__dadd_rn(s.x[j], -s.x[i]), __dmul_rn((double)nx, g.L[0]));
  const double ey = __dadd_rn(__dadd_rn(s.x[Nc + j], -s.x[Nc + i]), __dmul_rn((double)ny, g.L[1]));
  const double ez =
      __dadd_rn(__dadd_rn(s.x[2 * Nc + j], -s.x[2 * Nc + i]), __dmul_rn((double)nz, g.L[2]));
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
  return r2 < rns2;
}

// Half lists keep each unordered pair in one of its two atoms' lists: of the
// atom that lies behind along a fixed direction w, of the smaller index (or,
// for an image of the atom itself, the positive stencil offset) where both lie
// level.  In a solid every neighbour at d has one at about -d, so all atoms
// keep the same number (39 of 78 in argon, where the lanes of a warp walk
// their lists together); a parity rule on the indices left 39 +- 4, and a
// warp walked its longest, 48.  w is a direction along which no vector of a
// cubic lattice up to 4.3 half lattice constants is level (0.098 of one at
// least, 0.049 for simple cubic).  The place along w is an integer of the
// atom's record and the shifts are odd integers of the stencil offset, so
// (i, j, s) and (j, i, -s) decide alike whatever the rounding: the half list
// is exactly one of each mirror pair.  Both passed the same distance test.
struct HalfKey {
  float kx, ky, kz;  // units per A: 2^20 for a cell's extent along w
  int sx, sy, sz;    // a cell's extents
  __device__ __forceinline__ explicit HalfKey(const Grid &g) {
    const float wx = -0.1488063f, wy = 0.7473134f, wz = -0.6475951f;
    const float u = 1048576.0f / (fabsf(wx) * g.hf[0] + wy * g.hf[1] + fabsf(wz) * g.hf[2]);
    kx = wx * u;
    ky = wy * u;
    kz = wz * u;
    sx = __float2int_rn(kx * g.hf[0]);
    sy = __float2int_rn(ky * g.hf[1]);
    sz = __float2int_rn(kz * g.hf[2]);
  }
  // an atom's place along w (the integer in the low bits of 1.5 2^23 + p.w; 0
  // for a far atom, whose offsets are NaN)
  __device__ __forceinline__ int at(const float4 &p) const {
    const float f = __fmaf_rn(p.z, kz, __fmaf_rn(p.y, ky, __fmaf_rn(p.x, kx, 12582912.0f)));
    return f == f ? __float_as_int(f) : 0;
  }
  __device__ __forceinline__ int shift(uint32_t code) const {
    return nbr_s(code, 0) * sx + nbr_s(code, 1) * sy + nbr_s(code, 2) * sz;
  }
};
__device__ __forceinline__ bool half_keep(int i, int at_i, uint32_t code, int at_j) {
  const int j = nbr_j(code);
  const bool level = j == i ? (code & 63u) > 21u : i < j;
  return at_i != at_j ? at_i < at_j : level;
}

// where a build writes: the Verlet list (s.nbr), or with the outer list on
// the outer list (s.nbr1, radius rc + skin_outer, always full)
struct ListOut {
  uint32_t *nbr;
  int32_t *nnbr;
  int nmax;
  double rns2;
  int *max_seen;
};

// Verlet lists (the paper's 3x3x3 cell template): one warp per slice of at
// most 32 atoms of one cell, lanes over candidates.
//
// The candidates of a cell are its 27 template cells' atoms in template order,
// flattened: candidate p sits in the range whose cumulative length passes p,
// so every chunk of 32 candidates is full whatever the cells hold.  Phase 0:
// candidates farther than r_ns from the bounding box of the slice's atoms are
// left out, the others packed into the tile in their order (a distance to a
// box per candidate instead of one to every atom of the slice).
// Phase 1: a lane loads one of them, shifts it by
// its stencil offset and tests it against every atom of the slice,
//   r^2 - r_ns^2 = (c.c - r_ns^2) + p.p - 2 c.p,
// two atoms per packed FP32 instruction with their constants broadcast from
// shared memory; one ballot per atom and chunk is that atom's acceptance mask.
// Phase 2: lane k walks atom k's nonzero mask words bit by bit, one entry per
// step in every lane (the atoms of a cell have about equally many), and
// writes them from registers in groups of 8 (full sectors of the list
// layout).  Candidates sit in the lanes in descending order, so that the
// next one is the highest set bit (one instruction).
//
// What binds it is instruction issue: ~6 instructions per 32 tests, ~30 per
// 32 candidates loaded and ~15 per step of phase 2.  The version before gave
// each atom a thread that walked the candidates and staged each of them: 43
// instructions per candidate (tails of every cell's run, the stencil
// arithmetic per atom and cell, one shared store per candidate, lanes of two
// cells diverging).  Phase 2 with a lane per mask word and a scan of their bit
// counts was slower: the accepted candidates sit in few, dense words.
// Measured (ncu, one launch; that version -> lanes over candidates -> phase 0
// added): 388,204 argon atoms (529 candidates, 78 neighbours) 305 -> 213 ->
// 204 us; 442,368 atoms of 64 replicas of densities up to twice that (cells up
// to 10 A wide, up to ~1500 candidates) 510 -> 379 us; 8,388,608 atoms with the
// outer list (890 candidates, 136 entries) 9.1 -> 5.65 -> 5.12 ms; 640,000
// slab atoms 305 -> 290 us; 256 atoms 57 -> 21 -> 19 us, 32,000 71 -> 46 -> 43
// us.  A box of a cell of about r_ns keeps ~70% of the candidates, of a cell
// 1.15 times as wide ~60%.
//
// Error of the FP32 test: atoms in their cells (|p_d| <= 0.6 h) give |c| <=
// 2.8 h, each product and sum rounds to 2^-24 of at most 15 h^2, so r^2 is off
// by less than 5e-6 h^2; atoms clamped into an end cell of a free dimension
// (|p_d| <= 2 h) give 75 h^2 and 2.5e-5 h^2.  Candidates within a band four
// times that wide (Sys.build_band = 2e-5 h^2, and five times it) take the
// exact FP64 test of the definition, and so do far atoms (NaN offsets).
// The distance to the box is a difference of rounded coordinates: its square is
// off by less than 2e-6 h^2 in cells, 1e-5 h^2 with clamped atoms, and phase 0
// takes what is within r_ns^2 + 1e-4 h^2; a slice with a far atom has no box.
// Lists come out in the order of the candidates: template cell, then atom.
constexpr int kBWarps = 4;     // warps per block
constexpr int kTileCh = 32;    // chunks of 32 candidates per tile (the three phases per tile)
// Atoms of a slice at most, by the size of the system: short slices give a
// small system more warps (a warp's chain of dependent loads and shared
// reads takes ~10 us whatever its slice holds), long ones share the loading
// of the candidates.  The steps lie where the slices of one size no longer fit one
// round of blocks.  k_build in us with 8 / 16 / 32 atoms per slice: 9,724 EAM atoms
// 29 / 31 / 44, 13,500 EAM 29 / 35 / 47, 19,652 EAM 34 / 36 / 47 and LJ 36 / 35 / 48,
// 32,000 EAM 52 / 36 / 49 and LJ 53 / 41 / 44, 42,592 EAM 58 / 40 / 49 and LJ 65 /
// 43 / 52, 50,688 LJ 70 / 56 / 53, 55,296 EAM 73 / 62 / 53, 62,500 LJ 85 / 73 / 58,
// 131,072 (6 A lists) 137 / 100 / 90, 388,204 LJ 405 / 290 / 201.
inline int slice_atoms(int n) { return n < 24576 ? 8 : (n < 49152 ? 16 : 32); }
struct BuildWarp {
  uint32_t ent[kTileCh * 32];      // list entries of the tile's candidates, by chunk and lane
  uint4 mask[kTileCh / 2][16];     // per chunk and atom pair: (c, k), (c, k+1), (c+1, k), (c+1, k+1)
  float4 a0[16], a1[16];           // atom pairs: -2x, -2x', -2y, -2y' | -2z, -2z', p.p, p.p'
  float4 sh[28];                   // template cell: shift s h, entry code in .w
  int end[28];                     // end of the template cell's candidates (flattened)
  int off[28];                     // atom = candidate + off
  int key[32];                     // HALF: places of the slice's atoms along w
  int self[32];                    // where the slice's own atoms sit in the tile (-1: not in it)
  uint8_t chunk[kTileCh][32];      // phase 2: chunk of an atom's w-th nonzero mask word
};

constexpr uint32_t kNoEntry = 0xffffffffu;  // stencil code 63: no candidate has it

// floats in the order of signed integers (NaN past the infinities)
__device__ __forceinline__ int ordered_int(float v) {
  const int b = __float_as_int(v);
  return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float ordered_float(int b) {
  return __int_as_float(b ^ ((b >> 31) & 0x7fffffff));
}

template <bool HALF>
__global__ void __launch_bounds__(32 * kBWarps, 5) k_build(Sys s, ListOut lo_, int slice_max) {
  __shared__ BuildWarp sm_[kBWarps];
  if (!full_on(s) || s.half == 2) return;  // 2: forces straight from the cells, no list
  BuildWarp &sm = sm_[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const int N = s.st->N;
  const size_t Nc = s.N_cap;
  const float mid = (float)lo_.rns2;
  const int ngroups = lo_.nmax / kGroup;
  const unsigned full = 0xffffffffu;
  const int warps = gridDim.x * kBWarps;
  for (int base = slice_max * (blockIdx.x * kBWarps + (threadIdx.x >> 5)); base < N;
       base += slice_max * warps) {
    // slices: every cell's atoms in equal parts of at most slice_max; this
    // warp takes those that start in its slice_max atoms
    int n_sl = 0;
    bool lead = false;
    if (lane < slice_max && base + lane < N) {
      const uint32_t cc = s.cellc[base + lane];
      const Grid &g = s.grid[s.info[base + lane] >> 8];
      const int cell = dbg_idx(s, g.cell_off + cell_coord(cc, 0) +
                                      g.nc[0] * (cell_coord(cc, 1) + g.nc[1] * cell_coord(cc, 2)),
                               s.n_cells);
      const int c0 = s.cell_start[cell], n = s.cell_start[cell + 1] - c0;
      const int parts = (n + slice_max - 1) / slice_max;
      const int sz = parts > 0 ? (n + parts - 1) / parts : 1;
      const int k = base + lane - c0;
      lead = k % sz == 0;
      n_sl = min(sz, n - k);
    }
    for (unsigned leads = __ballot_sync(full, lead); leads; leads &= leads - 1) {
      const int l0 = __ffs(leads) - 1;
      const int a0 = base + l0, n = __shfl_sync(full, n_sl, l0);
      const uint32_t cc = s.cellc[a0];
      const Grid &g = s.grid[s.info[a0] >> 8];
      const HalfKey hk(g);
      const int c0 = cell_coord(cc, 0), c1 = cell_coord(cc, 1), c2 = cell_coord(cc, 2);
      // ---- the candidates: 27 runs of atoms, flattened --------------------
      int len = 0, first = 0;
      float4 sh = make_float4(0.f, 0.f, 0.f, 0.f);
      if (lane < 27) {
        const int sx = lane % 3 - 1, sy = (lane / 3) % 3 - 1, sz = lane / 9 - 1;
        int cx, cy, cz, nx, ny, nz;
        if (stencil_cell(c0, sx, g.nc[0], g.per[0], &cx, &nx) &&
            stencil_cell(c1, sy, g.nc[1], g.per[1], &cy, &ny) &&
            stencil_cell(c2, sz, g.nc[2], g.per[2], &cz, &nz)) {
          const int cj = dbg_idx(s, g.cell_off + cx + g.nc[0] * (cy + g.nc[1] * cz), s.n_cells);
          first = s.cell_start[cj];
          len = dbg_idx(s, s.cell_start[cj + 1], s.N_cap + 1, first) - first;
        }
        sh = make_float4((float)sx * g.hf[0], (float)sy * g.hf[1], (float)sz * g.hf[2],
                         __uint_as_float(pack_nbr(0, sx, sy, sz)));
      }
      int incl = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(full, incl, o);
        if (lane >= o) incl += t;
      }
      const int total = __shfl_sync(full, incl, 31);
      const float bx = 0.6f * g.hf[0], by = 0.6f * g.hf[1], bz = 0.6f * g.hf[2];
      // in its cell (false for NaN too)
      auto inside = [&](const float4 &p) {
        return fabsf(p.x) <= bx && fabsf(p.y) <= by && fabsf(p.z) <= bz;
      };
      __syncwarp();  // the previous slice's reads are done
      if (lane < 28) {
        sm.sh[lane] = sh;
        sm.end[lane] = incl;  // lane 27: the total
        sm.off[lane] = first - (incl - len);
      }
      bool out_a = false, far_a = false;
      float lo[3], hi[3];  // the slice's bounding box
      {
        float4 p = make_float4(0.f, 0.f, 0.f, 1e30f);  // no atom: far from everything
        if (lane < n) {
          p = __ldg(s.pf + a0 + lane);
          out_a = !inside(p);
          if (HALF) sm.key[lane] = hk.at(p);
          p.w = fmaf(p.z, p.z, fmaf(p.y, p.y, p.x * p.x));
          far_a = !(p.w == p.w);
        }
        const float pd[3] = {p.x, p.y, p.z};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          lo[d] = ordered_float(__reduce_min_sync(full, lane < n ? ordered_int(pd[d]) : INT_MAX));
          hi[d] = ordered_float(__reduce_max_sync(full, lane < n ? ordered_int(pd[d]) : INT_MIN));
        }
        float *q = reinterpret_cast<float *>(&sm.a0[lane >> 1]) + (lane & 1);
        q[0] = -2.f * p.x;
        q[2] = -2.f * p.y;
        q = reinterpret_cast<float *>(&sm.a1[lane >> 1]) + (lane & 1);
        q[0] = -2.f * p.z;
        q[2] = p.w;
      }
      __syncwarp();
      const float mx = 0.5f * (lo[0] + hi[0]), my = 0.5f * (lo[1] + hi[1]), mz = 0.5f * (lo[2] + hi[2]);
      const float wx = 0.5f * (hi[0] - lo[0]), wy = 0.5f * (hi[1] - lo[1]), wz = 0.5f * (hi[2] - lo[2]);
      const float cull = __any_sync(full, far_a) ? INFINITY : mid + 5.0f * s.build_band;
      int t_tile = 0;  // this lane's template cell (moves up with its candidates)
      int count = 0;  // this lane's atom
      int next_p = 0;
      for (bool one = true; next_p < total; one = false) {
        // ---- phase 0: the tile's candidates, those within reach of the box -
        int slots = 0;
        sm.self[lane] = -1;
        __syncwarp();
        int t = t_tile;
        float4 rn[2];  // the records of the next 64 candidates, loaded ahead
        int jn[2], tn[2];
        auto look = [&](int base_p) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int p = base_p + 32 * h + lane;
            tn[h] = -1;
            if (p < total) {
              while (p >= sm.end[t]) ++t;
              tn[h] = t;
              jn[h] = dbg_idx(s, p + sm.off[t], s.N_cap);
              rn[h] = __ldg(s.pf + jn[h]);
            }
          }
        };
        look(next_p);
        for (; next_p < total && slots <= 32 * kTileCh - 64; next_p += 64) {
          const float4 r[2] = {rn[0], rn[1]};
          const int jc[2] = {jn[0], jn[1]}, tc[2] = {tn[0], tn[1]};
          t_tile = t;
          look(next_p + 64);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            bool in = tc[h] >= 0;
            uint32_t code = 0;
            if (in) {
              const float4 d = sm.sh[tc[h]];
              code = __float_as_uint(d.w);
              const float gx = fmaxf(fabsf(r[h].x + d.x - mx) - wx, 0.0f);
              const float gy = fmaxf(fabsf(r[h].y + d.y - my) - wy, 0.0f);
              const float gz = fmaxf(fabsf(r[h].z + d.z - mz) - wz, 0.0f);
              // a far atom (NaN offsets) is within reach of everything
              in = !(fmaf(gz, gz, fmaf(gy, gy, gx * gx)) > cull) || !(r[h].x == r[h].x);
            }
            const unsigned b = __ballot_sync(full, in);
            const int at = slots + __popc(b & ((1u << lane) - 1u));
            if (in) {
              sm.ent[at] = code | ((uint32_t)jc[h] << 6);
              if (code == 21u && (unsigned)(jc[h] - a0) < (unsigned)n) sm.self[jc[h] - a0] = at;
            }
            slots += __popc(b);
          }
        }
        __syncwarp();
        const int n_ch = (slots + 31) >> 5;
        // ---- phase 1: two chunks of 32 candidates at a time ---------------
        float4 r2[2];  // the records of the next pair of chunks, loaded ahead
        uint32_t e2[2];
        auto fetch = [&](int c) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int p = 32 * (c + h) + 31 - lane;
            e2[h] = kNoEntry;
            if (p < slots) {
              e2[h] = sm.ent[p];
              r2[h] = __ldg(s.pf + nbr_j(e2[h]));
            }
          }
        };
        fetch(0);
        for (int c = 0; c < n_ch; c += 2) {
          float4 q[2];  // shifted candidate, c.c - r_ns^2
          uint32_t e[2];
          int at_c[2] = {0, 0};  // HALF: the candidate's place along w
          bool out_c = out_a, far_c = far_a;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            q[h] = make_float4(0.f, 0.f, 0.f, 1e30f);
            e[h] = e2[h];
            if (e[h] != kNoEntry) {
              const float4 r = r2[h];
              const float4 d = sm.sh[(e[h] & 3u) + 3u * ((e[h] >> 2) & 3u) + 9u * ((e[h] >> 4) & 3u)];
              const float x = r.x + d.x, y = r.y + d.y, z = r.z + d.z;
              q[h] = make_float4(x, y, z, fmaf(z, z, fmaf(y, y, x * x)) - mid);
              out_c = out_c || !inside(r);
              if (HALF) at_c[h] = hk.at(r) + hk.shift(e[h]);
              far_c = far_c || !(r.x == r.x);
            }
          }
          fetch(c + 2);
          float near = 1e30f;  // smallest distance of a test from r_ns^2
          auto keep = [&](int k, int h) {
            return !HALF || half_keep(a0 + k, sm.key[k], e[h], at_c[h]);
          };
#pragma unroll 4
          for (int k = 0; k < n; k += 2) {
            const float4 u = sm.a0[k >> 1], v = sm.a1[k >> 1];
            unsigned b[4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              float2 d2 = __fadd2_rn(make_float2(q[h].w, q[h].w), make_float2(v.z, v.w));
              d2 = __ffma2_rn(make_float2(q[h].x, q[h].x), make_float2(u.x, u.y), d2);
              d2 = __ffma2_rn(make_float2(q[h].y, q[h].y), make_float2(u.z, u.w), d2);
              d2 = __ffma2_rn(make_float2(q[h].z, q[h].z), make_float2(v.x, v.y), d2);
              near = fminf(near, fminf(fabsf(d2.x), fabsf(d2.y)));
              b[2 * h] = __ballot_sync(full, d2.x < 0.0f && keep(k, h));
              b[2 * h + 1] = __ballot_sync(full, d2.y < 0.0f && keep(k + 1, h));
            }
            if (lane == 0) sm.mask[c >> 1][k >> 1] = make_uint4(b[0], b[1], b[2], b[3]);
          }
          const float width = __any_sync(full, out_c) ? 5.0f * s.build_band : s.build_band;
          if (__any_sync(full, far_c || !(near > width))) {
            // rare: the two chunks again, with the exact test where needed
            __syncwarp();
            for (int k = 0; k < n; ++k) {
              const float *u = reinterpret_cast<const float *>(&sm.a0[k >> 1]) + (k & 1);
              const float *v = reinterpret_cast<const float *>(&sm.a1[k >> 1]) + (k & 1);
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const float d2 = fmaf(q[h].z, v[0], fmaf(q[h].y, u[2], fmaf(q[h].x, u[0], q[h].w + v[2])));
                bool acc = d2 < -width;
                if (!acc && !(d2 > width) && e[h] != kNoEntry)
                  acc = exact_pair(s, g, a0 + k, e[h], c0, c1, c2, lo_.rns2);
                const unsigned b = __ballot_sync(full, acc && keep(k, h));
                if (lane == 0)
                  reinterpret_cast<uint32_t *>(&sm.mask[c >> 1][k >> 1])[2 * h + (k & 1)] = b;
              }
            }
          }
        }
        __syncwarp();
        // an atom is no neighbour of itself (its images are)
        uint32_t *mw = reinterpret_cast<uint32_t *>(sm.mask) + 4 * (lane >> 1) + (lane & 1);
        auto word = [](int c) { return (c >> 1) * 64 + 2 * (c & 1); };
        const int self = sm.self[lane];
        if (lane < n && (unsigned)self < (unsigned)(32 * n_ch))
          mw[word(self >> 5)] &= ~(0x80000000u >> (self & 31));
        // ---- phase 2: this lane's atom takes its accepted entries ----------
        int words = 0, add = 0;  // its nonzero mask words (moved to the front), entries
        for (int c = 0; c < n_ch; ++c) {
          const uint32_t m = lane < n ? mw[word(c)] : 0u;
          if (m) {
            mw[word(words)] = m;
            sm.chunk[words][lane] = (uint8_t)c;
            ++words;
          }
          add += __popc(m);
        }
        uint32_t m = 0;
        int at = 0;
        const uint32_t *ent = sm.ent;
        // the next accepted entry (the lane's list goes on with pad entries)
        auto next = [&]() -> uint32_t {
          if (m == 0 && at < words) {
            m = mw[word(at)];
            ent = sm.ent + 32 * sm.chunk[at][lane];
            ++at;
          }
          const int z = __clz(m);
          const uint32_t e = ent[min(z, 31)];
          const bool some = m != 0;
          m ^= some ? 0x80000000u >> z : 0u;
          return some ? e : pad_entry(Nc);
        };
        const int most = __reduce_max_sync(full, add);
        if (one) {
          for (int k = 0; k < most; k += kGroup) {
            uint32_t w[kGroup];
#pragma unroll
            for (int q = 0; q < kGroup; ++q) w[q] = next();
            if (k < add && (k >> 3) < ngroups) {
              uint4 *o = reinterpret_cast<uint4 *>(lo_.nbr) + ((size_t)(k >> 3) * Nc + (a0 + lane)) * 2;
              // lists are written once per build and read by the next pass from
              // HBM: evict-first stores keep L2 for the records the builds gather
              __stcs(o, make_uint4(w[0], w[1], w[2], w[3]));
              __stcs(o + 1, make_uint4(w[4], w[5], w[6], w[7]));
            }
          }
        } else {  // crowded cells: further tiles go on inside the last group
          for (int k = 0; k < most; ++k) {
            const uint32_t e = next();
            if (k < add && ((count + k) >> 3) < ngroups) lo_.nbr[ell_index(count + k, a0 + lane, Nc)] = e;
          }
          if (lane < n)
            for (int k = count + add; (k & 7) && (k >> 3) < ngroups; ++k)
              lo_.nbr[ell_index(k, a0 + lane, Nc)] = pad_entry(Nc);
        }
        count += add;
        __syncwarp();
      }
      if (lane < n) {
        lo_.nnbr[a0 + lane] = count;
        if (count > lo_.nmax) {
          atomicOr(&s.st->bits, kStOverflow);
          atomicMax(lo_.max_seen, count);
          s.st->build_ovf = 1;
        }
      }
    }
  }
}

// ---- two-level lists: the Verlet list filtered from the outer list ----------
// Every build measures d, the largest displacement of an atom since the last
// full build (x_full: positions right after that build).  A pair closer than
// rc + skin now was closer than rc + skin + 2 d then, so while
// d <= (skin_outer - skin) / 2 the outer list holds every pair within
// rc + skin, and filtering it gives the exact Verlet list.
__global__ void __launch_bounds__(kBlk) k_outer_disp(Sys s) {
  if (!flag_on(s) || !s.outer_on || s.st->full) return;
  const int N = s.st->N;
  const size_t Nc = s.N_cap;
  double m = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    const double dx = s.x[i] - s.xfull[i], dy = s.x[Nc + i] - s.xfull[Nc + i],
                 dz = s.x[2 * Nc + i] - s.xfull[2 * Nc + i];
    const double d2 = dx * dx + dy * dy + dz * dz;
    // a non-finite position forces a full build (whose binning reports it)
    m = d2 == d2 ? fmax(m, d2) : INFINITY;
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  // non-negative doubles order like their bit patterns
  if ((threadIdx.x & 31) == 0) atomicMax(&s.st->dmax_key, __double_as_longlong(m));
}

__global__ void k_outer_decide(Sys s) {
  if (threadIdx.x != 0 || blockIdx.x != 0 || !flag_on(s) || !s.outer_on) return;
  DevStatus *st = s.st;
  if (!st->full) {
    // sqrt rounded up by one part in 2^40: the bound stays a bound
    const double d = sqrt(__longlong_as_double(st->dmax_key)) * (1.0 + 0x1p-40);
    st->d_acc = d;
    if (!(d <= s.outer_budget)) st->full = 1;
  }
  if (st->full) {
    st->d_acc = 0.0;
    st->outer_valid = 1;  // the chain below rebuilds the outer list
    st->n_full_builds += 1;
  }
  st->dmax_key = 0;
}

// full builds: x_full = x (after the re-sort); filter builds: the trigger's
// reference positions (FP64 x_ref and the FP32 cell-relative record the
// pre-filter reads) move to the current positions; atoms keep their cells,
// so the outer list's stencil codes stay exact
__global__ void __launch_bounds__(kBlk) k_outer_refresh(Sys s) {
  if (!flag_on(s) || !s.outer_on) return;
  const int N = s.st->N;
  const size_t Nc = s.N_cap;
  if (s.st->full) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x)
      for (int d = 0; d < 3; ++d) s.xfull[d * Nc + i] = s.x[d * Nc + i];
    return;
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    double p[3];
    const uint32_t cc = s.cellc[i];
    const uint32_t inf = s.info[i];
    const Grid &g = s.grid[inf >> 8];
    for (int d = 0; d < 3; ++d) {
      const double xv = s.x[d * Nc + i];
      s.xref[d * Nc + i] = xv;
      p[d] = xv - cell_center(g, d, cell_coord(cc, d));
    }
    if (!(inf & kInfoFar)) s.pf[i] = Mixed::make(p[0], p[1], p[2], inf);
  }
}

// the Verlet list (full or half) from the outer list: an FP32 pre-filter whose
// band (filt_lo .. filt_hi) is its own, and inside it the exact FP64 test that
// k_build ends in too, on the outer list's candidates in their order, so the
// list equals a build from the cells
template <bool HALF>
__global__ void __launch_bounds__(kBlk) k_build_filter(Sys s) {
  __shared__ uint32_t stage[2 * kGroup][kBlk];
  if (!flag_on(s) || !s.outer_on || s.half == 2) return;
  const int N = s.st->N;
  const size_t Nc = s.N_cap;
  const float lo_thr = s.filt_lo, hi_thr = s.filt_hi;
  const double rns2 = s.rns2;
  const int ngroups = s.nmax / kGroup;
  const int tx = threadIdx.x;
  for (int i = blockIdx.x * kBlk + tx; i < N; i += gridDim.x * kBlk) {
    const float4 pi = __ldg(s.pf + i);
    const Grid &g = s.grid[__float_as_uint(pi.w) >> 8];
    const uint32_t cc = s.cellc[i];
    const int c0 = cell_coord(cc, 0), c1 = cell_coord(cc, 1), c2 = cell_coord(cc, 2);
    const int n1 = min(s.nnbr1[i], s.nmax1);
    const HalfKey hk(g);
    const int at_i = hk.at(pi);
    int count = 0;
    auto flush = [&](int grp, int fill) {
      if (grp >= ngroups) return;
      const int h = (grp & 1) * kGroup;
      const uint32_t pad = pad_entry(Nc);
      uint32_t w[kGroup];
#pragma unroll
      for (int q = 0; q < kGroup; ++q) w[q] = q < fill ? stage[h + q][tx] : pad;
      uint4 *o = reinterpret_cast<uint4 *>(s.nbr) + ((size_t)grp * Nc + i) * 2;
      // lists are written once per build and read by the next pass from
      // HBM: evict-first stores keep L2 for the records the builds gather
      __stcs(o, make_uint4(w[0], w[1], w[2], w[3]));
      __stcs(o + 1, make_uint4(w[4], w[5], w[6], w[7]));
    };
    const uint4 *row = reinterpret_cast<const uint4 *>(s.nbr1) + (size_t)i * 2;
    // r^2 (FP32) of two candidates at once with the packed FP32 instructions:
    // d = (p_j - p_i) + s h, the stencil shifts s 4^d from the entries' codes
    // (cell size pre-scaled by 4^-d)
    const float2 mpx = make_float2(-pi.x, -pi.x), mpy = make_float2(-pi.y, -pi.y),
                 mpz = make_float2(-pi.z, -pi.z);
    const float2 hx2 = make_float2(g.hf[0], g.hf[0]),
                 hy2 = make_float2(0.25f * g.hf[1], 0.25f * g.hf[1]),
                 hz2 = make_float2(0.0625f * g.hf[2], 0.0625f * g.hf[2]);
    auto r2pair = [&](uint32_t ea, uint32_t eb, const float4 &qa, const float4 &qb) {
      const float2 sx = __fadd2_rn(make_float2(__uint_as_float((ea & 3u) | 0x4B000000u),
                                               __uint_as_float((eb & 3u) | 0x4B000000u)),
                                   make_float2(-8388609.0f, -8388609.0f));
      const float2 sy = __fadd2_rn(make_float2(__uint_as_float((ea & 12u) | 0x4B000000u),
                                               __uint_as_float((eb & 12u) | 0x4B000000u)),
                                   make_float2(-8388612.0f, -8388612.0f));
      const float2 sz = __fadd2_rn(make_float2(__uint_as_float((ea & 48u) | 0x4B000000u),
                                               __uint_as_float((eb & 48u) | 0x4B000000u)),
                                   make_float2(-8388624.0f, -8388624.0f));
      const float2 dx = __ffma2_rn(sx, hx2, __fadd2_rn(make_float2(qa.x, qb.x), mpx));
      const float2 dy = __ffma2_rn(sy, hy2, __fadd2_rn(make_float2(qa.y, qb.y), mpy));
      const float2 dz = __ffma2_rn(sz, hz2, __fadd2_rn(make_float2(qa.z, qb.z), mpz));
      return __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
    };
    // four candidates at a time: their gathers go out together
    auto block4 = [&](const uint32_t *e) {
      const int before = count;
      // whole groups: slots past n1 hold pad_entry, whose record (pf[N_cap])
      // lies 1e18 A away and fails the pre-filter outright
      float4 pj[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) pj[u] = __ldg(s.pf + dbg_idx(s, nbr_j(e[u]), Nc + 1, i));
      const float2 r01 = r2pair(e[0], e[1], pj[0], pj[1]);
      const float2 r23 = r2pair(e[2], e[3], pj[2], pj[3]);
      const float r2v[4] = {r01.x, r01.y, r23.x, r23.y};
      bool band = false;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t code = e[u];
        const float r2f = r2v[u];
        const bool ok = !HALF || half_keep(i, at_i, code, hk.at(pj[u]) + hk.shift(code));
        const bool acc = ok && r2f < lo_thr;
        band = band || (ok && !acc && !(r2f > hi_thr));
        stage[count & 15][tx] = code;  // kept only if accepted
        count += acc ? 1 : 0;
      }
      if (band) {
        count = before;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t code = e[u];
          const float r2f = r2v[u];
          const bool ok = !HALF || half_keep(i, at_i, code, hk.at(pj[u]) + hk.shift(code));
          bool acc = ok && r2f < lo_thr;
          if (ok && !acc && !(r2f > hi_thr)) acc = exact_pair(s, g, i, code, c0, c1, c2, rns2);
          stage[count & 15][tx] = code;
          count += acc ? 1 : 0;
        }
      }
      if ((before >> 3) != (count >> 3)) flush(before >> 3, kGroup);
    };
    // the next group's entries are loaded while this group runs (their HBM
    // latency overlaps the candidate gathers)
    uint4 na = make_uint4(0, 0, 0, 0), nb = na;
    if (n1 > 0) {
      ld_group(row, na, nb);
    }
    for (int k0 = 0; k0 < n1; k0 += kGroup) {
      const uint4 a = na, b = nb;
      row += Nc * 2;
      if (k0 + kGroup < n1) {
        ld_group(row, na, nb);
      }
      const uint32_t ea[4] = {a.x, a.y, a.z, a.w};
      const uint32_t eb[4] = {b.x, b.y, b.z, b.w};
      block4(ea);
      block4(eb);
    }
    if (count & 7) flush(count >> 3, count & 7);
    s.nnbr[i] = count;
    if (count > s.nmax) {
      atomicOr(&s.st->bits, kStOverflow);
      atomicMax(&s.st->max_nnbr, count);
      s.st->build_ovf = 1;
    }
  }
}

// A build that stepping triggered and whose list outgrew its capacity stops
// the stepping (st->abort): the lists are truncated, so no force pass may use
// them; the host regrows the workspace, carries the state over and resumes.
// graph_kernels: kernels of the conditional body that this launch ends (else 0).
__global__ void k_finish(Sys s, int graph_kernels) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  DevStatus *st = s.st;
  st->n_graph_kernels += graph_kernels;
  if (st->rebuild) {
    st->rebuild = 0;
    st->n_builds += 1;
    st->since_build = 0;
    if (st->step_build && st->build_ovf) st->abort = 1;
  }
}

// Replay of a filter build (checkpoint restore with two-level lists): the
// Verlet list is filtered from the outer list of the full build just
// replayed, at the positions now in x, as a stepping build would.
__global__ void k_replay_filter_head(Sys s) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  DevStatus *st = s.st;
  st->rebuild = 1;
  st->full = 0;
  st->win_active = 0;
  st->win_cut = -INFINITY;
  st->step_build = 0;
  st->build_ovf = 0;
  st->outer_valid = 1;
}

// gather copy of the positions in x with the cells of the last build (the
// expression of the step epilogue); ODD: only after a loop body that ended on
// the other copy, and not after a full build, which has written this one
template <class P, bool ODD>
__global__ void __launch_bounds__(kBlk) k_regather(Sys s, typename P::vec4 *out) {
  if (ODD && (!s.st->regather || full_on(s))) return;
  const int N = s.st->N;
  const size_t Nc = s.N_cap;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    const uint32_t inf = s.info[i];
    const Grid &g = s.grid[inf >> 8];
    const uint32_t cc = s.cellc[i];
    out[i] = P::make(s.x[i] - cell_center(g, 0, cell_coord(cc, 0)),
                     s.x[Nc + i] - cell_center(g, 1, cell_coord(cc, 1)),
                     s.x[2 * Nc + i] - cell_center(g, 2, cell_coord(cc, 2)), inf);
  }
}

inline int nblk(long long n, int b) { return (int)((n + b - 1) / b); }

}  // namespace

void launch_set_rebuild_flag(const Sys &s, cudaStream_t st) { k_set_flag<<<1, 32, 0, st>>>(s); }

// The chain is enqueued every step and usually has nothing to do: a grid of
// N/256 blocks that all exit at once still costs ~0.1 ms of block
// scheduling, so every kernel of the chain runs on a persistent grid (a few
// blocks per SM) with grid-stride loops; a skipped rebuild costs a few us.
int persistent_blocks(const void *fn, int threads, int smem) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem) != cudaSuccess ||
      occ <= 0)
    occ = 1;
  return sms * occ;
}

void launch_rebuild_head(const Sys &s, int count_step, cudaGraphConditionalHandle h,
                         cudaStream_t st) {
  k_pre<<<1, 32, 0, st>>>(s, count_step, 1, h);
}

int rebuild_chain_kernels(const Sys &s) {
  return (s.n_scan_blocks == 1 ? 9 : 11) + (s.win_on ? 4 : 0) + (s.outer_on ? 4 : 0);
}

void launch_loop_head(const Sys &s, int places, int kernels, cudaGraphConditionalHandle h,
                      cudaGraphConditionalHandle loop, cudaStream_t st) {
  k_loop_head<<<1, 32, 0, st>>>(s, places, kernels, h, loop);
}

void launch_set_left(const Sys &s, int left, cudaStream_t st) { k_set_left<<<1, 32, 0, st>>>(s, left); }

void launch_rebuild_body(const Sys &s, int target_pg, int precision, int from_graph, int loop,
                         cudaStream_t st) {
  static int g_atom = 0, g_build = 0, g_cells = 0, g_filter = 0;
  if (g_atom == 0) {
    g_atom = persistent_blocks((const void *)k_bin, kBlk, 0);
    // 4 rounds of blocks: slices differ, and the last round is a quarter of one
    g_build = 4 * persistent_blocks((const void *)k_build<false>, 32 * kBWarps, 0);
    g_cells = persistent_blocks((const void *)k_cell_sort, kBlk, 0);
    g_filter = persistent_blocks((const void *)k_build_filter<false>, kBlk, 0);
  }
  const int gN = std::min(g_atom, nblk(s.N_cap > 0 ? s.N_cap : 1, kBlk));
  const int gC = std::min(g_cells, nblk(s.N_cap > 0 ? s.N_cap : 1, kBlk));
  const int slice = slice_atoms(s.N_cap);
  const int gB = std::min(g_build, nblk(s.N_cap > 0 ? s.N_cap : 1, slice * kBWarps));
  const int gF = std::min(g_filter, nblk(s.N_cap > 0 ? s.N_cap : 1, kBlk));
  if (s.outer_on) {
    k_outer_disp<<<gN, kBlk, 0, st>>>(s);
    k_outer_decide<<<1, 32, 0, st>>>(s);
  }
  if (s.win_on) {
    k_win_stats<<<gN, kBlk, 0, st>>>(s);
    k_win_plan<<<1, kBlk, 0, st>>>(s);
    k_win_insert<<<gN, kBlk, 0, st>>>(s);
  }
  k_bin<<<gN, kBlk, 0, st>>>(s);
  if (s.n_scan_blocks == 1) {
    k_scan_apply<true><<<1, kScanThreads, 0, st>>>(s);
  } else {
    k_scan_reduce<<<s.n_scan_blocks, kScanThreads, 0, st>>>(s);
    k_scan_top<<<1, kScanThreads, 0, st>>>(s);
    k_scan_apply<false><<<s.n_scan_blocks, kScanThreads, 0, st>>>(s);
  }
  k_scatter<<<gN, kBlk, 0, st>>>(s);
  k_cell_sort<<<gC, kBlk, 0, st>>>(s);
  if (precision == 0)
    k_permute<Fp64><<<gN, kBlk, 0, st>>>(s, (dvec4 *)s.pg[target_pg]);
  else
    k_permute<Mixed><<<gN, kBlk, 0, st>>>(s, (float4 *)s.pg[target_pg]);
  k_copyback<<<gN, kBlk, 0, st>>>(s);
  if (s.win_on) k_win_trim<<<1, 32, 0, st>>>(s);
  if (!s.outer_on) {
    const ListOut lo{s.nbr, s.nnbr, s.nmax, s.rns2, &s.st->max_nnbr};
    if (s.half == 1)
      k_build<true><<<gB, 32 * kBWarps, 0, st>>>(s, lo, slice);
    else
      k_build<false><<<gB, 32 * kBWarps, 0, st>>>(s, lo, slice);
  } else {
    const ListOut lo{s.nbr1, s.nnbr1, s.nmax1, s.rns2_1, &s.st->max_nnbr1};
    k_build<false><<<gB, 32 * kBWarps, 0, st>>>(s, lo, slice);
    k_outer_refresh<<<gN, kBlk, 0, st>>>(s);
    if (s.half == 1)
      k_build_filter<true><<<gF, kBlk, 0, st>>>(s);
    else
      k_build_filter<false><<<gF, kBlk, 0, st>>>(s);
  }
  if (loop) {
    if (precision == 0)
      k_regather<Fp64, true><<<gN, kBlk, 0, st>>>(s, (dvec4 *)s.pg[target_pg]);
    else
      k_regather<Mixed, true><<<gN, kBlk, 0, st>>>(s, (float4 *)s.pg[target_pg]);
  }
  k_finish<<<1, 32, 0, st>>>(s, from_graph ? rebuild_chain_kernels(s) - 1 + (loop ? 1 : 0) : 0);
}

void launch_rebuild(const Sys &s, int target_pg, int precision, int count_step, cudaStream_t st) {
  k_pre<<<1, 32, 0, st>>>(s, count_step, 0, 0);
  launch_rebuild_body(s, target_pg, precision, 0, 0, st);
}

void launch_replay_filter(const Sys &s, int target_pg, int precision, cudaStream_t st) {
  k_replay_filter_head<<<1, 32, 0, st>>>(s);
  launch_rebuild_body(s, target_pg, precision, 0, 0, st);
}

void launch_regather(const Sys &s, int target_pg, int precision, cudaStream_t st) {
  const int g = std::min(1024, nblk(s.N_cap > 0 ? s.N_cap : 1, kBlk));
  if (precision == 0)
    k_regather<Fp64, false><<<g, kBlk, 0, st>>>(s, (dvec4 *)s.pg[target_pg]);
  else
    k_regather<Mixed, false><<<g, kBlk, 0, st>>>(s, (float4 *)s.pg[target_pg]);
}

int scan_blocks_for(int n_buckets) { return (n_buckets + kScanTile - 1) / kScanTile; }

namespace {
__global__ void k_set_piston(Sys s, const uint8_t *flags, int64_t n_flags) {
  const int N = s.st->N;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    const int o = s.id[i];
    const uint32_t pbit = (flags && o < n_flags && flags[o]) ? kInfoPiston : 0u;
    s.info[i] = (s.info[i] & ~kInfoPiston) | pbit;
    if (o < s.N_cap) s.info0[o] = (s.info0[o] & ~kInfoPiston) | pbit;
  }
}
}  // namespace

void launch_set_piston(const Sys &s, const uint8_t *flags, int64_t n_flags, cudaStream_t st) {
  const int g = std::min(1024, nblk(s.N_cap > 0 ? s.N_cap : 1, kBlk));
  k_set_piston<<<g, kBlk, 0, st>>>(s, flags, n_flags);
}

}  // namespace mdk
