// k_force.cu -- per-atom kernels around the force loop (GB300, sm_103a): the
// first half-kick and drift of a step from stored forces, the deterministic
// per-replica sums of energies and virials, and the state / force / per-atom
// copies between the internal cell order and the caller's order.
#include "k_pair.cuh"

namespace mdk {

namespace {

using namespace pair;

constexpr int kBlk = 256;

// ---- first half-kick + drift from the stored forces ---------------------------------
// The same arithmetic as the second half of the fused step epilogue of the
// force pass in use (FP64 forces: the kick c F and drift_publish; FP32 forces
// of the mixed full-list kernels, a.f32: the FP32 kick increment of the FP32
// force the last pass stored exactly, and drift32), so a run split over
// several mdk_step calls is bitwise the run in one call.
template <class P>
__global__ void __launch_bounds__(kBlk) k_kick_drift(Sys s, StepArgs a) {
  const int N = run_n(s, a);
  const int i = blockIdx.x * kBlk + threadIdx.x;
  if (i >= N) return;
  const size_t Nc = s.N_cap;
  const uint32_t inf = s.info[i];
  const int type = inf & 15u;
  double vx = s.v[i], vy = s.v[Nc + i], vz = s.v[2 * Nc + i];
  const bool mixed = sizeof(typename G<P>::R) == 4 && a.f32;
  if (inf & kInfoPiston) {
    vx = s.u_p;
    vy = 0.0;
    vz = 0.0;
  } else if (mixed) {
    vx += kick32(s, a, type, (float)s.f[i]);
    vy += kick32(s, a, type, (float)s.f[Nc + i]);
    vz += kick32(s, a, type, (float)s.f[2 * Nc + i]);
  } else {
    const double c = 0.5 * a.dt * s.acc_over_m[type];
    vx += c * s.f[i];
    vy += c * s.f[Nc + i];
    vz += c * s.f[2 * Nc + i];
  }
  if (mixed)
    drift32(s, a, i, inf, vx, vy, vz);
  else
    drift_publish<P>(s, a, i, inf, vx, vy, vz);
}

// ---- deterministic per-replica sums (fixed order, no atomics on the sums) -----------
// Every block sums one chunk of atoms of one replica (a fixed partition, so
// the result does not depend on the launch) and counts itself in; the block
// that completes a replica adds its chunks' partials in chunk order and hands
// the totals out.  The FP64 pipe of one SM binds a block, so chunks are small
// (red_chunk_for) and the block sum of eight values takes 9 additions per lane
// (block_sum8).  9,724 atoms 57 -> 9 us (two launches, 8192 atoms per block
// and 40 additions per lane before, plus two device copies per replica where
// the caller wants E and the virial), 8,388,608 atoms 168 -> 133 us.
constexpr int kRedThreads = 256;

// The block's sums of acc[0..7]; thread c < 8 gets the sum of value c.  Three
// exchanges halve the values that a lane carries while they double the lanes
// that are summed (lane l ends with value l >> 2), two more finish the warp;
// then warps in order.
__device__ __forceinline__ double block_sum8(double (&acc)[8]) {
  __shared__ double sh[8][kRedThreads / 32];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double v4[4], v2[2];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const bool up = lane & 16;
    const double keep = up ? acc[c + 4] : acc[c], give = up ? acc[c] : acc[c + 4];
    v4[c] = keep + __shfl_xor_sync(full, give, 16);
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const bool up = lane & 8;
    const double keep = up ? v4[c + 2] : v4[c], give = up ? v4[c] : v4[c + 2];
    v2[c] = keep + __shfl_xor_sync(full, give, 8);
  }
  const bool up = lane & 4;
  double v = (up ? v2[1] : v2[0]) + __shfl_xor_sync(full, up ? v2[0] : v2[1], 4);
  v += __shfl_xor_sync(full, v, 2);
  v += __shfl_xor_sync(full, v, 1);
  if ((lane & 3) == 0) sh[lane >> 2][wid] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 8)
#pragma unroll
    for (int w = 0; w < kRedThreads / 32; ++w) t += sh[threadIdx.x][w];
  return t;
}

__global__ void __launch_bounds__(kRedThreads) k_reduce(Sys s, int with_ke, double *E,
                                                       double *virial) {
  __shared__ bool last;
  const int r = blockIdx.x, k = blockIdx.y;
  const Grid &g = s.grid[r];
  const int n = (s.n_rep == 1) ? s.st->N : g.n_atoms;
  const size_t Nc = s.N_cap;
  const int q1 = min(n, (k + 1) * s.red_chunk);
  double acc[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = 0.0;
#pragma unroll 4
  for (int q = k * s.red_chunk + threadIdx.x; q < q1; q += kRedThreads) {
    const int i = g.atom_off + q;
    if (with_ke) acc[0] += s.ka[i];
    acc[1] += s.ea[i];
#pragma unroll
    for (int c = 0; c < 6; ++c) acc[2 + c] += s.wa[c * Nc + i];
  }
  double t = block_sum8(acc);
  double *part = s.red_part + (size_t)r * s.red_chunks * 8;
  if (threadIdx.x < 8) {
    part[(size_t)k * 8 + threadIdx.x] = t;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(s.red_done + r, 1u) == (unsigned)s.red_chunks - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = 0.0;
  for (int q = threadIdx.x; q < s.red_chunks; q += kRedThreads) {
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] += __ldcg(part + (size_t)q * 8 + c);
  }
  t = block_sum8(acc);
  const int c = threadIdx.x;
  if (c < 8) s.red[r * 9 + c] = t;
  if (E && c == 1) E[r] = t;
  if (virial && c >= 2 && c < 8) virial[6 * r + c - 2] = t;
  if (c == 0) {
    s.red[r * 9 + 8] = (double)n;
    s.red_done[r] = 0u;
  }
}

// ---- state in / out in the caller's order -------------------------------------------
template <class P>
__global__ void __launch_bounds__(kBlk) k_load_state(Sys s, const double *x, const double *v,
                                                     int target_pg) {
  const int N = s.st->N;
  const int i = blockIdx.x * kBlk + threadIdx.x;
  if (i >= N) return;
  const size_t Nc = s.N_cap;
  for (int d = 0; d < 3; ++d) {
    s.x[d * Nc + i] = x[3 * (size_t)i + d];
    s.v[d * Nc + i] = v ? v[3 * (size_t)i + d] : 0.0;
    s.f[d * Nc + i] = 0.0;
  }
  s.id[i] = i;
  s.info[i] = s.info0[i];
}

__global__ void __launch_bounds__(kBlk) k_store_state(Sys s, double *x, double *v) {
  const int N = s.st->N;
  const int i = blockIdx.x * kBlk + threadIdx.x;
  if (i >= N) return;
  const size_t Nc = s.N_cap;
  const size_t o = (size_t)s.id[i];
  for (int d = 0; d < 3; ++d) {
    if (x) x[3 * o + d] = s.x[d * Nc + i];
    if (v) v[3 * o + d] = s.v[d * Nc + i];
  }
}

__global__ void __launch_bounds__(kBlk) k_store_forces(Sys s, double *f) {
  const int N = s.st->N;
  const int i = blockIdx.x * kBlk + threadIdx.x;
  if (i >= N) return;
  const size_t Nc = s.N_cap;
  const size_t o = (size_t)s.id[i];
  for (int d = 0; d < 3; ++d) f[3 * o + d] = s.f[d * Nc + i];
}

__global__ void __launch_bounds__(kBlk) k_store_per_atom(Sys s, double *ua, double *wa) {
  const int N = s.st->N;
  const int i = blockIdx.x * kBlk + threadIdx.x;
  if (i >= N) return;
  const size_t Nc = s.N_cap;
  const size_t o = (size_t)s.id[i];
  if (ua) ua[o] = s.ea[i];
  if (wa)
    for (int c = 0; c < 6; ++c) wa[6 * o + c] = s.wa[c * Nc + i];
}



inline int nblk(long long n, int b) { return (int)((n + b - 1) / b); }

}  // namespace





void launch_kick_drift(const Sys &s, int precision, StepArgs a, cudaStream_t st) {
  const int g = nblk(s.N_cap > 0 ? s.N_cap : 1, kBlk);
  if (precision == 0)
    k_kick_drift<Fp64><<<g, kBlk, 0, st>>>(s, a);
  else
    k_kick_drift<Mixed><<<g, kBlk, 0, st>>>(s, a);
}

int launch_reduce(const Sys &s, int with_ke, double *E, double *virial, cudaStream_t st) {
  k_reduce<<<dim3(s.n_rep, s.red_chunks), kRedThreads, 0, st>>>(s, with_ke, E, virial);
  return 1;
}

namespace {
template <class P>
__global__ void k_init_far(Sys s) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const size_t Nc = s.N_cap;
  for (int b = 0; b < 2; ++b)
    reinterpret_cast<typename P::vec4 *>(s.pg[b])[Nc] = P::make(1e18, 1e18, 1e18, 0u);
  s.pf[Nc] = make_float4(1e18f, 1e18f, 1e18f, 0.0f);
}
}  // namespace

void launch_init_far(const Sys &s, int precision, cudaStream_t st) {
  if (precision == 0)
    k_init_far<Fp64><<<1, 32, 0, st>>>(s);
  else
    k_init_far<Mixed><<<1, 32, 0, st>>>(s);
}

void launch_load_state(const Sys &s, const double *x, const double *v, int precision,
                       int target_pg, cudaStream_t st) {
  const int g = nblk(s.N_cap > 0 ? s.N_cap : 1, kBlk);
  if (precision == 0)
    k_load_state<Fp64><<<g, kBlk, 0, st>>>(s, x, v, target_pg);
  else
    k_load_state<Mixed><<<g, kBlk, 0, st>>>(s, x, v, target_pg);
}

void launch_store_state(const Sys &s, double *x, double *v, cudaStream_t st) {
  k_store_state<<<nblk(s.N_cap > 0 ? s.N_cap : 1, kBlk), kBlk, 0, st>>>(s, x, v);
}

void launch_store_forces(const Sys &s, double *f, cudaStream_t st) {
  k_store_forces<<<nblk(s.N_cap > 0 ? s.N_cap : 1, kBlk), kBlk, 0, st>>>(s, f);
}

void launch_store_per_atom(const Sys &s, double *ua, double *wa, cudaStream_t st) {
  k_store_per_atom<<<nblk(s.N_cap > 0 ? s.N_cap : 1, kBlk), kBlk, 0, st>>>(s, ua, wa);
}



}  // namespace mdk
