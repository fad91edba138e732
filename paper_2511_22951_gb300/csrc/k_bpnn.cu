// k_bpnn.cu -- Behler-Parrinello passes: shared memory, choice of the kernel
// instance and launch; the instances of G4-only mixed models (k_bpnn.cuh).
#include "k_bpnn.cuh"

namespace mdk {

MDK_BPNN_INSTANCES(, Mixed, true)
MDK_BPNN_INSTANCES(extern, Mixed, false)
MDK_BPNN_INSTANCES(extern, Fp64, true)
MDK_BPNN_INSTANCES(extern, Fp64, false)

size_t bpnn_smem_bytes(const BPParams &p, int precision, int nmax, int *warps) {
  const size_t rsz = precision == 0 ? 8 : 4;
  const int nW = kBpIn * p.H1 + p.H1 + p.H1 * p.H2 + 2 * p.H2;
  const size_t wbytes = ((size_t)nW * rsz + 15) / 16 * 16;
  const size_t per = slab_bytes(nmax, bpnn_groups(p.nY), rsz);
  int w = precision == 0 ? 4 : 8;
  while (w > 1 && wbytes + (size_t)w * per > 200 * 1024) --w;
  if (warps) *warps = w;
  return wbytes + (size_t)w * per;
}

int configure_bpnn_smem(size_t bytes, int precision) {
  const int b = (int)bytes;
  cudaError_t e = precision == 0 ? bpnn_smem_attr<Fp64, true>(b) : bpnn_smem_attr<Mixed, true>(b);
  if (e == cudaSuccess)
    e = precision == 0 ? bpnn_smem_attr<Fp64, false>(b) : bpnn_smem_attr<Mixed, false>(b);
  return e == cudaSuccess ? 0 : 1;
}

void launch_bpnn(const Sys &s, const BPParams &p, int precision, Mode mode, StepArgs a,
                 cudaStream_t st) {
  int w = 1;
  const size_t sm = bpnn_smem_bytes(p, precision, s.nmax, &w);
  const long long n = s.N_cap > 0 ? s.N_cap : 1;
  const int grid = (int)((n + w - 1) / w);
  auto *pass = precision == 0 ? (p.any5 ? bpnn_pass<Fp64, false> : bpnn_pass<Fp64, true>)
                              : (p.any5 ? bpnn_pass<Mixed, false> : bpnn_pass<Mixed, true>);
  pass(s, p, a, grid, 32 * w, sm, st);
  launch_half_fin(s, precision, mode, a, st);
}

}  // namespace mdk
