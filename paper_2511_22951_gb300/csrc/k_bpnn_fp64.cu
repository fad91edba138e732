// k_bpnn_fp64.cu -- Behler-Parrinello kernel instances: G4-only FP64 models (k_bpnn.cuh).
#include "k_bpnn.cuh"

namespace mdk {

MDK_BPNN_INSTANCES(, Fp64, true)

}  // namespace mdk
