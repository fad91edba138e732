// k_bpnn_fp64_g5.cu -- Behler-Parrinello kernel instances: FP64 models with G5 functions (k_bpnn.cuh).
#include "k_bpnn.cuh"

namespace mdk {

MDK_BPNN_INSTANCES(, Fp64, false)

}  // namespace mdk
