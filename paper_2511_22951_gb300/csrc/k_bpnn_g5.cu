// k_bpnn_g5.cu -- Behler-Parrinello kernel instances: mixed models with G5 functions (k_bpnn.cuh).
#include "k_bpnn.cuh"

namespace mdk {

MDK_BPNN_INSTANCES(, Mixed, false)

}  // namespace mdk
