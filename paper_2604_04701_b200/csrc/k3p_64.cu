// K3, CTA-pair form: tiles of 64 columns.
#include "k3p_gemm_pair.cuh"

namespace muxq {
template cudaError_t launch_pair_bn<64, false>(const GemmArgs &, const GemmPlan &, cudaStream_t, bool *);
}
