// K3, CTA-pair form: tiles of 192 columns.
#include "k3p_gemm_pair.cuh"

namespace muxq {
template cudaError_t launch_pair_bn<192, false>(const GemmArgs &, const GemmPlan &, cudaStream_t, bool *);
}
