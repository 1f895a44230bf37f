// K3, CTA-pair form: tiles of 256 columns, cut along K.
#include "k3p_gemm_pair.cuh"

namespace muxq {
template cudaError_t launch_pair_bn<256, true>(const GemmArgs &, const GemmPlan &, cudaStream_t, bool *);
}
