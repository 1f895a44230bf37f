// K3, CTA-pair form: choice of the instantiation (k3p_gemm_pair.cuh; one file per tile width and cut, k3p_*.cu).
#include "kernels.h"

namespace muxq {

template <int BN, bool kCut>
cudaError_t launch_pair_bn(const GemmArgs &a, const GemmPlan &q, cudaStream_t s, bool *fits);

cudaError_t launch_gemm_pair(const GemmArgs &a, const GemmPlan &q, cudaStream_t s) {
    bool fits = true;
    if (q.parts > 1) {
        const cudaError_t e = q.bn == 256   ? launch_pair_bn<256, true>(a, q, s, &fits)
                              : q.bn == 192 ? launch_pair_bn<192, true>(a, q, s, &fits)
                              : q.bn == 128 ? launch_pair_bn<128, true>(a, q, s, &fits)
                                            : launch_pair_bn<64, true>(a, q, s, &fits);
        if (fits) return e;
    }
    GemmPlan whole = q;
    whole.whole_tiles = q.tiles;
    whole.parts = 1;
    return q.bn == 256   ? launch_pair_bn<256, false>(a, whole, s, &fits)
           : q.bn == 192 ? launch_pair_bn<192, false>(a, whole, s, &fits)
           : q.bn == 128 ? launch_pair_bn<128, false>(a, whole, s, &fits)
                         : launch_pair_bn<64, false>(a, whole, s, &fits);
}

}  // namespace muxq
