// k_quant_rows with one scale per tensor.
#include "k9_quant_rows.cuh"

namespace muxq {
namespace prep_rows {
template cudaError_t launch_rows<false>(const PrepArgs &, cudaLaunchConfig_t &, int);
}
}
