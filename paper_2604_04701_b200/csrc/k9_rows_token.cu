// k_quant_rows with one scale per token.
#include "k9_quant_rows.cuh"

namespace muxq {
namespace prep_rows {
template cudaError_t launch_rows<true>(const PrepArgs &, cudaLaunchConfig_t &, int);
}
}
