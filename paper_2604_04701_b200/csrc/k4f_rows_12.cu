// K4, fused form: up to 12 token rows of wide X.
#include "k4f_decode_fused.cuh"

namespace muxq {
namespace decode {
template cudaError_t launch_rows<12>(const DecodeFusedArgs &, const Geometry &, const cudaLaunchConfig_t &, int, bool, int);
}
}
