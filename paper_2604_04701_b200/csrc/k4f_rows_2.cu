// K4, fused form: up to 2 token rows.
#include "k4f_decode_fused.cuh"

namespace muxq {
namespace decode {
template cudaError_t launch_rows<2>(const DecodeFusedArgs &, const Geometry &, const cudaLaunchConfig_t &, int, bool, int);
}
}
