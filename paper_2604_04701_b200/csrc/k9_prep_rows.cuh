// Shared by the kernels of the two-launch preparation: k_channel_max (k9_prep_rows.cu) and k_quant_rows (k9_quant_rows.cuh, one file
// per granularity: the first launch from a file makes the driver load all kernels in it).
#pragma once
#include "kernels.h"
#include "quant.cuh"

namespace muxq {
namespace prep_rows {

constexpr int kT = 512;
constexpr int kWarps = kT / 32;
constexpr int kStatusCapacity = 5;  // MUXQ_ERR_CAPACITY
constexpr int kStatusTimeout = 6;   // MUXQ_ERR_TIMEOUT

// L2's policy for a load: a line that is not read again before others would push it out goes first.
__device__ __forceinline__ uint64_t l2_policy(bool last_use) {
    uint64_t p;
    if (last_use) asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    else asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// 16-byte load as a volatile statement: a batch of them is issued back to back before the first use, whatever the register
// allocator would rather do.  Plain for k_channel_max, which is running already while the launch before it still writes X;
// read-only (.nc) for k_quant_rows, which starts when X is complete.
__device__ __forceinline__ uint4 ld_v4(const void *p, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ uint4 ld_nc_v4(const void *p, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(pol));
    return v;
}

// The same under a predicate (v unchanged where `on` is 0): a branch around each load costs more than the load.
__device__ __forceinline__ void ld_nc_v4_if(uint4 &v, const void *p, int on, uint64_t pol) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %5, 0;\n\t@q ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %6;\n\t}"
                 : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w) : "l"(p), "r"(on), "l"(pol));
}

// X beyond kLongBytes does not stay in L2 from the first kernel to the second as it is: the codes written and the rows already
// done push out rows still to come.  So k_channel_max marks all but the last kKeepBytes as not needed again, and k_quant_rows
// every row that it has read.  Layers of 16384 rows, us: 5120 -> 1280 149 -> 143.5, 3072 -> 768 81.4 -> 77.9, 5120 -> 1280 per token
// 153.7 -> 148.3; 100 MB kept instead of 80: 144.1, none marked in the first kernel 145.1; 8192 x 3072 (50 MB) is the same either way.
constexpr size_t kLongBytes = 64u << 20, kKeepBytes = 80u << 20;

constexpr uint32_t kMarkedMaximum = 0xFFFFFFFFu;  // as channel 0's maximum: the workspace is marked (k_channel_max)

// Grid, shared memory and instantiation for a's rows; cfg: stream, block size and launch attributes.
template <bool kPerToken>
cudaError_t launch_rows(const PrepArgs &a, cudaLaunchConfig_t &cfg, int sms);

}  // namespace prep_rows
}  // namespace muxq
