// Shared by the one-launch decode kernels (k4f_decode_fused.cuh, k4r_decode_row.cu) and their launcher (k4f_decode_fused.cu).
#pragma once
#include <mutex>

#include "kernels.h"
#include "ptx.cuh"
#include "quant.cuh"

namespace muxq {
namespace decode {

constexpr int kT = 512;
constexpr int kWarps = kT / 32;
constexpr int kMaxK = 8192;
constexpr int kMaxBufs = 4;
constexpr int kMaxSmem = 220 * 1024;
// Two places per SM, this layer's CTA in one and the next layer's in the other: with room for a third, CTAs of one layer pile
// up on the SMs that empty first, and those set the pace (12 blocks of width 768 at M = 16, single calls: 432 us, with this floor 344).
constexpr int kMinSmem = 80 * 1024;
constexpr int kBesideSmem = 225 * 1024 - kMinSmem;  // beside at most this much there is room for another layer's CTA
constexpr int kStatusCapacity = 5;  // MUXQ_ERR_CAPACITY
constexpr int kStatusTimeout = 6;   // MUXQ_ERR_TIMEOUT

struct Geometry {
    int rows;      // output channels per chunk
    int bufs;      // chunks in shared memory
    int xpitch;    // bytes per row of codes (mma.sync tiles: 64 modulo 128, so that eight rows' 64 bytes meet no bank twice)
    int wpitch;    // bytes per row of W_q (likewise)
    int off_mask;  // behind the codes: [K] 0xFF at outlier channels (dot products: written only in pieces that hold one)
    int off_list;  // [K / 16] u16: pieces that hold an outlier channel; mma.sync tiles: [K / 64] bytes, segments that do
    int off_red;   // mma.sync tiles: [kWarps][128] partial sums
    int off_w;     // chunks of W_q
    int total;
};

__host__ __device__ constexpr int row_lanes(int MT) { return MT < 4 ? MT : 4; }  // lanes that share a group's token rows
// channels of X that the CTA's warps cover with `slices` slices each
__host__ __device__ constexpr int channels_of(int MT, int slices) { return slices * kWarps * 8 * (32 / row_lanes(MT)); }

__device__ __forceinline__ void bulk_load(void *smem_dst, const void *gsrc, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(smem_dst)),
                 "l"(gsrc), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// 16-byte load as a volatile statement: a batch of them is issued back to back before the first use.  Not a read-only (.nc) one:
// the kernel is running already while the launch before it still writes X.
__device__ __forceinline__ uint4 ld_v4(const void *p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// One split of L1 for every layer: an SM changes it only when it is empty, so with a split per kernel the next layer's CTAs
// pile up on the SMs that empty first (measured: 148 CTAs on 82 SMs).  Only the form that is about to run is set up: these
// calls make the driver load the kernel.
inline cudaError_t set_up(const void *kernel, PerDevice<int> &done, int dev) {
    std::lock_guard<std::mutex> lock(device_mutex());
    if (done.have[dev]) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    done.have[dev] = e == cudaSuccess;
    return e;
}

// Each form of the kernels in a file of its own: the first launch from a file makes the driver load all kernels in it.
// lanes: log2 of lanes per row of W_q - 3; alone: shared memory leaves no room for another layer's CTA on the SM.
template <int MT>
cudaError_t launch_rows(const DecodeFusedArgs &a, const Geometry &geo, const cudaLaunchConfig_t &cfg, int lanes, bool alone, int dev);
cudaError_t launch_row(const DecodeFusedArgs &a, const cudaLaunchConfig_t &cfg, int dev);  // M = 1, K <= 256 kRowMaxChunks, 32 rows a warp at most

constexpr int kRowT = 256;
constexpr int kRowWarps = kRowT / 32;
constexpr int kRowMaxChunks = 6;  // K <= 1536

}  // namespace decode
}  // namespace muxq
