// K5: weight quantization (Eq. 2), per tensor or per output channel, storing W_q transposed as
// [N, K] with K contiguous -- the K-major B operand of the INT8 tensor-core GEMM.  Runs once per
// weight, when a model is loaded.
//
// Bound by memory: W is read once (fp16) and W_q written once.  A CTA owns a tile of 64 output channels x kt input
// channels, brings it into shared memory with 16-byte asynchronous copies (all of them in flight at once) and writes
// it back transposed, 128 contiguous bytes of one output channel per eight lanes.
//   per output channel  the eight CTAs of a cluster split K between them and exchange the 64 channel maxima through
//                       distributed shared memory: one launch, no scratch, W never leaves the SMs in between.
//   per tensor          the maximum needs all of W: k_weight_absmax leaves one partial maximum per CTA, and the
//                       tile kernel, launched as its programmatic dependent, loads its tile before it waits for them.
//                       (The same form serves a per-channel W too tall for a cluster's shared memory, with the
//                       channel maxima taken from the detection kernel.)
// Measured, the four projections of a block of width 1280 per channel (59 MB of traffic, 8.9 us at 6.65 TB/s): 33.6 us of
// kernel time in 4 launches (44 with a division next to ties) against 83 us in 12 (memset, reduction with atomics, 32 x 32
// byte-store transpose) before; launched so that their set-up meets the end of the launch before (programmatic serialization, the wait
// ahead of the first load) 32.1 us, four calls through the binding 41.2 -> 32.9 us where calls follow one another (a first pass by itself 7 % less).  What is left is latency:
// 5.5 us for 1280 x 1280, a launch, one round of copies, two cluster barriers and the store.
#include "kernels.h"
#include "ptx.cuh"
#include "quant.cuh"

namespace muxq {

namespace {

constexpr int kThreads = 256;           // (the tile kernel also runs with twice as many)
constexpr int kCols = 64;               // output channels per tile: 128 bytes of a W row
constexpr int kCluster = 8;             // most CTAs that share the K range of one column stripe
constexpr int kMaxTileRows = 1600;      // 204,800 bytes of shared memory
constexpr int kTileRows = 128;          // tile height without a cluster

__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool valid) {  // zero-fills when not valid
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

// Chunk (16 bytes = 8 output channels) c8 of tile row `row` sits at c8 ^ (row / 16 mod 8): the eight lanes that
// read the same column pair at eight different groups of 16 rows then hit eight different bank groups.
__device__ __forceinline__ int tile_offset(int row, int c8) { return row * 128 + ((c8 ^ ((row >> 4) & 7)) << 4); }

__global__ void __launch_bounds__(kThreads) k_weight_absmax(const QuantWeightArgs a, float *partial) {
    // the dependent loads its tiles of W at once: behind the wait, when whatever precedes this kernel in the stream has completed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int G = a.N >> 3, total = gridDim.x * kThreads;
    const int drow = total / G, dg = total - drow * G;
    const int i0 = blockIdx.x * kThreads + threadIdx.x;
    int row = i0 / G, g = i0 - row * G;
    __half2 m = __float2half2_rn(0.f);
    while (row < a.K) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            v[u] = row < a.K ? ld_plain_v4(reinterpret_cast<const uint4 *>(a.W + (size_t)row * a.ldw) + g)
                             : make_uint4(0u, 0u, 0u, 0u);
            row += drow;
            g += dg;
            if (g >= G) { g -= G; ++row; }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const __half2 *h = reinterpret_cast<const __half2 *>(&v[u]);
            m = __hmax2(m, __hmax2(__hmax2(__habs2(h[0]), __habs2(h[1])), __hmax2(__habs2(h[2]), __habs2(h[3]))));
        }
    }
    __shared__ float s_max[kThreads / 32];
    const float mw = warp_max(fmaxf(__low2float(m), __high2float(m)));
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = mw;
    __syncthreads();
    if (threadIdx.x == 0) {
        float mx = s_max[0];
        for (int w = 1; w < kThreads / 32; ++w) mx = fmaxf(mx, s_max[w]);
        partial[blockIdx.x] = mx;
    }
}

// kShared: the cluster form, channel maxima from the tiles themselves; else scales from `partial` (per tensor) or from
// a.colmax_bits (per channel).
template <bool kShared, int kT>
__global__ void __launch_bounds__(kT) k_quant_weight(const QuantWeightArgs a, int kt, const float *partial,
                                                     int n_partial) {
    constexpr int kWarps = kT / 32;
    extern __shared__ __align__(16) uint8_t tile[];
    __shared__ float s_part[kWarps][kCols];
    __shared__ float s_colmax[kCols];  // this CTA's maxima, read by the other CTAs of the cluster
    __shared__ float s_scale[kCols];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int n0 = blockIdx.x * kCols, k0 = blockIdx.y * kt;
    const float qf = (float)a.qmax;
    const int c8 = t & 7;
    const bool col_ok = n0 + c8 * 8 < a.N;  // N % 8 == 0: a chunk is entirely inside or outside
    const __half *src = a.W + (size_t)k0 * a.ldw + n0 + c8 * 8;
    // (no early trigger here: a layer kernel behind this one reads W_q ahead of its own wait)
    if constexpr (kShared) asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int r = t >> 3; r < kt; r += kT / 8) {
        const bool ok = col_ok && k0 + r < a.K;
        cp_async16(tile + tile_offset(r, c8), ok ? src + (size_t)r * a.ldw : a.W, ok);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if constexpr (kShared) {
        __half2 m[4];
        m[0] = m[1] = m[2] = m[3] = __float2half2_rn(0.f);
        for (int r = t >> 3; r < kt; r += kT / 8) {  // the chunks this thread has copied itself
            const uint4 v = *reinterpret_cast<const uint4 *>(tile + tile_offset(r, c8));
            const __half2 *h = reinterpret_cast<const __half2 *>(&v);
#pragma unroll
            for (int i = 0; i < 4; ++i) m[i] = __hmax2(m[i], __habs2(h[i]));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float lo = __low2float(m[i]), hi = __high2float(m[i]);
#pragma unroll
            for (int o = 8; o < 32; o <<= 1) {
                lo = fmaxf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
            }
            if (lane < 8) *reinterpret_cast<float2 *>(&s_part[warp][lane * 8 + 2 * i]) = make_float2(lo, hi);
        }
        __syncthreads();
        if (t < kCols) {
            float mx = s_part[0][t];
#pragma unroll
            for (int w = 1; w < kWarps; ++w) mx = fmaxf(mx, s_part[w][t]);
            s_colmax[t] = mx;
        }
        cluster_sync_all();
        if (t < kCols) {
            float mx = 0.0f;
#pragma unroll
            for (int r = 0; r < (int)gridDim.y; ++r) {  // the cluster is the whole K range
                float v;
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(map_to_cta(smem_u32(&s_colmax[t]), r)));
                mx = fmaxf(mx, v);
            }
            const float s = mx > 0.0f ? __fdiv_rn(mx, qf) : 1.0f;
            s_scale[t] = s;
            if (blockIdx.y == 0 && n0 + t < a.N) a.s_w[n0 + t] = s;
        }
        // the other CTAs' maxima have been read; nobody leaves before everybody has (waited for at the end)
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        __syncthreads();
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (a.per_channel) {
            if (t < kCols) {
                const float cm = n0 + t < a.N ? __uint_as_float(a.colmax_bits[n0 + t]) : 0.0f;
                const float s = cm > 0.0f ? __fdiv_rn(cm, qf) : 1.0f;
                s_scale[t] = s;
                if (blockIdx.y == 0 && n0 + t < a.N) a.s_w[n0 + t] = s;
            }
        } else {
            float mx = 0.0f;
            for (int i = t; i < n_partial; i += kT) mx = fmaxf(mx, __ldcg(partial + i));
            mx = warp_max(mx);
            if (lane == 0) s_part[0][warp] = mx;
            __syncthreads();
            if (t < kCols) {
                mx = s_part[0][0];
#pragma unroll
                for (int w = 1; w < kWarps; ++w) mx = fmaxf(mx, s_part[0][w]);
                const float s = mx > 0.0f ? __fdiv_rn(mx, qf) : 1.0f;
                s_scale[t] = s;
                if (blockIdx.x == 0 && blockIdx.y == 0 && t == 0) a.s_w[0] = s;
            }
        }
        __syncthreads();
    }
    // A lane takes 16 input channels of two neighbouring output channels: warp = 4 column pairs of one chunk x 8 groups.
    const int chunk = warp & 7, pair = lane >> 3, n = n0 + chunk * 8 + pair * 2;
    const float s0 = s_scale[chunk * 8 + pair * 2], s1 = s_scale[chunk * 8 + pair * 2 + 1];
    const uint64_t inv2 = pack2(__frcp_rn(s0), __frcp_rn(s1)), neg_s2 = pack2(-s0, -s1);
    const bool wide = (a.ld_q & 15) == 0;
    for (int row0 = (lane & 7) * 16 + (warp >> 3) * 128; row0 < kt; row0 += 16 * kWarps) {
        uint32_t w0[4], w1[4];
        const uint8_t *p = tile + tile_offset(row0, chunk) + pair * 4;  // the 16 rows share one swizzle term
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t b0[4], b1[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(p + (q * 4 + i) * 128));
                const uint64_t c = quotient2(pack2(f.x, f.y), inv2, neg_s2);
                b0[i] = (uint32_t)c;
                b1[i] = (uint32_t)(c >> 32);
            }
            w0[q] = __byte_perm(__byte_perm(b0[0], b0[1], 0x0040), __byte_perm(b0[2], b0[3], 0x0040), 0x5410);
            w1[q] = __byte_perm(__byte_perm(b1[0], b1[1], 0x0040), __byte_perm(b1[2], b1[3], 0x0040), 0x5410);
        }
        const uint4 c0 = make_uint4(w0[0], w0[1], w0[2], w0[3]), c1 = make_uint4(w1[0], w1[1], w1[2], w1[3]);
        const int k = k0 + row0;
        if (n >= a.N || k >= a.K) continue;  // N is even: both columns are inside or outside
        int8_t *q0 = a.w_q + (size_t)n * a.ld_q + k, *q1 = q0 + a.ld_q;
        if (wide && k + 16 <= a.K) {
            *reinterpret_cast<uint4 *>(q0) = c0;
            *reinterpret_cast<uint4 *>(q1) = c1;
        } else {
            const uint32_t v0[4] = {c0.x, c0.y, c0.z, c0.w}, v1[4] = {c1.x, c1.y, c1.z, c1.w};
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                if (k + i < a.K) {
                    q0[i] = (int8_t)(v0[i >> 2] >> (8 * (i & 3)));
                    q1[i] = (int8_t)(v1[i >> 2] >> (8 * (i & 3)));
                }
            }
        }
    }
    if constexpr (kShared) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

cudaError_t set_smem(const void *fn, PerDevice<int> &done, int bytes) {
    const int dev = current_device();
    if (dev < 0) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(device_mutex());
    if (done.have[dev]) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.have[dev] = true;
    return e;
}

}  // namespace

bool quant_weight_in_cluster(const QuantWeightArgs &a) { return a.per_channel && a.K <= kCluster * kMaxTileRows; }

cudaError_t launch_quant_weight(const QuantWeightArgs &a, float *partial, cudaStream_t s) {
    const int stripes = (a.N + kCols - 1) / kCols, sms = num_sms();
    cudaLaunchConfig_t cfg{};
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (quant_weight_in_cluster(a)) {
        // The kernel is a chain of latencies (copies in, maxima, cluster exchange, codes out), so what counts is that all
        // CTAs are resident at once and that an SM has some 16 warps: the smallest cluster that still gives two CTAs per SM
        // (and a tile of at most 320 rows, so that four fit an SM), else eight CTAs; with fewer than two CTAs per SM, 16 warps
        // each.
        int c = 1;
        while (c < kCluster && (stripes * c < 2 * sms || a.K > c * 320)) c *= 2;
        const int kt = ((a.K + c - 1) / c + 15) & ~15;
        const bool few = stripes * c < 2 * sms;
        static PerDevice<int> done, done_few;
        const void *fn = few ? reinterpret_cast<const void *>(k_quant_weight<true, 2 * kThreads>)
                             : reinterpret_cast<const void *>(k_quant_weight<true, kThreads>);
        cudaError_t e = set_smem(fn, few ? done_few : done, kMaxTileRows * 128);
        if (e != cudaSuccess) return e;
        cfg.gridDim = dim3(stripes, c);
        cfg.blockDim = dim3(few ? 2 * kThreads : kThreads);
        cfg.dynamicSmemBytes = (size_t)kt * 128;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = c; attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
        return few ? cudaLaunchKernelEx(&cfg, k_quant_weight<true, 2 * kThreads>, a, kt, (const float *)nullptr, 0)
                   : cudaLaunchKernelEx(&cfg, k_quant_weight<true, kThreads>, a, kt, (const float *)nullptr, 0);
    }
    int n_partial = 0;
    if (!a.per_channel) {
        const long long chunks = (long long)a.K * (a.N >> 3);
        n_partial = 4 * sms;
        if (n_partial > kQuantWeightPartials) n_partial = kQuantWeightPartials;
        const long long most = (chunks + 4 * kThreads - 1) / (4 * kThreads);  // at least four loads per thread
        if (n_partial > most) n_partial = (int)most;
        cfg.gridDim = dim3(n_partial);
        cfg.blockDim = dim3(kThreads);
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k_weight_absmax, a, partial);
        if (e != cudaSuccess) return e;
    }
    cfg.blockDim = dim3(kThreads);
    cfg.gridDim = dim3(stripes, (a.K + kTileRows - 1) / kTileRows);
    cfg.dynamicSmemBytes = kTileRows * 128;
    cfg.numAttrs = a.per_channel ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, k_quant_weight<false, kThreads>, a, kTileRows, (const float *)partial, n_partial);
}

}  // namespace muxq
