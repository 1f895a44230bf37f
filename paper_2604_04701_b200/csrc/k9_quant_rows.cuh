// k_quant_rows: redistribution and quantization of token rows held in registers (k9_prep_rows.cu has the overview).
#pragma once
#include "k9_prep_rows.cuh"

namespace muxq {
namespace prep_rows {

namespace {

// ---------------------------------------------------------------- what the channel maxima say
struct ChannelFacts {
    float s;            // Eq. 1, per tensor
    int r_true, r;      // outlier channels; those listed
    uint32_t ticket;    // (thread 0) how many CTAs had read the maxima before this one
    bool marked;        // nothing else holds: an earlier call on the workspace timed out
};

// Every CTA derives O (ascending, into s_oidx) and the per-tensor scale from the K maxima for itself, CTA 0 publishes them.  The ticket comes back while the rows are at work: release_maxima() looks at it behind them.  on_group(g, flags) is called for every group of 8 channels
// (bit j of flags: channel 8g + j is in O).
template <class OnGroup>
__device__ __forceinline__ ChannelFacts channel_facts(const PrepArgs &a, uint16_t *s_oidx, OnGroup on_group) {
    __shared__ uint32_t s_max[kWarps];
    __shared__ int s_cnt[2][kWarps];
    __shared__ uint32_t s_marked;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int K = a.K, G = K >> 3;
    const float down = __int_as_float((127 - a.exp_factor) << 23);  // 2^-e
    const float qf = (float)a.qmax;
    float bmax = 0.0f;
    uint32_t gm[2] = {0u, 0u};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int g = t + i * kT;
        if (g < G) {
            const uint4 x = __ldcg(reinterpret_cast<const uint4 *>(a.colmax_rep) + 2 * g);
            const uint4 y = __ldcg(reinterpret_cast<const uint4 *>(a.colmax_rep) + 2 * g + 1);
            const float cm[8] = {__uint_as_float(x.x), __uint_as_float(x.y), __uint_as_float(x.z), __uint_as_float(x.w),
                                 __uint_as_float(y.x), __uint_as_float(y.y), __uint_as_float(y.z), __uint_as_float(y.w)};
            if (g == 0) s_marked = x.x == kMarkedMaximum;
            if (blockIdx.x == 0) {
                reinterpret_cast<uint4 *>(a.colmax_bits)[2 * g] = x;
                reinterpret_cast<uint4 *>(a.colmax_bits)[2 * g + 1] = y;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bool flagged = cm[j] > a.tau;  // strict (Section III-C)
                gm[i] |= flagged ? 1u << j : 0u;
                bmax = fmaxf(bmax, flagged ? cm[j] * down : cm[j]);  // power-of-two scaling: exact
            }
            on_group(g, gm[i]);
        }
    }
    const uint32_t wmax = __reduce_max_sync(0xffffffffu, __float_as_uint(bmax));
    int incl[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        incl[i] = __popc(gm[i]);
        if (__any_sync(0xffffffffu, gm[i] != 0u)) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int n = __shfl_up_sync(0xffffffffu, incl[i], o);
                if (lane >= o) incl[i] += n;
            }
        }
        if (lane == 31) s_cnt[i][warp] = incl[i];
    }
    if (lane == 0) s_max[warp] = wmax;
    __syncthreads();
    const uint32_t mx = __reduce_max_sync(0xffffffffu, s_max[lane & (kWarps - 1)]);
    ChannelFacts f;
    f.marked = s_marked != 0u;
    if (f.marked) return f;
    f.ticket = 0;
    f.s = mx ? __fdiv_rn(__uint_as_float(mx), qf) : 1.0f;
    // groups t and t + kT stand in ascending order: all of the first round come before the second
    const int n0 = lane < kWarps ? s_cnt[0][lane] : 0, n1 = lane < kWarps ? s_cnt[1][lane] : 0;
    const int total0 = __reduce_add_sync(0xffffffffu, n0);
    f.r_true = total0 + __reduce_add_sync(0xffffffffu, n1);
    f.r = min(f.r_true, a.cap);
    if (__any_sync(0xffffffffu, (gm[0] | gm[1]) != 0u)) {
        int base = __reduce_add_sync(0xffffffffu, lane < warp ? n0 : 0);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            int pos = base + incl[i] - __popc(gm[i]);
            for (uint32_t mm = gm[i]; mm; mm &= mm - 1, ++pos) {
                const int ch = 8 * (t + i * kT) + __ffs(mm) - 1;
                if (pos < a.cap) {
                    s_oidx[pos] = (uint16_t)ch;
                    if (blockIdx.x == 0) a.outlier_idx[pos] = ch;
                }
            }
            base = total0 + __reduce_add_sync(0xffffffffu, lane < warp ? n1 : 0);
        }
    }
    if (t == 0) {
        if (blockIdx.x == 0) {
            a.ctrl->s_x = f.s;
            a.ctrl->inv_s_x = __frcp_rn(f.s);
            a.ctrl->n_outliers = f.r_true;
            if (f.r_true > a.cap && a.dev_status) atomicMax(a.dev_status, kStatusCapacity);
        }
        f.ticket = atomicAdd(&a.ctrl->readers, 1u);  // (behind the barrier: the maxima have been read)
    }
    __syncthreads();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    return f;
}

// The CTA with the last ticket knows that every CTA has read the maxima: zero again for the next call.
__device__ __forceinline__ void release_maxima(const PrepArgs &a, const ChannelFacts &f) {
    if (threadIdx.x >= 32 || __shfl_sync(0xffffffffu, f.ticket, 0) != gridDim.x - 1) return;
    for (int i = threadIdx.x; i < (a.K >> 2); i += 32) reinterpret_cast<uint4 *>(a.colmax_rep)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x == 0) a.ctrl->readers = 0u;
}

// What else the GEMM wants, spread over the grid: the memory it expects cleared, the zeros behind the Aux codes of a row (it
// reads Aux columns in steps of 32), and W_aux[n, c*j + i] = W_q[n, O_j], a 4-byte word per thread.  request() asks the bytes of
// a thread's first word into L2 ahead of the rows, gather() moves them behind.
struct AuxWork {
    int c, used, words, w_total, wi;
    __device__ __forceinline__ AuxWork(const PrepArgs &a, int r) {
        c = (1 << a.exp_factor) - 1;
        used = c * r;
        words = ((used + 31) & ~31) >> 2;
        w_total = a.w_aux ? a.N * words : 0;
        // (short inputs leave the last warps without rows)
        wi = ((kWarps - 1 - (int)(threadIdx.x >> 5)) * (int)gridDim.x + (int)blockIdx.x) * 32 + (int)(threadIdx.x & 31);
    }
    __device__ __forceinline__ void request(const PrepArgs &a, const uint16_t *s_oidx) const {
        // (the GEMM before this call has finished with the memory cleared here, the one behind it waits for this grid)
        for (uint32_t i = blockIdx.x * kT + threadIdx.x; i < (a.zero_bytes >> 4); i += gridDim.x * kT)
            static_cast<uint4 *>(a.zero)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (a.aux_q && used < 4 * words)
            for (int m = wi; m < a.M; m += gridDim.x * kT)
                for (int b = used; b < 4 * words; ++b) a.aux_q[(size_t)m * a.ld_aux + b] = 0;
        if (wi < w_total) {
            const int n = wi / words, col = 4 * (wi - n * words);
            if (col < used) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.w_q + (size_t)n * a.ldw + s_oidx[col / c]));
            if (col + 3 < used) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.w_q + (size_t)n * a.ldw + s_oidx[(col + 3) / c]));
        }
    }
    __device__ __forceinline__ void gather(const PrepArgs &a, const uint16_t *s_oidx) const {
        for (int i = wi; i < w_total; i += gridDim.x * kT) {
            const int n = i / words, col = 4 * (i - n * words);
            const int8_t *wr = a.w_q + (size_t)n * a.ldw;
            uint32_t packed = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (col + b < used) packed |= (uint32_t)(uint8_t)wr[s_oidx[(col + b) / c]] << (8 * b);
            *reinterpret_cast<uint32_t *>(a.w_aux + (size_t)n * a.ld_waux + col) = packed;
        }
    }
};

// c copies of a code into the Aux columns of one outlier channel (Eq. 5, shared scale)
__device__ __forceinline__ void store_aux(int8_t *p, int c, int8_t code) {
    p[0] = code;
    if (c > 1) p[1] = code, p[2] = code;
    if (c > 3) p[3] = code, p[4] = code, p[5] = code, p[6] = code;
}

// ---------------------------------------------------------------- quantization
// kW warps share a token row, kC 16-byte chunks of it per lane: the row is in registers, X is read once here.  Where a warp's
// chunks hold an outlier channel they are multiplied by the channel factors, 1 or 2^-e (Eq. 4), in fp16 as they are taken up: one
// shared load and four instructions per chunk, whatever the number of outlier channels.  The codes also go through shared
// memory, from where one lane per outlier channel copies its code to the Aux columns (Eq. 5, shared scale).
//
// An fp16 product with 2^-e is exact unless it is below 2^-14, and then off by at most 2^-25.  With a scale of at least 2^-11
// such a value has code 0 either way, and a maximum of at least 2^-14 is exact; a row with a smaller scale takes the true
// division throughout.
constexpr float kSafe = 1.0f / 2048.0f;

template <bool kPerToken, int kW, int kC>
__global__ void __launch_bounds__(kT, 2) k_quant_rows(const PrepArgs a) {
    constexpr int kGroups = kWarps / kW;
    constexpr int kLanes = 32 * kW;
    constexpr int kFull = kC == 8 ? 5 : kC - 1;  // chunk columns that every lane has
    // channel factors [K] fp16 | codes of a row's chunks [kWarps][kC * 32] uint2 | O [cap] u16
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_any;  // bit w: warp w of a row holds an outlier channel
    __shared__ float s_rowmax[2][kWarps];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int K = a.K, G = K >> 3, M = a.M;
    const int group = warp / kW, l = t - group * kLanes;  // lane within the row's group
    uint4 *s_mul = reinterpret_cast<uint4 *>(smem);
    uint2 *s_code = reinterpret_cast<uint2 *>(smem + 2 * (size_t)K);
    uint16_t *s_oidx = reinterpret_cast<uint16_t *>(s_code + kWarps * kC * 32);
    const uint32_t down16 = (uint32_t)(15 - a.exp_factor) << 10;  // 2^-e in fp16
    const float qf = (float)a.qmax;
    const int stride = gridDim.x * kGroups;

    // rows in descending order; the first one is requested before anything else
    int row = M - 1 - (group * gridDim.x + blockIdx.x);
    const __half *xp = a.X + (ptrdiff_t)row * a.ldx;  // (not dereferenced for row < 0)
    const ptrdiff_t xstep = (ptrdiff_t)stride * a.ldx;
    const uint64_t pol = l2_policy((size_t)a.M * a.K * 2 > kLongBytes);
    uint4 v[kC];
#pragma unroll
    for (int i = 0; i < kC; ++i) {
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        if (row >= 0 && (i < kFull || l + i * kLanes < G)) v[i] = ld_nc_v4(reinterpret_cast<const uint4 *>(xp) + l + i * kLanes, pol);
    }
    if (t == 0) s_any = 0u;
    __syncthreads();  // (free: the maxima are not there yet)
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const ChannelFacts f = channel_facts(a, s_oidx, [&](int g, uint32_t flags) {
        uint32_t mul[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            mul[j] = ((flags >> (2 * j)) & 1u ? down16 : 0x3C00u) | ((flags >> (2 * j + 1)) & 1u ? down16 : 0x3C00u) << 16;
        s_mul[g] = make_uint4(mul[0], mul[1], mul[2], mul[3]);
        if (flags) atomicOr(&s_any, 1u << ((g / 32) % kW));
    });
    if (f.marked) {  // nothing is computed on half-merged maxima, and nothing is cleared, until muxq_workspace_init
        if (blockIdx.x == 0 && t == 0 && a.dev_status) atomicMax(a.dev_status, kStatusTimeout);
        return;
    }
    const int r = f.r;
    const AuxWork aw(a, r);
    aw.request(a, s_oidx);

    // ------------------------------------------------------------ rows
    const bool scaled = (s_any >> (warp % kW)) & 1u;  // this warp has chunks with an outlier channel
    uint2 *const codes = s_code + warp * (kC * 32) + lane;
    // Aux: lane j looks after O_j where the channel's chunk is this warp's (beyond 32 of them one lane after several)
    auto code_of = [&](int j) -> const int8_t * {
        const int ch = s_oidx[j], g = ch >> 3;
        return (g >> 5) % kW == warp % kW ? reinterpret_cast<const int8_t *>(s_code + warp * (kC * 32) + g / kLanes * 32 + (g & 31)) + (ch & 7)
                                          : nullptr;
    };
    const bool mirror = a.aux_q && scaled;
    const int8_t *const code0 = mirror && lane < r ? code_of(lane) : nullptr;
    const int aux0 = aw.c * lane;
    float sr = f.s, inv = __frcp_rn(sr);
    bool tiny = !kPerToken && f.r_true && sr < kSafe;
    uint32_t flip = 0;
    for (; row >= 0; row -= stride) {
        // Eq. 4: Body
        if (scaled)
#pragma unroll
            for (int i = 0; i < kC; ++i) {
                const uint4 k4 = s_mul[i < kFull ? l + i * kLanes : min(l + i * kLanes, G - 1)];
                const __half2 *k = reinterpret_cast<const __half2 *>(&k4);
                __half2 *h = reinterpret_cast<__half2 *>(&v[i]);
#pragma unroll
                for (int j = 0; j < 4; ++j) h[j] = __hmul2(h[j], k[j]);
            }
        if (kPerToken) {
            __half2 hm = __float2half2_rn(0.f);
#pragma unroll
            for (int i = 0; i < kC; ++i) {
                const __half2 *h = reinterpret_cast<const __half2 *>(&v[i]);
                hm = __hmax2(hm, __hmax2(__hmax2(__habs2(h[0]), __habs2(h[1])), __hmax2(__habs2(h[2]), __habs2(h[3]))));
            }
            float om = fmaxf(__low2float(hm), __high2float(hm));
            for (tiny = false;;) {
                uint32_t rm = __reduce_max_sync(0xffffffffu, __float_as_uint(om));
                if (kW > 1) {  // one barrier per row: the other buffer is written next
                    if (lane == 0) s_rowmax[flip][warp] = __uint_as_float(rm);
                    asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(kLanes) : "memory");
#pragma unroll
                    for (int w = 0; w < kW; ++w) rm = max(rm, __float_as_uint(s_rowmax[flip][group * kW + w]));
                    flip ^= 1u;
                }
                om = __uint_as_float(rm);
                if (tiny || !f.r_true || om >= qf * kSafe) break;
                tiny = true;  // (the same for all warps of the row)
                om = 0.0f;
#pragma unroll 1
                for (int ch = 8 * l; ch < K; ch += (ch & 7) == 7 ? 8 * kLanes - 7 : 1)
                    om = fmaxf(om, fabsf(__half2float(xp[ch]) * __half2float(reinterpret_cast<const __half *>(s_mul)[ch])));
            }
            sr = om > 0.0f ? __fdiv_rn(om, qf) : 1.0f;
            if (l == 0) a.s_x_rows[row] = sr;
            inv = __frcp_rn(sr);
        }
        const uint64_t inv2 = pack2(inv, inv), neg_s2 = pack2(-sr, -sr);
        uint2 *q = reinterpret_cast<uint2 *>(a.body_q + (ptrdiff_t)row * a.ld_q);
        const __half *const xrow = xp;
        xp -= xstep;
        const bool more = row >= stride;
#pragma unroll
        for (int i = 0; i < kC; ++i) {
            const uint2 code = quotient8(v[i], inv2, neg_s2);
            if (i < kFull || l + i * kLanes < G) q[l + i * kLanes] = code;
            ld_nc_v4_if(v[i], reinterpret_cast<const uint4 *>(xp) + l + i * kLanes, more && (i < kFull || l + i * kLanes < G), pol);
            codes[32 * i] = code;
        }
        if (tiny) {
#pragma unroll 1
            for (int ch = 8 * l; ch < K; ch += (ch & 7) == 7 ? 8 * kLanes - 7 : 1) {
                const float y = __half2float(xrow[ch]) * __half2float(reinterpret_cast<const __half *>(s_mul)[ch]);
                const int8_t code = (int8_t)quant_exact(y, sr, qf);
                reinterpret_cast<int8_t *>(q)[ch] = code;
                reinterpret_cast<int8_t *>(codes + 32 * ((ch >> 3) / kLanes))[ch & 7] = code;
            }
        }
        if (mirror) {
            __syncwarp();
            int8_t *aux = a.aux_q + (ptrdiff_t)row * a.ld_aux;
            if (code0) store_aux(aux + aux0, aw.c, *code0);
            for (int j = lane + 32; j < r; j += 32)
                if (const int8_t *p = code_of(j)) store_aux(aux + aw.c * j, aw.c, *p);
            __syncwarp();
        }
    }
    release_maxima(a, f);
    aw.gather(a, s_oidx);
}

}  // namespace

template <bool kPerToken>
cudaError_t launch_rows(const PrepArgs &a, cudaLaunchConfig_t &cfg, int sms) {
    // warps per row: at most five chunks a lane (eight beyond K = 5120); chunks per lane: as few as hold the row, an empty
    // chunk column costs what a full one does
    const int G = a.K >> 3;
    const int w = G <= 160 ? 1 : G <= 320 ? 2 : 4, chunks = (G + 32 * w - 1) / (32 * w);
    // two CTAs per SM; short inputs: at least four busy warps per CTA, but 64 CTAs for the gather of W_aux (whole layers with N =
    // 768, without that line -> with it, us: 17 x 1280 12.6 -> 10.4, 64 x 1280 11.0 -> 10.5; 148 CTAs: 10.9)
    long long ctas = ((long long)a.M * w + 3) / 4;
    if (ctas < 64) ctas = 64;
    if (ctas > 2 * sms) ctas = 2 * sms;
    cfg.gridDim = dim3((unsigned)ctas);
    using Fn = void (*)(PrepArgs);
    static const Fn fns[] = {
        k_quant_rows<kPerToken, 1, 1>, k_quant_rows<kPerToken, 1, 2>, k_quant_rows<kPerToken, 1, 3>, k_quant_rows<kPerToken, 1, 4>,
        k_quant_rows<kPerToken, 1, 5>, k_quant_rows<kPerToken, 2, 3>, k_quant_rows<kPerToken, 2, 4>, k_quant_rows<kPerToken, 2, 5>,
        k_quant_rows<kPerToken, 4, 3>, k_quant_rows<kPerToken, 4, 4>, k_quant_rows<kPerToken, 4, 5>, k_quant_rows<kPerToken, 4, 8>};
    const int kc = chunks > 5 ? 8 : chunks;  // of the instantiation
    const int pick = w == 1 ? kc - 1 : (w == 2 ? 5 : 8) + (kc == 8 ? 3 : kc - 3);
    auto smem = [](int K, int columns, int cap) { return 2 * K + kWarps * columns * 256 + 2 * cap; };
    static PerDevice<int> done[sizeof fns / sizeof *fns];
    const int dev = current_device();
    if (dev < 0) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(device_mutex());
        if (!done[pick].have[dev]) {  // (only what is about to run: the call makes the driver load the kernel)
            const cudaError_t e = cudaFuncSetAttribute(fns[pick], cudaFuncAttributeMaxDynamicSharedMemorySize, smem(kPrepMaxK, 8, kMaxOutlierCap));
            if (e != cudaSuccess) return e;
            done[pick].have[dev] = true;
        }
    }
    cfg.dynamicSmemBytes = smem(a.K, kc, a.cap);
    return cudaLaunchKernelEx(&cfg, fns[pick], a);
}

}  // namespace prep_rows
}  // namespace muxq
