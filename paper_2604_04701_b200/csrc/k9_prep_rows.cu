// Activation preparation for muxq_linear as two launches: per-channel abs-max (Section III-C), then redistribution and
// quantization of Eq. 4-5 and Eq. 1.
//
//   k_channel_max   a CTA reads a stripe of up to 256 channels (a warp: 512 contiguous bytes of a token row, eight rows in
//                   flight per lane) and merges its maxima with integer atomicMax on the bit patterns (maxima of
//                   non-negative floats: exact, order independent).
//   k_quant_rows    a group of one, two or four warps holds a token row in registers, so X is read once here, whatever the
//                   scale: per token the row's maximum of Body comes from the registers; per tensor the scale comes from
//                   the channel maxima.  Every CTA derives O and the per-tensor scale from the K maxima for itself while
//                   its first rows are on their way.
//
// Both are launched with programmatic stream serialization: k_channel_max waits for the work before it and then lets the
// second kernel start, which may therefore read X at once and waits (for the maxima) only after that; the GEMM starts
// behind the second in the same way.  The boundary between two launches costs less than a cooperative launch and its
// grid-wide barrier (k12_prep.cu), and nothing is held in shared memory.  Rows are visited in ascending order by the first
// kernel and in descending order by the second: the rows read last are still in L2 when X is larger than that.
//
// Bound: short inputs by latency (64 x 1280: 3 us per kernel beyond an empty launch, from the maxima to the first code), long
// ones by HBM in the first kernel (16384 x 5120: 5.7 TB/s alone; in a layer it shares HBM with the write-back of the last GEMM's
// Y) and in the second by L2 and HBM together with some 65 warp instructions per 256 channels (18944 x 1280: 12 us without
// outlier channels, 15.5 us with any number of them; with a test and a division for values next to a tie, and outlier channels
// done over one by one, 24 us and more).  Whole layers with N = 768, this form before -> now, us: per tensor 8192 x 1280 26.3 -> 24.3; per
// token 8192 x 1280 29.5 -> 25.1; alone with N = 128: 8192 x 1280 with 32 outlier channels 26.2 -> 20.0, 8192 x 5120 69.1 -> 57.3,
// 16384 x 1280 36.5 -> 30.4.
//
// The accumulators are zero between calls (the same contract as the cooperative kernel): the CTA of k_quant_rows that takes
// the last ticket knows that every CTA has read them and clears them.
#include "kernels.h"
#include "quant.cuh"

namespace muxq {

namespace {

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

__global__ void __launch_bounds__(kT, 2) k_channel_max(const PrepArgs a, int stripes, int width, int slices, int first_rows) {
    __shared__ uint4 s_part[kWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int stripe = blockIdx.x % stripes, slice = blockIdx.x / stripes;
    const int g = stripe * width + lane, G = a.K >> 3;
    const bool on = lane < width && g < G;
    const int step = slices * kWarps;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // behind the wait: the dependent may read X at once
    __half2 m[4];
    m[0] = m[1] = m[2] = m[3] = __float2half2_rn(0.f);
    if (on) {
        const __half *p = a.X + (size_t)g * 8;
        auto take = [&](const uint4 &v) {
            const __half2 *h = reinterpret_cast<const __half2 *>(&v);
#pragma unroll
            for (int i = 0; i < 4; ++i) m[i] = __hmax2(m[i], __habs2(h[i]));
        };
        int row = slice * kWarps + warp;
        for (; row + 7 * step < a.M; row += 8 * step) {
            uint4 v[8];
            const uint64_t pol = l2_policy(row < first_rows);
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = ld_v4(p + (size_t)(row + u * step) * a.ldx, pol);
#pragma unroll
            for (int u = 0; u < 8; ++u) take(v[u]);
        }
        if (row < a.M) {  // up to seven more
            uint4 v[7];
            const uint64_t pol = l2_policy(row < first_rows);
#pragma unroll
            for (int u = 0; u < 7; ++u) {
                v[u] = make_uint4(0u, 0u, 0u, 0u);
                if (row + u * step < a.M) v[u] = ld_v4(p + (size_t)(row + u * step) * a.ldx, pol);
            }
#pragma unroll
            for (int u = 0; u < 7; ++u) take(v[u]);
        }
    }
    s_part[warp][lane] = *reinterpret_cast<const uint4 *>(m);
    __syncthreads();
    if (threadIdx.x < 128) {  // two channels per thread
        const int l = threadIdx.x >> 2, i = threadIdx.x & 3;
        const int gg = stripe * width + l;
        if (l < width && gg < G) {
            __half2 x = __float2half2_rn(0.f);
#pragma unroll
            for (int w = 0; w < kWarps; ++w) x = __hmax2(x, reinterpret_cast<const __half2 *>(&s_part[w][l])[i]);
            const uint32_t lo = __float_as_uint(__low2float(x)), hi = __float_as_uint(__high2float(x));
            uint32_t *acc = a.colmax_rep + gg * 8 + 2 * i;
            if (lo) atomicMax(acc, lo);
            if (hi) atomicMax(acc + 1, hi);
        }
    }
}

// ---------------------------------------------------------------- what the channel maxima say
struct ChannelFacts {
    float s;            // Eq. 1, per tensor
    int r_true, r;      // outlier channels; those listed
    uint32_t ticket;    // (thread 0) how many CTAs had read the maxima before this one
};

// Every CTA derives O (ascending, into s_oidx) and the per-tensor scale from the K maxima for itself, CTA 0 publishes them (unless
// the workspace is marked: an earlier call timed out and left half-merged maxima).  The ticket comes back while the rows are at work: release_maxima() looks at it behind them.  on_group(g, flags) is called for every group of 8 channels
// (bit j of flags: channel 8g + j is in O).
template <class OnGroup>
__device__ __forceinline__ ChannelFacts channel_facts(const PrepArgs &a, bool marked, uint16_t *s_oidx, OnGroup on_group) {
    __shared__ uint32_t s_max[kWarps];
    __shared__ int s_cnt[2][kWarps];
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
            if (blockIdx.x == 0 && !marked) {
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
                    if (blockIdx.x == 0 && !marked) a.outlier_idx[pos] = ch;
                }
            }
            base = total0 + __reduce_add_sync(0xffffffffu, lane < warp ? n1 : 0);
        }
    }
    if (t == 0 && !marked) {
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

    // (on its way together with the maxima)
    const bool marked = (__ldcg(&a.ctrl->arrived) & kPrepPoisonBit) != 0u;
    const ChannelFacts f = channel_facts(a, marked, s_oidx, [&](int g, uint32_t flags) {
        uint32_t mul[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            mul[j] = ((flags >> (2 * j)) & 1u ? down16 : 0x3C00u) | ((flags >> (2 * j + 1)) & 1u ? down16 : 0x3C00u) << 16;
        s_mul[g] = make_uint4(mul[0], mul[1], mul[2], mul[3]);
        if (flags) atomicOr(&s_any, 1u << ((g / 32) % kW));
    });
    if (marked) {  // nothing is computed on half-merged maxima, and nothing is cleared, until muxq_workspace_init
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
    static PerDevice<int> done;
    const int dev = current_device();
    if (dev < 0) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(device_mutex());
        if (!done.have[dev]) {
            for (const Fn f : fns) {
                const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem(kPrepMaxK, 8, kMaxOutlierCap));
                if (e != cudaSuccess) return e;
            }
            done.have[dev] = true;
        }
    }
    cfg.dynamicSmemBytes = smem(a.K, kc, a.cap);
    return cudaLaunchKernelEx(&cfg, fns[pick], a);
}

}  // namespace

// The cooperative kernel keeps the own-scale reading of Aux, and long narrow inputs under one scale, whose rows mostly fit its
// shared memory: it reads X once.  Whole layers with N = 768, cooperative / these, us: per tensor 2048 x 512 13.8 / 13.1, 4096 x
// 512 14.5 / 14.7, 4096 x 1280 17.0 / 15.7, 8192 x 768 18.1 / 18.3, 8192 x 1536 25.6 / 25.7, 8192 x 2048 33.0 / 30.0, 16384 x 1280
// 37.3 / 38.6, 16384 x 2048 55.3 / 55.2; per token 2048 x 400 15.2 / 13.7, 32768 x 400 49.5 / 48.0, 16384 x 1280 47.5 / 40.4.
bool prep_rows_preferred(const PrepArgs &a) {
    if (a.aux_own || a.K > kPrepMaxK) return false;
    return a.per_token || a.K >= 2048 || a.M <= (a.K > 512 ? 6144 : 3072);
}

cudaError_t launch_prep_rows(const PrepArgs &a, cudaStream_t s) {
    const int sms = num_sms();
    if (sms < 1) return cudaErrorInvalidDevice;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // stripes of equal width (at most 32 groups of 8 channels), token rows dealt out to the warps of the CTAs of a stripe
    const int G = a.K >> 3, stripes = (G + 31) / 32, width = (G + stripes - 1) / stripes;
    auto slices_for = [&](int ctas) {
        const int most = (a.M + kWarps - 1) / kWarps;
        int n = ctas / stripes;
        if (n < 1) n = 1;
        return n < most ? n : most;
    };
    cfg.blockDim = dim3(kT);
    const int slices = slices_for(2 * sms);
    cfg.gridDim = dim3(stripes * slices);
    const size_t bytes = (size_t)a.M * a.K * 2;
    const int first_rows = bytes > kLongBytes && bytes > kKeepBytes ? a.M - (int)(kKeepBytes / 2 / a.K) : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_channel_max, a, stripes, width, slices, first_rows);
    if (e != cudaSuccess) return e;
    return a.per_token ? launch_rows<true>(a, cfg, sms) : launch_rows<false>(a, cfg, sms);
}

}  // namespace muxq
