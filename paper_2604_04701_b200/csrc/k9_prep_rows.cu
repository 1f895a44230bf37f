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
// Bound: short inputs by latency (M = 128, K = 768: 1.8 + 4 us), long ones by HBM in the first kernel (16384 x 5120: 5.7
// TB/s alone; in a layer it shares HBM with the write-back of the last GEMM's Y) and by instruction issue (some 80 per 256
// channels) and HBM in the second.  Whole layers with N = 768, cooperative kernel -> these (us): per tensor 64 x 768 12.6
// -> 10.7, 2048 x 1280 16.7 -> 15.5, 2048 x 4096 28.7 -> 23.9, 16384 x 4096 106 -> 98; per token 64 x 768 14.6 -> 11.9,
// 2048 x 1280 19.8 -> 17.3, 8192 x 3072 55.9 -> 51.1, 16384 x 4096 137 -> 113.
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

// 16-byte read-only load as a volatile statement: a batch of them is issued back to back before the first use, whatever the
// register allocator would rather do.
__device__ __forceinline__ uint4 ld_nc_v4(const void *p) {
    uint4 v;
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// Two fp32 operations per instruction (each rounded like the scalar one).
__device__ __forceinline__ uint64_t pack2(float x, float y) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}

// 8 codes by the true division (Eq. 1), out of line: about one chunk in a thousand needs it
// (values, not a reference: an array whose address is taken would live in local memory everywhere)
static __device__ __noinline__ uint2 exact8(uint64_t x0, uint64_t x1, uint64_t x2, uint64_t x3, float s, float qf) {
    const float2 p0 = unpack2(x0), p1 = unpack2(x1), p2 = unpack2(x2), p3 = unpack2(x3);
    const float f[8] = {p0.x, p0.y, p1.x, p1.y, p2.x, p2.y, p3.x, p3.y};
    uint32_t b[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) b[i] = (uint32_t)quant_exact(f[i], s, qf);
    return pack8(b);
}

__global__ void __launch_bounds__(kT, 2) k_channel_max(const PrepArgs a, int stripes, int width, int slices) {
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
        for (int row = slice * kWarps + warp; row < a.M; row += 8 * step) {
            uint4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = ld_nc_v4(p + (size_t)min(row + u * step, a.M - 1) * a.ldx);  // (behind the end: the last row again)
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const __half2 *h = reinterpret_cast<const __half2 *>(&v[u]);
#pragma unroll
                for (int i = 0; i < 4; ++i) m[i] = __hmax2(m[i], __habs2(h[i]));
            }
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

// ---------------------------------------------------------------- quantization
// kW warps share a token row, kC 16-byte chunks of it per lane (kC * kW * 32 * 8 >= K): the row is in registers, the next one
// on its way.  All channels are quantized alike; an outlier channel is then done over by the lane that owns its chunk, as
// Eq. 4 wants it, into Body_q (a byte behind the chunk's own store) and into the Aux columns that mirror it.
constexpr uint16_t kNone = 0xFFFF;

template <bool kPerToken, int kW, int kC>
__global__ void __launch_bounds__(kT, 2) k_quant_rows(const PrepArgs a) {
    constexpr int kGroups = kWarps / kW;
    constexpr int kLanes = 32 * kW;
    // |.| masks of the channels outside O [K] u16 (per token) | O [cap] u16 | next outlier channel of the same lane [cap] u16
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_head[kLanes];  // first outlier channel of lane l's chunks: its place in O
    __shared__ uint32_t s_any[32];       // bit w of s_any[i]: warp w of a row holds an outlier channel in chunk column i
    __shared__ uint32_t s_max[kWarps];
    __shared__ int s_cnt[2][kWarps];
    __shared__ int s_last;
    __shared__ float s_rowmax[2][kWarps];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int K = a.K, G = K >> 3, M = a.M;
    const int group = warp / kW, l = t - group * kLanes;  // lane within the row's group
    uint16_t *s_oidx = reinterpret_cast<uint16_t *>(smem + (kPerToken ? 2 * (size_t)K : 0));
    uint16_t *s_next = s_oidx + a.cap;
    const float down = __int_as_float((127 - a.exp_factor) << 23);  // 2^-e
    const float qf = (float)a.qmax;
    const int c = (1 << a.exp_factor) - 1;
    const int stride = gridDim.x * kGroups;

    // rows in descending order; the first one is requested before anything else
    int row = M - 1 - (group * gridDim.x + blockIdx.x);
    const __half *xp = a.X + (ptrdiff_t)row * a.ldx;  // (not dereferenced for row < 0)
    const ptrdiff_t xstep = (ptrdiff_t)stride * a.ldx;
    const int qstep = stride * a.ld_q;  // (ld_q is K here: at most some 40 M)
    uint4 v[kC];
#pragma unroll
    for (int i = 0; i < kC; ++i) {
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        if (row >= 0 && l + i * kLanes < G) v[i] = ld_nc_v4(reinterpret_cast<const uint4 *>(xp) + l + i * kLanes);
    }
    if (t < 32) s_any[t] = 0u;
    if (t < kLanes) s_head[t] = kNone;
    __syncthreads();  // (free: the maxima are not there yet)
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // ------------------------------------------------------------ scale, O and its owners, from the channel maxima
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
            if (blockIdx.x == 0) {
                reinterpret_cast<uint4 *>(a.colmax_bits)[2 * g] = x;
                reinterpret_cast<uint4 *>(a.colmax_bits)[2 * g + 1] = y;
            }
            uint32_t keep[4];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bool flagged = cm[j] > a.tau;  // strict (Section III-C)
                gm[i] |= flagged ? 1u << j : 0u;
                bmax = fmaxf(bmax, flagged ? cm[j] * down : cm[j]);  // power-of-two scaling: exact
                if (j & 1) keep[j >> 1] |= flagged ? 0u : 0x7FFF0000u;
                else keep[j >> 1] = flagged ? 0u : 0x7FFFu;
            }
            if (kPerToken) reinterpret_cast<uint4 *>(smem)[g] = make_uint4(keep[0], keep[1], keep[2], keep[3]);
            if (gm[i]) atomicOr(&s_any[g / kLanes], 1u << ((g / 32) % kW));
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
    const float s = mx ? __fdiv_rn(__uint_as_float(mx), qf) : 1.0f;  // Eq. 1, per tensor
    // groups t and t + kT stand in ascending order: all of the first round come before the second
    const int n0 = lane < kWarps ? s_cnt[0][lane] : 0, n1 = lane < kWarps ? s_cnt[1][lane] : 0;
    const int total0 = __reduce_add_sync(0xffffffffu, n0);
    const int r_true = total0 + __reduce_add_sync(0xffffffffu, n1), r = min(r_true, a.cap);
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
            a.ctrl->s_x = s;
            a.ctrl->inv_s_x = __frcp_rn(s);
            a.ctrl->n_outliers = r_true;
            if (a.dev_status) {
                if (r_true > a.cap) atomicMax(a.dev_status, kStatusCapacity);
                // a cooperative preparation on this workspace ran into a time-out and left its mark
                if (__ldcg(&a.ctrl->arrived) & kPrepPoisonBit) atomicMax(a.dev_status, kStatusTimeout);
            }
        }
        s_last = atomicAdd(&a.ctrl->readers, 1u) == gridDim.x - 1 ? 1 : 0;  // (behind the barrier: the maxima have been read)
    }
    __syncthreads();
    if (s_last) {  // every CTA has read the maxima: zero again for the next call
        for (int i = t; i < (K >> 2); i += kT) reinterpret_cast<uint4 *>(a.colmax_rep)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (t == 0) a.ctrl->readers = 0u;
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (r) {  // every outlier channel into the list of the lane that owns its chunk
        for (int j = t; j < r; j += kT) s_next[j] = (uint16_t)atomicExch(&s_head[(s_oidx[j] >> 3) % kLanes], (uint32_t)j);
        __syncthreads();
    }

    // (the GEMM before this call has finished with the memory cleared here, the one behind it waits for this grid)
    for (uint32_t i = blockIdx.x * kT + t; i < (a.zero_bytes >> 4); i += gridDim.x * kT)
        static_cast<uint4 *>(a.zero)[i] = make_uint4(0u, 0u, 0u, 0u);

    // W_aux[n, c*j + i] = W_q[n, O_j]: a 4-byte word per lane, 32 words per warp, spread over the grid.  The GEMM reads the
    // Aux columns in steps of 32: codes, then zeros up to the next multiple.  The bytes of a thread's first word are
    // requested into L2 here and moved behind the rows.
    const int used = c * r, words = ((used + 31) & ~31) >> 2;
    const int w_total = a.w_aux ? a.N * words : 0, threads = gridDim.x * kT;
    const int wi = ((kWarps - 1 - warp) * (int)gridDim.x + (int)blockIdx.x) * 32 + lane;  // (short inputs leave the last warps without rows)
    if (wi < w_total) {
        const int n = wi / words, col = 4 * (wi - n * words);
        if (col < used) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.w_q + (size_t)n * a.ldw + s_oidx[col / c]));
        if (col + 3 < used) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.w_q + (size_t)n * a.ldw + s_oidx[(col + 3) / c]));
    }

    // ------------------------------------------------------------ rows
    uint32_t scaled = 0;  // chunk columns of this warp with an outlier channel (warp-uniform)
    if (kPerToken)
#pragma unroll
        for (int i = 0; i < kC; ++i) scaled |= ((s_any[i] >> (warp % kW)) & 1u) << i;
    const uint32_t own0 = r ? s_head[l] : kNone;
    const int ch0 = own0 != kNone ? s_oidx[own0] : 0;
    __half x0 = __float2half(0.0f);
    if (own0 != kNone && row >= 0) x0 = __ldg(xp + ch0);
    float lo, hi;
    if (!kPerToken) recip_bracket(__frcp_rn(s), lo, hi);
    const uint64_t magic2 = pack2(12582912.0f, 12582912.0f);  // 1.5 * 2^23 (quant8_bracket)
    int8_t *q = a.body_q + (ptrdiff_t)row * a.ld_q;
    uint32_t flip = 0;
    for (; row >= 0; row -= stride, xp -= xstep, q -= qstep) {
        float sr = s;
        if (kPerToken) {
            // the row's maximum of Body: channels outside O in fp16, those in O in fp32 times 2^-e (both exact)
            __half2 hm = __float2half2_rn(0.f);
#pragma unroll
            for (int i = 0; i < kC; ++i) {
                uint32_t x[4] = {v[i].x & 0x7FFF7FFFu, v[i].y & 0x7FFF7FFFu, v[i].z & 0x7FFF7FFFu, v[i].w & 0x7FFF7FFFu};
                if ((scaled >> i) & 1u) {
                    const uint4 keep = reinterpret_cast<const uint4 *>(smem)[min(l + i * kLanes, G - 1)];
                    x[0] &= keep.x; x[1] &= keep.y; x[2] &= keep.z; x[3] &= keep.w;
                }
                const __half2 *h = reinterpret_cast<const __half2 *>(x);
                hm = __hmax2(hm, __hmax2(__hmax2(h[0], h[1]), __hmax2(h[2], h[3])));
            }
            float om = fmaxf(__low2float(hm), __high2float(hm));
            if (own0 != kNone) {
                om = fmaxf(om, fabsf(__half2float(x0) * down));
                for (uint32_t j = s_next[own0]; j != kNone; j = s_next[j]) om = fmaxf(om, fabsf(__half2float(xp[s_oidx[j]]) * down));
            }
            uint32_t rm = __reduce_max_sync(0xffffffffu, __float_as_uint(om));
            if (kW > 1) {  // one barrier per row: the other buffer is written next
                if (lane == 0) s_rowmax[flip][warp] = __uint_as_float(rm);
                asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(kLanes) : "memory");
#pragma unroll
                for (int w = 0; w < kW; ++w) rm = max(rm, __float_as_uint(s_rowmax[flip][group * kW + w]));
                flip ^= 1u;
            }
            sr = rm ? __fdiv_rn(__uint_as_float(rm), qf) : 1.0f;
            recip_bracket(__frcp_rn(sr), lo, hi);
            if (l == 0) a.s_x_rows[row] = sr;
        }
        const uint64_t lo2 = pack2(lo, lo), hi2 = pack2(hi, hi);
        const bool more = row >= stride;
#pragma unroll
        for (int i = 0; i < kC; ++i) {
            const __half2 *h = reinterpret_cast<const __half2 *>(&v[i]);
            uint64_t f[4];
            uint32_t cb[8], diff = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // quant8_bracket, two values at a time
                const float2 p = __half22float2(h[j]);
                f[j] = pack2(p.x, p.y);
                const float2 th = unpack2(fma2(f[j], hi2, magic2)), tl = unpack2(fma2(f[j], lo2, magic2));
                cb[2 * j] = __float_as_uint(th.x);
                cb[2 * j + 1] = __float_as_uint(th.y);
                diff |= cb[2 * j] ^ __float_as_uint(tl.x);
                diff |= cb[2 * j + 1] ^ __float_as_uint(tl.y);
            }
            uint2 code = pack8(cb);
            if (diff) code = exact8(f[0], f[1], f[2], f[3], sr, qf);  // next to a tie: rare (and in outlier channels, done over below)
            if (l + i * kLanes < G) {
                reinterpret_cast<uint2 *>(q)[l + i * kLanes] = code;
                if (more) v[i] = ld_nc_v4(reinterpret_cast<const uint4 *>(xp - xstep) + l + i * kLanes);
            }
        }
        if (own0 != kNone) {
            const float olo = lo * down, ohi = hi * down;
            float x = __half2float(x0);
            if (more) x0 = __ldg(xp - xstep + ch0);
            int ch = ch0;
            for (uint32_t j = own0;;) {
                const uint32_t ca = __float_as_uint(fmaf(x, ohi, 12582912.0f)), cb = __float_as_uint(fmaf(x, olo, 12582912.0f));
                const int8_t code = (int8_t)(ca == cb ? (int)ca : quant_exact(x * down, sr, qf));
                q[ch] = code;
                if (a.aux_q) {
                    int8_t *aq = a.aux_q + (size_t)row * a.ld_aux + c * j;  // Aux_q[m, c*j + t] (Eq. 5, shared scale)
                    for (int k = 0; k < c; ++k) aq[k] = code;
                }
                j = s_next[j];
                if (j == kNone) break;
                ch = s_oidx[j];
                x = __half2float(xp[ch]);
            }
        }
        if (a.aux_q && used + l < 4 * words) a.aux_q[(size_t)row * a.ld_aux + used + l] = 0;
    }

    for (int i = wi; i < w_total; i += threads) {
        const int n = i / words, col = 4 * (i - n * words);
        const int8_t *wr = a.w_q + (size_t)n * a.ldw;
        uint32_t packed = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if (col + b < used) packed |= (uint32_t)(uint8_t)wr[s_oidx[(col + b) / c]] << (8 * b);
        *reinterpret_cast<uint32_t *>(a.w_aux + (size_t)n * a.ld_waux + col) = packed;
    }
}

template <bool kPerToken>
cudaError_t launch_rows(const PrepArgs &a, cudaLaunchConfig_t &cfg, int sms) {
    // warps per row: at most five chunks a lane (eight beyond K = 5120); chunks per lane: as few as hold the row, an empty
    // chunk column costs what a full one does
    const int G = a.K >> 3;
    const int w = G <= 160 ? 1 : G <= 320 ? 2 : 4, chunks = (G + 32 * w - 1) / (32 * w);
    // two CTAs per SM; short inputs: at least four busy warps per CTA
    long long ctas = ((long long)a.M * w + 3) / 4;
    if (ctas > 2 * sms) ctas = 2 * sms;
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.dynamicSmemBytes = (kPerToken ? (size_t)a.K * 2 : 0) + (size_t)a.cap * 4;
    using Fn = void (*)(PrepArgs);
    static const Fn fns[] = {
        k_quant_rows<kPerToken, 1, 2>, k_quant_rows<kPerToken, 1, 3>, k_quant_rows<kPerToken, 1, 4>, k_quant_rows<kPerToken, 1, 5>,
        k_quant_rows<kPerToken, 2, 3>, k_quant_rows<kPerToken, 2, 4>, k_quant_rows<kPerToken, 2, 5>,
        k_quant_rows<kPerToken, 4, 3>, k_quant_rows<kPerToken, 4, 4>, k_quant_rows<kPerToken, 4, 5>, k_quant_rows<kPerToken, 4, 8>};
    static PerDevice<int> done;
    const int dev = current_device();
    if (dev < 0) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(device_mutex());
        if (!done.have[dev]) {
            for (const Fn f : fns) {
                const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 8192 + 4 * kMaxOutlierCap);
                if (e != cudaSuccess) return e;
            }
            done.have[dev] = true;
        }
    }
    const Fn fn = w == 1   ? fns[chunks <= 2 ? 0 : chunks - 2]
                  : w == 2 ? fns[4 + chunks - 3]
                           : fns[chunks <= 5 ? 7 + chunks - 3 : 10];
    return cudaLaunchKernelEx(&cfg, fn, a);
}

}  // namespace

// The cooperative kernel keeps the own-scale reading of Aux, and long narrow inputs, whose rows mostly fit its shared memory:
// it reads X once and spends fewer instructions per row.  Whole layers with N = 768, cooperative / these, us: per tensor 2048 x
// 512 13.7 / 13.8, 4096 x 512 14.7 / 15.6, 4096 x 1040 18.9 / 18.1, 5000 x 1040 20.2 / 20.8, 16384 x 1536 43.7 / 44.5, 16384 x
// 2048 55.6 / 54.7; per token 3000 x 400 16.6 / 16.9, 6000 x 512 19.0 / 19.1, 16384 x 768 36.5 / 36.0.
bool prep_rows_preferred(const PrepArgs &a) {
    if (a.aux_own || a.K > kPrepMaxK) return false;
    if (a.per_token) return a.K > 512 || a.M <= 2048;
    return a.K >= 2048 || a.M <= (a.K > 512 ? 4608 : 1536);
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
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_channel_max, a, stripes, width, slices);
    if (e != cudaSuccess) return e;
    return a.per_token ? launch_rows<true>(a, cfg, sms) : launch_rows<false>(a, cfg, sms);
}

}  // namespace muxq
