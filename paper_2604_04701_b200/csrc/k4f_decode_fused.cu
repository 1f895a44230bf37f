// K4, fused form: the whole MUXQ layer for M <= 16 token rows in ONE launch -- detection (Section III-C), redistribution
// (Eq. 4-5), quantization (Eq. 1), the INT8 products with the Aux correction (Eq. 7) and the dequantization (Eq. 3).
//
// At these sizes a layer is a chain of latencies: the launch before it ends, its X is read, scaled, multiplied, stored.  The
// kernel keeps that chain short:
//   ahead      A CTA owns a contiguous block of output channels (N / SMs of them).  Their rows of W_q -- one contiguous
//              piece of memory -- are requested with a bulk asynchronous copy before the programmatic wait: they depend on
//              nothing, so they arrive while the launch before this one still runs.  The kernel lets its own dependents
//              start at once for the same reason.
//   X          Every CTA reads the few rows of X itself and quantizes them into shared memory (redundant, but no exchange
//              between CTAs).  A warp takes slices of 32 / RL groups of 8 channels, RL = min(MT, 4) lanes share a group's
//              rows; the channel maxima and flags stay in the lanes, two slices per warp stay in registers between the two
//              passes.  One barrier for the scale, one for the codes.
//   products   M <= 4: kLanes lanes per row of W_q, 16 bytes at a time, as 4-way byte dot products with every token row's
//              codes; the Aux term (Aux_q == Body_q[:, O], shared scale) is a pass of its own over the 16-channel pieces that
//              hold an outlier channel, with the codes masked.  The lanes of a row add up by exchanging halves, so that each
//              ends up with token rows of its own to dequantize and store.
//              M > 4: mma.sync tiles of 16 token rows x 8 output channels over 64-byte segments (lane (g, q) supplies 16 bytes
//              of token rows g, g + 8 and of W_q row g; the K order inside a segment is permuted alike for both), the warps
//              of a tile split K and add up through shared memory.  The legacy INT8 mma.sync issues about every 32 cycles
//              per SM sub-partition, which is what the dot products of four token rows cost.
//   reports    An extra CTA does the first step only and leaves channel maxima, O, r and scale(s) in the workspace, so that no
//              working CTA has the listing of O on its path.
// Layers whose share of W_q does not fit shared memory at once run through a ring of up to four chunks of rows.
// Measured (layers of a step in a CUDA graph, us per layer, the preceding form of this kernel -> here; per-tensor scales):
//                M = 1         M = 4         M = 16
//   528 x 2112   9.5 -> 2.1   10.9 -> 3.6   17.4 -> 5.4
//   768 x 3072   4.2 -> 2.8    4.8 -> 3.8    6.9 -> 5.9
//   1280 x 1280  4.1 -> 2.7    5.0 -> 3.8    6.7 -> 6.9
//   1280 x 5120  5.2 -> 3.9    6.1 -> 5.6    8.5 -> 8.1
//   5120 x 1280  7.9 -> 4.9    9.6 -> 8.4   16.7 -> 15.8
// What bounds it: at M = 1 the chain wait - X - scale - products - store; at M = 16 the redundant quantization of X.
#include "kernels.h"
#include "ptx.cuh"
#include "quant.cuh"

namespace muxq {

namespace {

constexpr int kT = 512;
constexpr int kWarps = kT / 32;
constexpr int kMaxK = 8192;
constexpr int kMaxBufs = 4;
constexpr int kMaxSmem = 220 * 1024;
// Two places per SM, this layer's CTA in one and the next layer's in the other: with room for a third, CTAs of one layer pile
// up on the SMs that empty first, and those set the pace (12 blocks of width 768 at M = 16, single calls: 432 us, with this floor 344).
constexpr int kMinSmem = 80 * 1024;
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

__device__ __forceinline__ void mma_s8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                       uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

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

__host__ __device__ constexpr int row_lanes(int MT) { return MT < 4 ? MT : 4; }  // lanes that share a group's token rows
// channels of X that the CTA's warps cover with `slices` slices each
__host__ __device__ constexpr int channels_of(int MT, int slices) { return slices * kWarps * 8 * (32 / row_lanes(MT)); }

// kHold: slices of a warp that stay in registers between the two passes.  Where that is all of X there is one batch and no loop
// around it; else the first batch is read last and stays.  Beyond 32 registers of X per thread one CTA per SM (such layers fill the
// shared memory of one anyway).
template <int MT, int kLanes, int kHold>
__global__ void __launch_bounds__(kT, kHold * (MT / row_lanes(MT)) > 8 ? 1 : 2) k_decode_fused(const DecodeFusedArgs a, const Geometry geo) {
    constexpr int RL = row_lanes(MT);
    constexpr int U = MT / RL;            // token rows per lane
    constexpr int CG = 32 / RL;           // groups of 8 channels per slice
    constexpr bool kAll = MT < 12 || kHold == 2;  // all of X (launch_decode_fused)
    constexpr bool kMma = MT >= 8;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t bar_full[kMaxBufs], bar_empty[kMaxBufs];
    __shared__ float s_max[kWarps][16];
    __shared__ float s_scale[16];
    __shared__ int s_nlist, s_r;
    __shared__ uint32_t s_abort;

    // From the trigger on the next kernel of the stream may become resident and fetch its own weights.  With few rows its start
    // gets in the way of this kernel's first loads, so it comes behind them (36 blocks of width 1280 at M = 1: 665 us with the
    // trigger here, 611 there, 767 behind the codes); with M > 4 the quantization is long enough to hide that (1280 -> 1280 at
    // M = 16: 6.9 us a layer with the trigger here, 7.6 there).
    if (kMma) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int t = threadIdx.x, lane = t & 31, warp = __shfl_sync(0xffffffffu, t >> 5, 0);
    const int K = a.K, G = K >> 3, M = a.M;
    const int workers = (int)gridDim.x - 1;
    const bool side = (int)blockIdx.x == workers;  // the reporting CTA
    const int n_begin = side ? 0 : (int)((long long)a.N * blockIdx.x / workers);
    const int n_end = side ? 0 : (int)((long long)a.N * (blockIdx.x + 1) / workers);
    const int n_rows = n_end - n_begin, chunks = (n_rows + geo.rows - 1) / geo.rows;
    int8_t *xq = reinterpret_cast<int8_t *>(smem);
    uint8_t *s_mask = smem + geo.off_mask;
    uint16_t *s_list = reinterpret_cast<uint16_t *>(smem + geo.off_list);
    uint8_t *s_w = smem + geo.off_w;
    volatile uint32_t *abort_flag = &s_abort;

    // ---------------------------------------------------------------- ahead of the wait: weights
    auto fetch = [&](int c) {  // warp 0
        const int b = geo.bufs == 1 ? 0 : c % geo.bufs, rows = min(geo.rows, n_rows - c * geo.rows);
        uint8_t *dst = s_w + (size_t)b * geo.rows * geo.wpitch;
        const int8_t *src = a.w_q + (size_t)(n_begin + c * geo.rows) * a.ldw;
        if (lane == 0) mbar_expect_tx(&bar_full[b], (uint32_t)(rows * K));
        __syncwarp();
        if (a.ldw == K && geo.wpitch == K) {
            if (lane == 0) bulk_load(dst, src, (uint32_t)(rows * K), &bar_full[b]);
        } else {
            for (int r = lane; r < rows; r += 32) bulk_load(dst + (size_t)r * geo.wpitch, src + (size_t)r * a.ldw, (uint32_t)K, &bar_full[b]);
        }
    };
    if (warp == 0) {
        if (lane == 0) {
            for (int b = 0; b < geo.bufs; ++b) {
                mbar_init(&bar_full[b], 1);
                mbar_init(&bar_empty[b], kWarps);
            }
            s_abort = 0u;
            s_nlist = 0;
            s_r = 0;
            fence_barrier_init();
        }
        __syncwarp();
        for (int c = 0; c < min(chunks, geo.bufs); ++c) fetch(c);
    }
    const float sw0 = __ldg(a.s_w);  // a constant of the layer like W_q
    {
        // X, which may still be being written, is asked into L2 (where those writes arrive too: nothing stale can come of it),
        // a share per CTA; likewise this CTA's per-channel scales and bias
        const int lines = (K + 63) >> 6;  // of 128 bytes per token row, give or take one
        for (int i = t * (int)gridDim.x + (int)blockIdx.x; i < M * lines; i += kT * (int)gridDim.x) {
            const int m = i / lines;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.X + (size_t)m * a.ldx + (i - m * lines) * 64));
        }
        if (t * 32 < n_rows) {
            if (a.per_vec) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.s_w + n_begin + t * 32));
            if (a.bias) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.bias + n_begin + t * 32));
        }
    }
    if (kMma) {
        for (int i = t; i < K >> 4; i += kT) reinterpret_cast<uint4 *>(s_mask)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (int i = t; i < (K + 63) >> 6; i += kT) smem[geo.off_list + i] = 0;
        // codes behind channel K in the last segment: zero, whatever stands behind the rows of W_q
        const int tail = (64 - (K & 63)) & 63;
        for (int i = t; i < MT * tail; i += kT) xq[(i / tail) * geo.xpitch + K + i % tail] = 0;
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // ---------------------------------------------------------------- X: channel maxima, flags, maxima of Body
    const int cg = lane % CG, rg = lane / CG;
    const float down = __int_as_float((127 - a.exp_factor) << 23);  // 2^-e
    const float qf = (float)a.qmax;
    const int rounds = (G + kWarps * CG - 1) / (kWarps * CG), batches = kAll ? 1 : (rounds + kHold - 1) / kHold;
    uint4 v[kHold][U];
    uint32_t masks[kHold];  // the lane's 8 channels
    auto load = [&](int round, uint4 (&x)[U]) {
        const int g = (round * kWarps + warp) * CG + cg;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int m = rg + RL * u;
            x[u] = make_uint4(0u, 0u, 0u, 0u);
            if (m < M && g < G) x[u] = ld_v4(a.X + (size_t)m * a.ldx + g * 8);
        }
    };
    auto channel_max = [&](const uint4 (&x)[U], __half2 (&cm)[4]) {
        cm[0] = cm[1] = cm[2] = cm[3] = __float2half2_rn(0.f);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const __half2 *h = reinterpret_cast<const __half2 *>(&x[u]);
#pragma unroll
            for (int i = 0; i < 4; ++i) cm[i] = __hmax2(cm[i], __habs2(h[i]));
        }
#pragma unroll
        for (int o = CG; o < 32; o <<= 1)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t w = __shfl_xor_sync(0xffffffffu, *reinterpret_cast<uint32_t *>(&cm[i]), o);
                cm[i] = __hmax2(cm[i], *reinterpret_cast<const __half2 *>(&w));
            }
    };
    auto flags = [&](const __half2 (&cm)[4]) {
        uint32_t mask = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (__low2float(cm[i]) > a.tau) mask |= 1u << (2 * i);  // strict (Section III-C)
            if (__high2float(cm[i]) > a.tau) mask |= 2u << (2 * i);
        }
        return mask;
    };
    float rm[U];
#pragma unroll
    for (int u = 0; u < U; ++u) rm[u] = 0.0f;
    for (int p = batches - 1; p >= 0; --p) {
#pragma unroll
        for (int h = 0; h < kHold; ++h)
            if (h < 2 || p * kHold + h < rounds) load(p * kHold + h, v[h]);
#pragma unroll
        for (int h = 0; h < kHold; ++h) {
            if (p * kHold + h >= rounds) break;
            const int g = ((p * kHold + h) * kWarps + warp) * CG + cg;
            __half2 cm[4];
            channel_max(v[h], cm);
            const uint32_t mask = flags(cm);
            masks[h] = mask;
            // row maxima of Body (Eq. 4): the channels outside O in fp16 as they are, those in O in fp32 times 2^-e (exact)
            uint32_t keep[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                keep[i] = 0x7FFF7FFFu & ~(((mask >> (2 * i)) & 1u ? 0xFFFFu : 0u) | ((mask >> (2 * i)) & 2u ? 0xFFFF0000u : 0u));
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t x[4] = {v[h][u].x & keep[0], v[h][u].y & keep[1], v[h][u].z & keep[2], v[h][u].w & keep[3]};
                const __half2 *q = reinterpret_cast<const __half2 *>(x);
                const __half2 hm = __hmax2(__hmax2(q[0], q[1]), __hmax2(q[2], q[3]));
                rm[u] = fmaxf(rm[u], fmaxf(__low2float(hm), __high2float(hm)));
            }
            if (mask) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    float f[8];
                    unpack8(v[h][u], f);
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if ((mask >> i) & 1u) rm[u] = fmaxf(rm[u], fabsf(f[i] * down));
                }
            }
            // pieces of 16 channels with an outlier channel: their masks and a list of them
            const uint32_t both = mask | __shfl_xor_sync(0xffffffffu, mask, 1);
            if (both && rg == 0 && g < G) {
                uint2 mb;  // 0xFF at the outlier channels (bit i of a nibble to byte i)
                mb.x = ((mask & 15u) * 0x00204081u & 0x01010101u) * 0xFFu;
                mb.y = ((mask >> 4) * 0x00204081u & 0x01010101u) * 0xFFu;
                *reinterpret_cast<uint2 *>(s_mask + g * 8) = mb;
                if (kMma) smem[geo.off_list + (g >> 3)] = 1;
                else if ((cg & 1) == 0) s_list[atomicAdd(&s_nlist, 1)] = (uint16_t)(g >> 1);
            }
            if (side && g < G) {
                if (rg == 0) {
                    const float2 c0 = __half22float2(cm[0]), c1 = __half22float2(cm[1]), c2 = __half22float2(cm[2]), c3 = __half22float2(cm[3]);
                    reinterpret_cast<float4 *>(a.colmax)[2 * g] = make_float4(c0.x, c0.y, c1.x, c1.y);
                    reinterpret_cast<float4 *>(a.colmax)[2 * g + 1] = make_float4(c2.x, c2.y, c3.x, c3.y);
                    s_w[g] = (uint8_t)mask;  // (no weights here: room for the flags of the listing below)
                }
            }
        }
    }
    if (!a.per_vec) {
#pragma unroll
        for (int u = 1; u < U; ++u) rm[0] = fmaxf(rm[0], rm[u]);
        const uint32_t b = __reduce_max_sync(0xffffffffu, __float_as_uint(rm[0]));
        if (lane == 0) s_max[warp][0] = __uint_as_float(b);
    } else {
#pragma unroll
        for (int o = 1; o < CG; o <<= 1)
#pragma unroll
            for (int u = 0; u < U; ++u) rm[u] = fmaxf(rm[u], __shfl_xor_sync(0xffffffffu, rm[u], o));
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (cg == 0) s_max[warp][rg + RL * u] = rm[u];
    }
    __syncthreads();
    if (!kMma) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (see the top)
    // ---------------------------------------------------------------- scale(s) (Eq. 1)
    float s = 1.0f;
    if (!a.per_vec) {
        const uint32_t mx = __reduce_max_sync(0xffffffffu, __float_as_uint(s_max[lane & (kWarps - 1)][0]));
        if (mx) s = __fdiv_rn(__uint_as_float(mx), qf);
        if (t < 16) s_scale[t] = s;
    } else {
        const int m = t >> 4;  // 16 lanes per token row (512 threads: rows 0..31, MT of them in use)
        float mx = m < MT ? s_max[t & 15][m] : 0.0f;
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (m < 16 && (t & 15) == 0) s_scale[m] = mx > 0.0f ? __fdiv_rn(mx, qf) : 1.0f;
        __syncthreads();
    }
    if (side) {
        // ------------------------------------------------------------ reports
        if (a.per_vec && t < M) a.s_x_rows[t] = s_scale[t];
        if (warp == 0) {
            int carry = 0;
            for (int base = 0; base < G; base += 32) {
                const int g = base + lane;
                uint32_t m = g < G ? s_w[g] : 0u;
                if (!__any_sync(0xffffffffu, m != 0u)) continue;
                const int cnt = __popc(m);
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int n = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += n;
                }
                int pos = carry + incl - cnt;
                for (; m; m &= m - 1, ++pos)
                    if (pos < a.cap) a.outlier_idx[pos] = 8 * g + __ffs(m) - 1;
                carry += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) {
                a.ctrl->n_outliers = carry;
                if (!a.per_vec) {
                    a.ctrl->s_x = s;
                    a.ctrl->inv_s_x = __frcp_rn(s);
                }
                if (carry > a.cap && a.dev_status) atomicMax(a.dev_status, kStatusCapacity);
            }
        }
        return;
    }

    // ---------------------------------------------------------------- codes of X into shared memory
    {
        float sc[U], inv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            sc[u] = a.per_vec ? s_scale[rg + RL * u] : s;
            inv[u] = u == 0 || a.per_vec ? __frcp_rn(sc[u]) : inv[0];
        }
        for (int p = 0; p < batches; ++p) {
            if (!kAll && p) {
#pragma unroll
                for (int h = 0; h < kHold; ++h)
                    if (p * kHold + h < rounds) load(p * kHold + h, v[h]);
            }
#pragma unroll
            for (int h = 0; h < kHold; ++h) {
                if (p * kHold + h >= rounds) break;
                const int g = ((p * kHold + h) * kWarps + warp) * CG + cg;
                if (!kAll && p) {
                    __half2 cm[4];
                    channel_max(v[h], cm);
                    masks[h] = flags(cm);
                }
                if (g >= G) continue;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int m = rg + RL * u;
                    if (m >= M) break;
                    float f[8];
                    unpack8(v[h][u], f);
                    if (masks[h])
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if ((masks[h] >> i) & 1u) f[i] *= down;  // exact
                    *reinterpret_cast<uint2 *>(xq + (size_t)m * geo.xpitch + g * 8) = quotient8(f, inv[u], sc[u]);
                }
            }
        }
    }
    __syncthreads();

    // ---------------------------------------------------------------- products
    bool ok = true;
    int b = 0;
    uint32_t phase = 0;
    for (int c = 0; c < chunks; ++c) {
        const int rows = min(geo.rows, n_rows - c * geo.rows), n0 = n_begin + c * geo.rows;
        ok = mbar_wait_warp(&bar_full[b], phase, abort_flag, a.spin);
        if (!kMma && !ok) break;
        const uint8_t *wc = s_w + (size_t)b * geo.rows * geo.wpitch;
        auto emit = [&](int m, int n, int acc) {
            const size_t o = (size_t)m * a.ldy + n;
            if (a.out_kind == 2) {
                reinterpret_cast<int32_t *>(a.Y)[o] = acc;
            } else {
                const float sw = a.per_vec ? __ldg(a.s_w + n) : sw0;
                float y = __fmul_rn(__fmul_rn(s_scale[m], sw), __int2float_rn(acc));  // Eq. 3
                if (a.bias) y = __fadd_rn(y, __ldcg(a.bias + n));
                if (a.out_kind == 1) reinterpret_cast<float *>(a.Y)[o] = y;
                else reinterpret_cast<__half *>(a.Y)[o] = __float2half_rn(y);
            }
        };
        if constexpr (!kMma) {
            constexpr int kRowsPerWarp = 32 / kLanes;
            const int sub = lane / kLanes, l = lane % kLanes, pieces = K >> 4, n_list = s_nlist;
            for (int r0 = warp * kRowsPerWarp; r0 < rows; r0 += kWarps * kRowsPerWarp) {
                const int r = min(r0 + sub, rows - 1);
                const uint8_t *wr = wc + (size_t)r * geo.wpitch;
                int acc[MT];
#pragma unroll
                for (int m = 0; m < MT; ++m) acc[m] = 0;
                auto dot = [&](int p, const uint4 &w, const uint4 &mk) {
#pragma unroll
                    for (int m = 0; m < MT; ++m) {
                        const uint4 x = *reinterpret_cast<const uint4 *>(xq + (size_t)m * geo.xpitch + p * 16);
                        acc[m] = __dp4a((int)w.x, (int)(x.x & mk.x), acc[m]);
                        acc[m] = __dp4a((int)w.y, (int)(x.y & mk.y), acc[m]);
                        acc[m] = __dp4a((int)w.z, (int)(x.z & mk.z), acc[m]);
                        acc[m] = __dp4a((int)w.w, (int)(x.w & mk.w), acc[m]);
                    }
                };
                if (n_list) {  // Aux first, times c, then Body on top (Eq. 7)
                    for (int i = l; i < n_list; i += kLanes) {
                        const int p = s_list[i];
                        dot(p, *reinterpret_cast<const uint4 *>(wr + p * 16), *reinterpret_cast<const uint4 *>(s_mask + p * 16));
                    }
#pragma unroll
                    for (int m = 0; m < MT; ++m) acc[m] *= a.c;
                }
                const uint4 all = make_uint4(~0u, ~0u, ~0u, ~0u);
#pragma unroll(MT <= 2 ? 4 : 2)
                for (int p = l; p < pieces; p += kLanes) dot(p, *reinterpret_cast<const uint4 *>(wr + p * 16), all);
                // the lanes of the row add up; each exchange halves the token rows a lane is left with
                int m_mine = 0;
                {
                    int o = kLanes / 2;
#pragma unroll
                    for (int n2 = MT / 2; n2 >= 1; n2 >>= 1, o >>= 1) {
                        const bool up = (l & o) != 0;
#pragma unroll
                        for (int j = 0; j < n2; ++j) {
                            const int give = up ? acc[j] : acc[j + n2], mine = up ? acc[j + n2] : acc[j];
                            acc[j] = mine + __shfl_xor_sync(0xffffffffu, give, o);
                        }
                        m_mine += up ? n2 : 0;
                    }
#pragma unroll
                    for (; o >= 1; o >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
                }
                if (r0 + sub < rows && m_mine < M && (l & (kLanes / MT - 1)) == 0) emit(m_mine, n0 + r, acc[0]);
            }
            if (c + geo.bufs < chunks) {
                __syncwarp();
                if (lane == 0) mbar_arrive(&bar_empty[b]);
                if (warp == 0) {
                    ok = mbar_wait_warp(&bar_empty[b], phase, abort_flag, a.spin);
                    if (!ok) break;
                    fetch(c + geo.bufs);
                }
            }
        } else {
            // teams of warps, one tile of 8 output channels at a time per team
            if (__syncthreads_or(!ok)) { ok = false; break; }
            const int g = lane >> 2, q = lane & 3, nseg = (K + 63) >> 6;
            const int tiles = (rows + 7) >> 3, teams = tiles < kWarps ? tiles : kWarps, wpt = kWarps / teams;
            const int team = warp / wpt, wi = warp - team * wpt;
            int *red = reinterpret_cast<int *>(smem + geo.off_red);
            const uint8_t *segflag = smem + geo.off_list;
            const int8_t *xrow = xq + g * geo.xpitch + q * 16;
            for (int t0 = 0; t0 < tiles; t0 += teams) {
                int acc[2][4], aux[4] = {0, 0, 0, 0};
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[0][j] = acc[1][j] = 0;
                if (team < teams && t0 + team < tiles) {
                    const uint8_t *wrow = wc + (size_t)min((t0 + team) * 8 + g, rows - 1) * geo.wpitch + q * 16;
#pragma unroll 2
                    for (int seg = wi; seg < nseg; seg += wpt) {
                        const uint4 w = *reinterpret_cast<const uint4 *>(wrow + seg * 64);
                        const uint4 x0 = *reinterpret_cast<const uint4 *>(xrow + seg * 64);
                        uint4 x1 = make_uint4(0u, 0u, 0u, 0u);
                        if (MT > 8) x1 = *reinterpret_cast<const uint4 *>(xrow + 8 * geo.xpitch + seg * 64);
                        mma_s8(acc[0], x0.x, x1.x, x0.y, x1.y, w.x, w.y);
                        mma_s8(acc[1], x0.z, x1.z, x0.w, x1.w, w.z, w.w);
                        if (segflag[seg]) {  // warp-uniform: Aux term on the outlier channels of this segment
                            uint4 mk = make_uint4(0u, 0u, 0u, 0u);
                            if (seg * 64 + q * 16 < K) mk = *reinterpret_cast<const uint4 *>(s_mask + seg * 64 + q * 16);
                            mma_s8(aux, x0.x & mk.x, x1.x & mk.x, x0.y & mk.y, x1.y & mk.y, w.x, w.y);
                            mma_s8(aux, x0.z & mk.z, x1.z & mk.z, x0.w & mk.w, x1.w & mk.w, w.z, w.w);
                        }
                    }
                }
                // this warp's 16 x 8 part: rows g, g + 8, columns 2q, 2q + 1; acc_b + c * acc_a (Eq. 7)
                int2 *mine = reinterpret_cast<int2 *>(red + warp * 128);
                mine[g * 4 + q] = make_int2(acc[0][0] + acc[1][0] + a.c * aux[0], acc[0][1] + acc[1][1] + a.c * aux[1]);
                mine[(g + 8) * 4 + q] = make_int2(acc[0][2] + acc[1][2] + a.c * aux[2], acc[0][3] + acc[1][3] + a.c * aux[3]);
                __syncthreads();
                for (int e = t; e < 128 * teams; e += kT) {
                    const int tt = e >> 7, el = e & 127, m = el >> 3, r = (t0 + tt) * 8 + (el & 7);
                    if (m < M && r < rows) {
                        int sum = 0;
                        for (int w = 0; w < wpt; ++w) sum += red[(tt * wpt + w) * 128 + el];
                        emit(m, n0 + r, sum);
                    }
                }
                __syncthreads();
            }
            if (warp == 0 && c + geo.bufs < chunks) fetch(c + geo.bufs);  // (everybody has passed the barrier above)
        }
        if (++b == geo.bufs) { b = 0; phase ^= 1u; }
    }
    if (!ok) {
        // time-out: the copies on their way land in this CTA's shared memory, so the warp that issued them stays (bounded)
        if (warp == 0)
            for (int i = 0; i < 1000; ++i) __nanosleep(1000);
        if (lane == 0 && a.dev_status) atomicMax(a.dev_status, kStatusTimeout);
    }
}

// M = 1: a token row is little enough for every warp to quantize all of it for itself, in registers -- no barrier, no exchange
// and no shared memory between X and the products.  Lane l holds the codes of the 8-channel groups l, l + 32, ... and
// multiplies them with the same bytes of the rows of W_q that are its warp's.
constexpr int kRowT = 256;
constexpr int kRowWarps = kRowT / 32;
constexpr int kRowMaxChunks = 6;  // K <= 1536

template <int kC>
__global__ void __launch_bounds__(kRowT, 2) k_decode_row(const DecodeFusedArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];  // this CTA's rows of W_q
    __shared__ uint64_t bar_full;
    __shared__ uint32_t s_abort;
    const int t = threadIdx.x, lane = t & 31, warp = __shfl_sync(0xffffffffu, t >> 5, 0);
    const int K = a.K, G = K >> 3;
    const int workers = (int)gridDim.x - 1;
    const bool side = (int)blockIdx.x == workers;
    const int n_begin = side ? 0 : (int)((long long)a.N * blockIdx.x / workers);
    const int rows = side ? 0 : (int)((long long)a.N * (blockIdx.x + 1) / workers) - n_begin;
    if (warp == 0) {
        if (lane == 0) {
            mbar_init(&bar_full, 1);
            s_abort = 0u;
            fence_barrier_init();
            mbar_expect_tx(&bar_full, (uint32_t)(rows * K));
        }
        __syncwarp();
        const int8_t *src = a.w_q + (size_t)n_begin * a.ldw;
        if (a.ldw == K) {
            if (lane == 0 && rows) bulk_load(smem, src, (uint32_t)(rows * K), &bar_full);
        } else {
            for (int r = lane; r < rows; r += 32) bulk_load(smem + (size_t)r * K, src + (size_t)r * a.ldw, (uint32_t)K, &bar_full);
        }
    }
    // this warp's rows, a lane each for scale, bias and result.  The bias is no constant of the layer (it may be what the launch
    // before this one stores, a residual): asked into L2 here, read behind the wait.
    const int per = (rows + kRowWarps - 1) / kRowWarps, r0 = warp * per, mine = max(min(per, rows - r0), 0);
    const int n_mine = n_begin + r0 + lane;
    const float sw = __ldg(a.s_w + (a.per_vec && lane < mine ? n_mine : 0));
    if (a.bias && lane < mine) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.bias + n_mine));
    for (int i = t * (int)gridDim.x + (int)blockIdx.x; i < (K + 63) >> 6; i += kRowT * (int)gridDim.x)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.X + i * 64));  // (see k_decode_fused)
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const float down = __int_as_float((127 - a.exp_factor) << 23);  // 2^-e
    const float qf = (float)a.qmax;
    uint4 v[kC];
#pragma unroll
    for (int i = 0; i < kC; ++i) {
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        if (lane + 32 * i < G) v[i] = ld_v4(reinterpret_cast<const uint4 *>(a.X) + lane + 32 * i);
    }
    const float bv = a.bias && lane < mine ? __ldcg(a.bias + n_mine) : 0.0f;
    // |x| > threshold for fp16 x: against the largest fp16 not above the threshold (strict, Section III-C)
    const __half2 tau2 = __half2half2(__float2half_rd(a.tau));
    uint32_t flagged = 0;  // bit i: chunk i of some lane of the warp holds an outlier channel
    float bmax = 0.0f;
#pragma unroll
    for (int i = 0; i < kC; ++i) {
        const __half2 *h = reinterpret_cast<const __half2 *>(&v[i]);
        __half2 m = __hmax2(__hmax2(__habs2(h[0]), __habs2(h[1])), __hmax2(__habs2(h[2]), __habs2(h[3])));
        if (__any_sync(0xffffffffu, __hgt2_mask(m, tau2) != 0u)) {
            flagged |= 1u << i;
            float f[8];
            unpack8(v[i], f);
#pragma unroll
            for (int j = 0; j < 8; ++j) bmax = fmaxf(bmax, fabsf(f[j]) > a.tau ? fabsf(f[j]) * down : fabsf(f[j]));  // Eq. 4: exact
        } else {
            bmax = fmaxf(bmax, fmaxf(__low2float(m), __high2float(m)));
        }
    }
    const uint32_t mx = __reduce_max_sync(0xffffffffu, __float_as_uint(bmax));
    const float s = mx ? __fdiv_rn(__uint_as_float(mx), qf) : 1.0f;  // Eq. 1
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (see k_decode_fused)
    auto mask_of = [&](const uint4 &x) {
        float f[8];
        unpack8(x, f);
        uint32_t mask = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) mask |= (fabsf(f[j]) > a.tau ? 1u : 0u) << j;
        return mask;
    };
    if (side) {
        // ------------------------------------------------------------ reports (k_decode_fused)
        if (warp == 0) {
            int carry = 0;
#pragma unroll
            for (int i = 0; i < kC; ++i) {
                const int g = lane + 32 * i;
                if (g < G) {
                    float f[8];
                    unpack8(v[i], f);
                    reinterpret_cast<float4 *>(a.colmax)[2 * g] = make_float4(fabsf(f[0]), fabsf(f[1]), fabsf(f[2]), fabsf(f[3]));
                    reinterpret_cast<float4 *>(a.colmax)[2 * g + 1] = make_float4(fabsf(f[4]), fabsf(f[5]), fabsf(f[6]), fabsf(f[7]));
                }
                if (!((flagged >> i) & 1u)) continue;
                uint32_t m = mask_of(v[i]);
                const int cnt = __popc(m);
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int n = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += n;
                }
                int pos = carry + incl - cnt;
                for (; m; m &= m - 1, ++pos)
                    if (pos < a.cap) a.outlier_idx[pos] = 8 * g + __ffs(m) - 1;
                carry += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) {
                a.ctrl->n_outliers = carry;
                if (a.per_vec) a.s_x_rows[0] = s;
                else {
                    a.ctrl->s_x = s;
                    a.ctrl->inv_s_x = __frcp_rn(s);
                }
                if (carry > a.cap && a.dev_status) atomicMax(a.dev_status, kStatusCapacity);
            }
        }
        return;
    }
    // codes; in flagged chunks also the masks of the outlier channels' bytes
    const float inv = __frcp_rn(s);
    float lo, hi;
    recip_bracket(inv, lo, hi);
    uint2 code[kC];
#pragma unroll
    for (int i = 0; i < kC; ++i) {
        float f[8];
        unpack8(v[i], f);
        uint32_t mask = 0;
        if ((flagged >> i) & 1u) {
            mask = mask_of(v[i]);
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if ((mask >> j) & 1u) f[j] *= down;  // exact
        }
        if (bracket8(f, lo, hi, code[i])) code[i] = quotient8(f, inv, s);
        if ((flagged >> i) & 1u) {  // (the values are not needed any more: their place keeps the masks)
            v[i].x = ((mask & 15u) * 0x00204081u & 0x01010101u) * 0xFFu;
            v[i].y = ((mask >> 4) * 0x00204081u & 0x01010101u) * 0xFFu;
        }
    }
    const bool ok = mbar_wait_warp(&bar_full, 0u, &s_abort, a.spin);
    if (!ok) {  // (as in k_decode_fused)
        if (warp == 0)
            for (int i = 0; i < 1000; ++i) __nanosleep(1000);
        if (lane == 0 && a.dev_status) atomicMax(a.dev_status, kStatusTimeout);
        return;
    }
    int acc = 0;  // lane j: output channel r0 + j
#pragma unroll 1
    for (int j = 0; j < mine; ++j) {
        const uint2 *w = reinterpret_cast<const uint2 *>(smem + (size_t)(r0 + j) * K) + lane;
        int body = 0, aux = 0;
#pragma unroll
        for (int i = 0; i < kC; ++i) {
            if (lane + 32 * i < G) {
                const uint2 x = w[32 * i];
                body = __dp4a((int)x.x, (int)code[i].x, body);
                body = __dp4a((int)x.y, (int)code[i].y, body);
                if ((flagged >> i) & 1u) {  // Aux_q == Body_q[:, O] (Eq. 5, shared scale)
                    aux = __dp4a((int)x.x, (int)(code[i].x & v[i].x), aux);
                    aux = __dp4a((int)x.y, (int)(code[i].y & v[i].y), aux);
                }
            }
        }
        const int sum = __reduce_add_sync(0xffffffffu, body + a.c * aux);  // Eq. 7
        if (lane == j) acc = sum;
    }
    if (lane < mine) {
        if (a.out_kind == 2) {
            reinterpret_cast<int32_t *>(a.Y)[n_mine] = acc;
        } else {
            float y = __fmul_rn(__fmul_rn(s, sw), __int2float_rn(acc));  // Eq. 3
            if (a.bias) y = __fadd_rn(y, bv);
            if (a.out_kind == 1) reinterpret_cast<float *>(a.Y)[n_mine] = y;
            else reinterpret_cast<__half *>(a.Y)[n_mine] = __float2half_rn(y);
        }
    }
}

Geometry geometry(int MT, int K, int rows_per_cta) {
    Geometry g;
    const int odd = MT >= 8 ? K + ((64 - K) & 127) : K;  // 64 modulo 128
    g.xpitch = MT >= 8 && odd < K + 48 ? odd + (odd < ((K + 63) & ~63) ? 128 : 0) : odd;  // a whole last segment of codes
    g.wpitch = odd;
    g.off_mask = MT * g.xpitch;
    g.off_list = g.off_mask + K;
    g.off_red = (g.off_list + K / 8 + 127) & ~127;
    g.off_w = g.off_red + (MT >= 8 ? kWarps * 128 * 4 : 0);
    // the CTA's whole share at once where it fits (a ring leaves no room for a second CTA on the SM either: 8192 x 2048 at M = 4
    // 14.6 us with one from 64 KB on, 12.8 without); else a ring
    g.rows = rows_per_cta;
    g.bufs = 1;
    if (g.off_w + rows_per_cta * g.wpitch + 64 > kMaxSmem) {
        g.rows = 48 * 1024 / g.wpitch;
        if (g.rows > 32) g.rows = 32;
        g.bufs = (kMaxSmem - 64 - g.off_w) / (g.rows * g.wpitch);
        if (g.bufs > kMaxBufs) g.bufs = kMaxBufs;
    }
    g.total = g.off_w + g.bufs * g.rows * g.wpitch + 64;  // (a last segment may read behind the last row)
    if (MT > 8 && g.total < 16 * g.xpitch) g.total = 16 * g.xpitch;  // its tiles read 16 rows of codes and drop what is none
    if (g.total < g.off_w + K / 8) g.total = g.off_w + K / 8;  // the reporting CTA's flags
    return g;
}

}  // namespace

bool decode_fused_supported(int M, int K) { return M >= 1 && M <= 16 && K % 16 == 0 && K <= kMaxK; }

cudaError_t launch_decode_fused(const DecodeFusedArgs &a0, cudaStream_t s) {
    const int sms = num_sms(), dev = current_device();
    if (sms < 1 || dev < 0) return cudaErrorInvalidDevice;
    DecodeFusedArgs a = a0;
    a.spin = test_hooks().spin_limit ? test_hooks().spin_limit : kSpinLimit;
    // Token rows of the instantiation, and whether X is wider than its first form keeps in registers.  M = 9..12 have a form of
    // their own only there: it saves a quarter of what is read twice (8192 x 2048 at M = 12 21.4 -> 19.2 us; with all of X in
    // registers the form for 16 rows is as fast or faster, 768 x 768 4.2 against 4.4 us).
    const int up = a.M <= 2 ? a.M : a.M <= 4 ? 4 : a.M <= 8 ? 8 : 16;
    const bool wide = a.K > channels_of(up, 2);
    const int MT = up == 16 && wide && a.M <= 12 ? 12 : up;
    // One CTA per SM, the reporting one included: a grid of more would put two CTAs of the same layer on some SM (the next
    // layer's take every SM's second place) and that SM would set the pace.
    const int workers = a.N < sms ? a.N : sms - 1, rows = (a.N + workers - 1) / workers;
    const Geometry geo = geometry(MT, a.K, rows);
    using Fn = void (*)(DecodeFusedArgs, Geometry);
    using RowFn = void (*)(DecodeFusedArgs);
    static const Fn fns[] = {
        k_decode_fused<1, 8, 2>, k_decode_fused<1, 16, 2>, k_decode_fused<1, 32, 2>, k_decode_fused<2, 8, 2>,
        k_decode_fused<2, 16, 2>, k_decode_fused<2, 32, 2>, k_decode_fused<4, 8, 2>, k_decode_fused<4, 16, 2>,
        k_decode_fused<4, 32, 2>, k_decode_fused<8, 32, 2>, k_decode_fused<16, 32, 2>,
        // wide X
        k_decode_fused<2, 8, 4>, k_decode_fused<2, 16, 4>, k_decode_fused<2, 32, 4>, k_decode_fused<4, 8, 8>,
        k_decode_fused<4, 16, 8>, k_decode_fused<4, 32, 8>, k_decode_fused<8, 32, 4>, k_decode_fused<8, 32, 8>,
        k_decode_fused<12, 32, 6>, k_decode_fused<16, 32, 5>};
    static const RowFn row_fns[5] = {k_decode_row<2>, k_decode_row<3>, k_decode_row<4>, k_decode_row<5>, k_decode_row<kRowMaxChunks>};
    static PerDevice<int> done;
    {
        std::lock_guard<std::mutex> lock(device_mutex());
        if (!done.have[dev]) {
            // One split of L1 for every layer: an SM changes it only when it is empty, so with a split per kernel the next
            // layer's CTAs pile up on the SMs that empty first (measured: 148 CTAs on 82 SMs).
            auto set = [](const void *f) {
                const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
                return e != cudaSuccess ? e : cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
            };
            cudaError_t e = cudaSuccess;
            for (const Fn f : fns)
                if (e == cudaSuccess) e = set(reinterpret_cast<const void *>(f));
            for (const RowFn f : row_fns)
                if (e == cudaSuccess) e = set(reinterpret_cast<const void *>(f));
            if (e != cudaSuccess) return e;
            done.have[dev] = true;
        }
    }
    if (geo.total > kMaxSmem || geo.bufs < 1 || geo.rows < 1) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(workers + 1);
    cfg.blockDim = dim3(kT);
    cfg.dynamicSmemBytes = (size_t)(geo.total < kMinSmem ? kMinSmem : geo.total);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (a.M == 1 && a.K <= 256 * kRowMaxChunks && rows * a.K <= 64 * 1024 && rows <= 32 * kRowWarps) {
        cfg.blockDim = dim3(kRowT);
        cfg.dynamicSmemBytes = (size_t)(rows * a.K < kMinSmem ? kMinSmem : rows * a.K);
        const int chunks = (a.K + 255) / 256;
        return cudaLaunchKernelEx(&cfg, row_fns[chunks <= 2 ? 0 : chunks - 2], a);
    }
    // lanes per row of W_q: as many as let every row of the CTA (of a chunk) be worked on at once
    const int r = geo.rows < rows ? geo.rows : rows, lanes = r <= kWarps ? 2 : r <= 2 * kWarps ? 1 : 0;
    const int i = !wide ? (MT == 1 ? lanes : MT == 2 ? 3 + lanes : MT == 4 ? 6 + lanes : MT == 8 ? 9 : 10)
                        : (MT == 2 ? 11 + lanes : MT == 4 ? 14 + lanes : MT == 8 ? (a.K > channels_of(8, 4) ? 18 : 17) : MT == 12 ? 19 : 20);
    return cudaLaunchKernelEx(&cfg, fns[i], a, geo);
}

}  // namespace muxq
