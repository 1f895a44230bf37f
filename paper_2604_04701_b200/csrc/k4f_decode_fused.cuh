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
//   528 x 2112   9.1 -> 2.2   11.2 -> 3.4   17.8 -> 4.5
//   768 x 3072   4.1 -> 2.5    4.7 -> 3.4    5.6 -> 4.8
//   1280 x 1280  4.3 -> 2.9    4.9 -> 3.7    6.5 -> 5.6
//   1280 x 5120  5.0 -> 3.7    5.8 -> 5.0    7.5 -> 6.7
// What bounds it: at M = 1 the chain wait - X - scale - products - store; at M = 16 the redundant quantization of X.
#pragma once
#include "k4f_common.cuh"

namespace muxq {
namespace decode {
namespace {

__device__ __forceinline__ void mma_s8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                       uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// kHold: slices of a warp that stay in registers between the two passes.  Where that is all of X (kAll) there is one batch and no
// loop around it; else the first batch is read last and stays.  Beyond 32 registers of X per thread one CTA per SM.
template <int MT, int kLanes, int kHold, bool kAll>
__global__ void __launch_bounds__(kT, kHold * (MT / row_lanes(MT)) > 8 ? 1 : 2) k_decode_fused(const DecodeFusedArgs a, const Geometry geo) {
    constexpr int RL = row_lanes(MT);
    constexpr int U = MT / RL;            // token rows per lane
    constexpr int CG = 32 / RL;           // groups of 8 channels per slice
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

}  // namespace

template <int MT>
cudaError_t launch_rows(const DecodeFusedArgs &a, const Geometry &geo, const cudaLaunchConfig_t &cfg, int lanes, bool alone, int dev) {
    using Fn = void (*)(DecodeFusedArgs, Geometry);
    Fn fns[6] = {};
    int i = lanes;
    if constexpr (MT == 1) {
        fns[0] = k_decode_fused<1, 8, 2, true>; fns[1] = k_decode_fused<1, 16, 2, true>; fns[2] = k_decode_fused<1, 32, 2, true>;
    } else if constexpr (MT <= 4) {
        constexpr int kWide = MT == 2 ? 4 : 8;
        fns[0] = k_decode_fused<MT, 8, 2, true>; fns[1] = k_decode_fused<MT, 16, 2, true>; fns[2] = k_decode_fused<MT, 32, 2, true>;
        fns[3] = k_decode_fused<MT, 8, kWide, true>; fns[4] = k_decode_fused<MT, 16, kWide, true>; fns[5] = k_decode_fused<MT, 32, kWide, true>;
        if (a.K > channels_of(MT, 2)) i += 3;
    } else if constexpr (MT == 8) {
        fns[0] = k_decode_fused<8, 32, 2, true>; fns[1] = k_decode_fused<8, 32, 4, true>;
        fns[2] = k_decode_fused<8, 32, 4, false>; fns[3] = k_decode_fused<8, 32, 8, true>;
        i = a.K <= channels_of(8, 2) ? 0 : a.K <= channels_of(8, 4) ? 1 : !alone ? 2 : 3;
    } else if constexpr (MT == 12) {
        fns[0] = k_decode_fused<12, 32, 6, false>;  // (alone only)
        i = 0;
    } else {
        fns[0] = k_decode_fused<16, 32, 2, true>; fns[1] = k_decode_fused<16, 32, 2, false>; fns[2] = k_decode_fused<16, 32, 5, false>;
        i = a.K <= channels_of(16, 2) ? 0 : !alone ? 1 : 2;
    }
    static PerDevice<int> done[6];
    const cudaError_t e = set_up(reinterpret_cast<const void *>(fns[i]), done[i], dev);
    return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, fns[i], a, geo);
}

}  // namespace decode
}  // namespace muxq
