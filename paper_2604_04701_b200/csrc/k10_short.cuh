// Short inputs (decode steps of several sequences, short prompts): the whole MUXQ layer in one launch, shared between the CTAs of a
// cluster along K -- detection (Section III-C), redistribution (Eq. 4-5), quantization (Eq. 1), the INT8 products with the Aux
// correction on the tensor cores (Eq. 7) and the dequantization (Eq. 3).
//
// A cluster owns a block of output channels, its CTAs a slice of the input channels each, for all token rows:
//   ahead      the CTA's part of W_q comes by TMA before the programmatic wait (a constant of the layer).
//   X          channel maxima of a slice need nobody else; the scale needs one exchange: every CTA stores its maximum (per token: its
//              rows' maxima) into the shared memory of the others, whose mbarrier counts the bytes in.
//   products   codes go straight into the swizzled A operand.  Up to 16 token rows (the operand has 128) a copy in which the channels
//              outside O are zero stands in the rows behind them: one product per step gives both sums of Eq. 7, whatever the number
//              of outlier channels and c, and a lane adds c times the row of its copy.  Beyond, a step of 32 channels that holds
//              an outlier channel has such a copy and is multiplied c more times with it: the weighted sum on one accumulator.
//              Rows behind those are whatever the memory holds; their sums are not looked at.
//   sums       every CTA stores its partial sums of a row into the shared memory of the CTA that finishes the row (integers: exact in
//              any order); then Eq. 3.
//   reports    channel maxima, O, r and scales by a cluster of its own that has no products; beyond 16 rows also codes and Aux block,
//              and W_aux by the others, from the bytes of W_q that they hold, while the sums are on their way.
//
// Bound by the chain of latencies, cycles from the wait on at 8 x 768 -> 768 in clusters of 8 (when outlier channels still cost products of
// their own): X 620, maxima 110, exchange 590, scale and codes 1110, products 1060, sums 870, output 1050; with cluster barriers instead
// of the counted stores both exchanges took twice that, with the partial sums row by row (16-byte stores 272 bytes apart) 128 rows took
// 2800 cycles to send instead of 1400, and a single cluster for all reports 20 to 45 us (W_aux).  At 128 rows the quantization (2300)
// and the sums (2800) count.
//
// A wait that runs out: the CTA that gives up stays until the others of its cluster have gone or given up as well, and products and
// copies on their way end first; what is stored then is in bounds.
#pragma once
#include <cuda.h>

#include "gemm_common.cuh"
#include "k4f_common.cuh"

namespace muxq {
namespace shorts {

constexpr int kT = 512;
constexpr int kWarps = kT / 32;
constexpr int kMaxRanks = 8;
constexpr int kMaxM = 128;
constexpr int kMaxKc = 1024;
constexpr int kStatusCapacity = 5;  // MUXQ_ERR_CAPACITY
constexpr int kStatusTimeout = 6;   // MUXQ_ERR_TIMEOUT

struct Plan {
    int ranks, clusters, bn;  // CTAs of a cluster; clusters with products, output channels of each
    int kc, kb;               // input channels of a CTA (a multiple of 32), blocks of 128 of them
    int mr;                   // token rows of the A operand (a multiple of 8)
    int rows;                 // token rows that a CTA finishes
    int pitch;                // bytes from four output channels of the partial sums to the next four: an odd multiple of 16
    int chunks, groups;       // 16-byte chunks of X per token row; token rows read at a time
    int a_block;              // bytes of the A operand per block of 128 channels
    int off_m, off_w, off_p, total;  // (off_m: from a code to its copy)
    int cols;                 // columns of tensor memory
    int line_shift;           // log2 of the threads that share out the token rows: a power of two, 32 to 128
    int skip;                 // -1; a test names a block of W_q that is not loaded so that a wait runs out
    uint32_t late;            // 0; a test names warps that give up at once, on the exchange of the maxima (16 + w: on the products)
};

struct Args {
    DecodeFusedArgs d;
    ShortOut out;
};

// Stores into the shared memory of a CTA of the cluster that count their bytes on an mbarrier there.
__device__ __forceinline__ void st_async(uint32_t addr, uint32_t bar, uint32_t x, uint32_t y) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(addr), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async(uint32_t addr, uint32_t bar, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// kHold: 16-byte chunks of X per thread that stay in registers between the two passes over X (kAll: that is all of them; else
// the first ones are read last and stay).  kFull: more than 16 token rows.
template <int kHold, bool kAll, bool kFull>
__global__ void __launch_bounds__(kT, 2) k_short(const __grid_constant__ CUtensorMap tm_w, const Args arg, const Plan g) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_w, bar_acc, bar_x, bar_p;
    __shared__ uint32_t s_tmem, s_abort;
    __shared__ uint2 s_slot[kMaxRanks][kWarps];  // of all CTAs: maximum of Body and number of outlier channels per warp of channels
    __shared__ __align__(16) uint32_t s_peer_row[kMaxRanks][kMaxM], s_row[kMaxM];  // per token: row maxima of all CTAs, of this one
    __shared__ float s_scale[kMaxM];
    __shared__ __align__(4) uint8_t s_flag[kMaxKc / 8];  // outlier channels, 8 to a byte
    __shared__ uint16_t s_list[kMaxKc];                  // ... in ascending order
    __shared__ int4 s_found;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const DecodeFusedArgs &a = arg.d;
    const ShortOut &out = arg.out;
    const int t = threadIdx.x, lane = t & 31, warp = __shfl_sync(0xffffffffu, t >> 5, 0);
    const int ranks = g.ranks, rank = (int)cluster_ctarank(), cluster = (int)blockIdx.x / ranks;
    const bool side = cluster == g.clusters;  // the reporting cluster
    const int M = a.M, K = a.K, n0 = cluster * g.bn;
    const int k0 = rank * g.kc, kn = max(0, min(g.kc, K - k0)), steps = (kn + 31) >> 5;
    const int words = 4 * g.chunks, nw = (words + 31) >> 5;  // pairs of channels of a slice, warps that look after them
    const int own_rows = max(0, min(g.rows, M - rank * g.rows));
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - smem_u32(smem_raw));
    volatile uint32_t *abort_flag = &s_abort;

    // ---------------------------------------------------------------- ahead of the wait
    if (warp == 0) {
        if (lane == 0) {
            mbar_init(&bar_w, 1);
            mbar_init(&bar_acc, 1);
            mbar_init(&bar_x, 1);
            mbar_init(&bar_p, 1);
            s_abort = 0u;
            fence_barrier_init();
            mbar_expect_tx(&bar_x, (uint32_t)(ranks * (nw * 8 + (a.per_vec ? (M + 3) / 4 * 16 : 0))));
            if (!side) {
                mbar_expect_tx(&bar_p, (uint32_t)(ranks * own_rows * g.bn * 4));
                const int boxes = (kn + 127) >> 7;
                if (boxes) mbar_expect_tx(&bar_w, (uint32_t)(boxes * g.bn * 128));
                for (int j = 0; j < boxes; ++j)
                    if (j != g.skip) tma_load_2d(smem + g.off_w + j * g.bn * 128, &tm_w, &bar_w, k0 + 128 * j, n0);
            }
        }
        __syncwarp();
    } else if (warp == 1 && !side) {
        tmem_alloc(&s_tmem, (uint32_t)g.cols);
        tmem_relinquish();
    }
    if (t < kMaxM) s_row[t] = 0u;
    if (t == kMaxM) s_found = make_int4(0, 0, 0, 0);
    const int rg = t / g.chunks, cg = t - rg * g.chunks;
    const bool on = rg < g.groups && 8 * cg < kn;
    // (divisions ahead of the wait: behind it they would be on the chain)
    const int quads = g.bn >> 2, fin_r = t / quads, fin_q = t - fin_r * quads;                                // to finish: row, four channels
    const int sum_m = (warp & 3) * 32 + lane, sum_to = min(sum_m / g.rows, ranks - 1), sum_row = sum_m - sum_to * g.rows;  // partial sums: row, whose
    {   // X is asked into L2, a share per CTA (where what still writes it writes to as well); so are scales and bias
        const int lines = (K + 63) >> 6;
        for (int i = t * (int)gridDim.x + (int)blockIdx.x; i < M * lines; i += kT * (int)gridDim.x) {
            const int m = i / lines;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.X + (size_t)m * a.ldx + (i - m * lines) * 64));
        }
        if (t * 32 < g.bn && n0 + t * 32 < a.N) {
            if (a.per_vec) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.s_w + n0 + t * 32));
            if (a.bias) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.bias + n0 + t * 32));
        }
    }
    const float sw0 = __ldg(a.s_w);
    const uint32_t spin_x = (g.late >> warp) & 1u ? 0u : a.spin;  // polls for the exchange
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    cluster_arrive();
    const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
    cluster_wait();  // the others have started: their shared memory may be written
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // ---------------------------------------------------------------- X: channel maxima of the slice
    const float down = __int_as_float((127 - a.exp_factor) << 23);  // 2^-e
    const float qf = (float)a.qmax;
    const int iters = (M + g.groups - 1) / g.groups, batches = kAll ? 1 : (iters + kHold - 1) / kHold;
    const bool marked = kFull && (__ldcg(&a.ctrl->arrived) & kPrepPoisonBit);  // an earlier call on the workspace timed out
    uint4 v[kHold];
    auto load = [&](int p) {
#pragma unroll
        for (int i = 0; i < kHold; ++i) {
            const int m = rg + (p * kHold + i) * g.groups;
            v[i] = make_uint4(0u, 0u, 0u, 0u);
            if (on && m < M) v[i] = decode::ld_v4(a.X + (size_t)m * a.ldx + k0 + 8 * cg);
        }
    };
    {
        __half2 cm[4];
        cm[0] = cm[1] = cm[2] = cm[3] = __float2half2_rn(0.f);
        for (int p = batches - 1; p >= 0; --p) {
            load(p);
#pragma unroll
            for (int i = 0; i < kHold; ++i) {
                const __half2 *h = reinterpret_cast<const __half2 *>(&v[i]);
#pragma unroll
                for (int j = 0; j < 4; ++j) cm[j] = __hmax2(cm[j], __habs2(h[j]));
            }
        }
        if (rg < g.groups) reinterpret_cast<uint4 *>(smem)[t] = *reinterpret_cast<const uint4 *>(cm);
    }
    __syncthreads();
    float lo = 0.0f, hi = 0.0f;
    if (warp < nw) {
        __half2 m = __float2half2_rn(0.f);
        if (t < words)
#pragma unroll 4
            for (int r = 0; r < g.groups; ++r) m = __hmax2(m, reinterpret_cast<const __half2 *>(smem)[r * words + t]);
        lo = __low2float(m);
        hi = __high2float(m);
        const bool f0 = lo > a.tau, f1 = hi > a.tau;  // strict (Section III-C)
        const uint32_t mx = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(f0 ? lo * down : lo, f1 ? hi * down : hi)));  // Eq. 4
        const uint32_t b0 = __ballot_sync(0xffffffffu, f0), b1 = __ballot_sync(0xffffffffu, f1);
        if (lane < ranks)
            st_async(map_to_cta(smem_u32(&s_slot[rank][warp]), lane), map_to_cta(smem_u32(&bar_x), lane), mx, (uint32_t)(__popc(b0) + __popc(b1)));
        const int at = lane & ~3;
        uint32_t flags = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) flags |= ((b0 >> (at + j)) & 1u) << (2 * j) | ((b1 >> (at + j)) & 1u) << (2 * j + 1);
        if ((lane & 3) == 0 && t < words) s_flag[t >> 2] = (uint8_t)flags;
    }
    __syncthreads();
    const uint32_t mask = on ? s_flag[cg] : 0u;
    if (a.per_vec) {
        uint32_t keep[4];  // pairs of channels outside O
#pragma unroll
        for (int j = 0; j < 4; ++j) keep[j] = ~(((mask >> (2 * j)) & 1u ? 0xFFFFu : 0u) | ((mask >> (2 * j)) & 2u ? 0xFFFF0000u : 0u));
        // Maxima of chunks go to shared memory, where as many threads as there are look after a token row each (M + 1 words from chunk to
        // chunk: neither side meets a bank twice; the operand that stands there later has more than the room).
        float *const part = reinterpret_cast<float *>(smem) + cg * (M + 1);
        for (int p = 0; p < batches; ++p) {
            if (!kAll && p) load(p);
#pragma unroll
            for (int i = 0; i < kHold; ++i) {
                const int m = rg + (p * kHold + i) * g.groups;
                if (rg >= g.groups || m >= M) break;
                const uint32_t x[4] = {v[i].x & keep[0], v[i].y & keep[1], v[i].z & keep[2], v[i].w & keep[3]};
                const __half2 *q = reinterpret_cast<const __half2 *>(x);
                const __half2 hm = __hmax2(__hmax2(__habs2(q[0]), __habs2(q[1])), __hmax2(__habs2(q[2]), __habs2(q[3])));
                float rm = fmaxf(__low2float(hm), __high2float(hm));
                if (mask) {
                    float f[8];
                    unpack8(v[i], f);
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if ((mask >> j) & 1u) rm = fmaxf(rm, fabsf(f[j] * down));
                }
                part[m] = rm;
            }
        }
        if (!kAll && batches > 1) load(0);
        __syncthreads();
        const int m_own = t & ((1 << g.line_shift) - 1);
        if (m_own < M) {
            float r = 0.0f;
#pragma unroll 4
            for (int i = t >> g.line_shift; i < g.chunks; i += kT >> g.line_shift) r = fmaxf(r, reinterpret_cast<const float *>(smem)[i * (M + 1) + m_own]);
            atomicMax(&s_row[m_own], __float_as_uint(r));
        }
        __syncthreads();
        const int to = t >> (g.line_shift - 2), m = 4 * (t & ((1 << (g.line_shift - 2)) - 1));  // (8 ranks x 32 threads at most)
        if (to < ranks && m < M) {
            const uint4 r = *reinterpret_cast<const uint4 *>(&s_row[m]);
            st_async(map_to_cta(smem_u32(&s_peer_row[rank][m]), to), map_to_cta(smem_u32(&bar_x), to), r.x, r.y, r.z, r.w);
        }
    }
    bool ok = mbar_wait_warp_cluster(&bar_x, 0u, abort_flag, spin_x) && !marked;

    // ---------------------------------------------------------------- scale(s) (Eq. 1)
    uint32_t mx = 0;
    if ((lane & 7) < ranks)
        for (int w = lane >> 3; w < nw; w += 4) mx = max(mx, s_slot[lane & 7][w].x);
    mx = __reduce_max_sync(0xffffffffu, mx);
    const float s = mx ? __fdiv_rn(__uint_as_float(mx), qf) : 1.0f;
    if (a.per_vec) {
        if (t < M) {
            uint32_t r = 0;
#pragma unroll
            for (int i = 0; i < kMaxRanks; ++i)
                if (i < ranks) r = max(r, s_peer_row[i][t]);
            s_scale[t] = r ? __fdiv_rn(__uint_as_float(r), qf) : 1.0f;
        }
        __syncthreads();
    }

    // ---------------------------------------------------------------- codes
    if (ok) {
        const bool copied = !kFull || (on && *reinterpret_cast<const uint32_t *>(s_flag + (cg & ~3)) != 0u);
        const uint32_t m0 = ((mask & 15u) * 0x00204081u & 0x01010101u) * 0xFFu, m1 = ((mask >> 4) * 0x00204081u & 0x01010101u) * 0xFFu;
        uint8_t *col = smem + (cg >> 4) * g.a_block + (cg & 1) * 8;
        const int piece = (cg & 15) >> 1;
        float sc = s, inv = __frcp_rn(s);
        for (int p = 0; p < batches; ++p) {
            if (!kAll && p) load(p);
#pragma unroll
            for (int i = 0; i < kHold; ++i) {
                const int m = rg + (p * kHold + i) * g.groups;
                if (!on || m >= M) break;
                if (a.per_vec) {
                    sc = s_scale[m];
                    inv = __frcp_rn(sc);
                }
                float f[8];
                unpack8(v[i], f);
                if (mask)
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if ((mask >> j) & 1u) f[j] *= down;  // exact
                const uint2 code = quotient8(f, inv, sc);
                uint8_t *at = col + m * 128 + ((piece ^ (m & 7)) << 4);
                *reinterpret_cast<uint2 *>(at) = code;
                if (copied) *reinterpret_cast<uint2 *>(at + g.off_m) = make_uint2(code.x & m0, code.y & m1);
            }
        }
    }
    // Every warp has polled for itself, and one may have run out of polls just before the last bytes came for the others.  The reporting
    // cluster gives up as a whole then.  In the others (where the vote costs 0.1 us) only warp 1 lists outlier channels, and where it has
    // given up there are none; sums of codes that are missing are sums of whatever is there, and those that are never sent end the wait for them.
    fence_proxy_async();
    if (side) ok = __syncthreads_and(ok);
    else __syncthreads();

    bool issued = false;  // (warp 0) products are on their way

    // Where the outlier channels stand in O: how many there are, before the slice, in the slice, and which those are (one warp).
    auto list_outliers = [&]() {
        int total = 0, first = 0, own = 0;
        if ((lane & 7) < ranks)
            for (int w = lane >> 3, r = lane & 7; w < nw; w += 4) {
                const int n = (int)s_slot[r][w].y;
                total += n;
                first += r < rank ? n : 0;
                own += r == rank ? n : 0;
            }
        total = __reduce_add_sync(0xffffffffu, total);
        first = __reduce_add_sync(0xffffffffu, first);
        own = __reduce_add_sync(0xffffffffu, own);
        if (lane == 0) s_found = make_int4(total, first, own, 0);
        int carry = 0;
        for (int c = 0; c < g.chunks; c += 32) {
            uint32_t f = c + lane < g.chunks ? s_flag[c + lane] : 0u;
            if (!__any_sync(0xffffffffu, f != 0u)) continue;
            const int n = __popc(f);
            int incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += x;
            }
            int pos = carry + incl - n;
            for (; f; f &= f - 1, ++pos) s_list[pos] = (uint16_t)(8 * (c + lane) + __ffs(f) - 1);
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
    };
    // row r of a swizzled operand of `rows` rows, byte k
    auto byte_at = [&](uint8_t *tile, int rows, int r, int k) { return tile + (k >> 7) * rows * 128 + r * 128 + ((((k >> 4) & 7) ^ (r & 7)) << 4) + (k & 15); };

    // Rows of an operand's outlier channels, each c times (Aux, W_aux): n_aux of them from place `first` in O on.  A thread puts a word
    // together, neighbours take neighbouring words, a row as many threads as it has words (bytes only in words that are shared with the next
    // CTA).  Measured, rows of layers, us: byte by byte, two threads to a row, 20 x 1280 -> 1280 with 64 outlier channels and c = 7 17.7,
    // with 200 40 (the three launches 14.3 and 22.7), so 11.6 and 16; with 8 channels, c = 3, even.
    auto repeat_outliers = [&](int8_t *dst, int ld, int rows, uint8_t *tile, int tile_rows, int first, int n_aux) {
        const int c = a.c, b0 = c * first, b1 = b0 + c * n_aux, w0 = b0 >> 2, n_words = ((b1 + 3) >> 2) - w0;  // (columns below 2^16)
        if (n_aux < 1) return;
        const int sh = min(5, 32 - __clz(n_words - 1));
        const uint32_t recip = c == 3 ? 0x55555556u : 0x24924925u;  // 2^32 / 3, / 7, rounded up
#pragma unroll 1
        for (int r = t >> sh; r < rows; r += kT >> sh)
#pragma unroll 1
            for (int x = t & ((1 << sh) - 1); x < n_words; x += 1 << sh) {
                const int col = 4 * (w0 + x);
                uint32_t v = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int q = c == 1 ? col + i : (int)__umulhi((uint32_t)(col + i), recip);
                    v |= (uint32_t)*byte_at(tile, tile_rows, r, s_list[min(max(q - first, 0), n_aux - 1)]) << (8 * i);
                }
                int8_t *p = dst + (size_t)r * ld + col;
                if (col >= b0 && col + 4 <= b1) {
                    *reinterpret_cast<uint32_t *>(p) = v;
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (col + i >= b0 && col + i < b1) p[i] = (int8_t)(v >> (8 * i));
                }
            }
    };

    if (side) {
        // ------------------------------------------------------------ reports
        if (ok) {
            if (warp == 1) list_outliers();
            __syncthreads();
            const int total = s_found.x, first = s_found.y, own = s_found.z;
            for (int j = t; j < own && first + j < a.cap; j += kT) a.outlier_idx[first + j] = k0 + s_list[j];
            if (2 * t < kn) *reinterpret_cast<float2 *>(a.colmax + k0 + 2 * t) = make_float2(lo, hi);
            if (rank == 0) {
                if (a.per_vec && t < M) a.s_x_rows[t] = s_scale[t];
                if (t == 0) {
                    a.ctrl->n_outliers = total;
                    if (!a.per_vec) {
                        a.ctrl->s_x = s;
                        a.ctrl->inv_s_x = __frcp_rn(s);
                    }
                    if (total > a.cap && a.dev_status) atomicMax(a.dev_status, kStatusCapacity);
                }
            }
            if constexpr (kFull) {
                const int listed = min(total, a.cap), n_aux = max(0, min(own, listed - first)), c = a.c, used = c * listed;
                const int zeros = ((used + 31) & ~31) - used, per_row = kn >> 3;
                for (int i = t; i < M * per_row; i += kT) {
                    const int m = i / per_row, k = (i - m * per_row) * 8;
                    *reinterpret_cast<uint2 *>(out.body_q + (size_t)m * out.ld_q + k0 + k) = *reinterpret_cast<const uint2 *>(byte_at(smem, g.mr, m, k));
                }
                repeat_outliers(out.aux_q, out.ld_aux, M, smem, g.mr, first, n_aux);
                if (lane < zeros)
                    for (int m = warp * ranks + rank; m < M; m += kWarps * ranks) out.aux_q[(size_t)m * out.ld_aux + used + lane] = 0;
            }
        }
    } else {
        // ------------------------------------------------------------ products
        if (warp == 0 && steps && ok) {
            ok = mbar_wait_warp(&bar_w, 0u, abort_flag, a.spin);
            tc_fence_after();
            if (ok) {
                const uint32_t idesc = idesc_i8(gemm::BM, g.bn);
                const uint32_t step_flags = lane < steps ? reinterpret_cast<const uint32_t *>(s_flag)[lane] : 0u;  // (at most 32 steps)
                const uint32_t outliers = __ballot_sync(0xffffffffu, step_flags != 0u);
                for (int st = 0; st < steps; ++st) {
                    const uint64_t ad = smem_desc_sw128(base + (st >> 2) * g.a_block) + 2 * (st & 3);
                    const uint64_t bd = smem_desc_sw128(base + g.off_w + (st >> 2) * g.bn * 128) + 2 * (st & 3);
                    mma_i8_ss_elect(tmem, ad, bd, idesc, st ? 1u : 0u);
                    if (kFull && ((outliers >> st) & 1u))  // Aux_q == Body_q[:, O] (Eq. 5), c times (Eq. 7)
                        for (int i = 0; i < a.c; ++i) mma_i8_ss_elect(tmem, ad + (g.off_m >> 4), bd, idesc, 1u);
                }
                mma_commit_elect(&bar_acc);
                issued = true;
            }
        }
        if (kFull && warp) {  // (while the products are at work)
            if (warp == 1 && ok) list_outliers();
            if (ok && steps) ok = mbar_wait_warp(&bar_w, 0u, abort_flag, a.spin);  // (W_q's bytes are read below)
        }
        if (ok && steps) ok = mbar_wait_warp(&bar_acc, 0u, abort_flag, (g.late >> (16 + warp)) & 1u ? 0u : a.spin);
        tc_fence_after();

        // ------------------------------------------------------------ partial sums to the CTAs that finish the rows
        const int quad = warp & 3;
        if (ok && quad * 32 < M) {
            const uint32_t bar = map_to_cta(smem_u32(&bar_p), sum_to);
            const uint32_t dst = map_to_cta(base + g.off_p, sum_to) + (uint32_t)(rank * quads * g.pitch + sum_row * 16);
            for (int i = warp >> 2; i < g.bn >> 4; i += 4) {
                uint32_t x[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) x[j] = 0u;
                if (steps) {
                    tmem_ld_32x16(tmem + ((uint32_t)(quad * 32) << 16) + 16 * i, x);
                    tmem_ld_wait();
                }
                if (!kFull)  // (8 or 16 rows behind: a lane of the same warp)
#pragma unroll
                    for (int j = 0; j < 16; ++j) x[j] += (uint32_t)a.c * __shfl_sync(0xffffffffu, x[j], (lane + g.mr) & 31);
                if (sum_m < M)
#pragma unroll
                    for (int j = 0; j < 4; ++j) st_async(dst + (4 * i + j) * g.pitch, bar, x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
            }
        }
        if constexpr (kFull) {  // W_aux, while the sums are on their way
            __syncthreads();
            const int total = s_found.x, first = s_found.y, own = s_found.z;
            const int listed = min(total, a.cap), n_aux = max(0, min(own, listed - first)), c = a.c, used = c * listed;
            const int zeros = ((used + 31) & ~31) - used, n = min(g.bn, a.N - n0);
            if (ok) repeat_outliers(out.w_aux + (size_t)n0 * out.ld_waux, out.ld_waux, n, smem + g.off_w, g.bn, first, n_aux);
            if (ok && lane < zeros)
                for (int i = warp * ranks + rank; i < n; i += kWarps * ranks) out.w_aux[(size_t)(n0 + i) * out.ld_waux + used + lane] = 0;
        }
        if (ok) ok = mbar_wait_warp_cluster(&bar_p, 0u, abort_flag, a.spin);

        // ------------------------------------------------------------ this CTA's rows: sums of all slices, Eq. 3
        if (ok) {
            int r = fin_r, q = fin_q;
            for (int i = t; i < own_rows * quads; i += kT, r = i / quads, q = i - r * quads) {
                const int n = n0 + 4 * q, mm = rank * g.rows + r;
                if (n >= a.N) continue;
                const uint8_t *p = smem + g.off_p + q * g.pitch + r * 16;
                int4 part[kMaxRanks];
#pragma unroll
                for (int x = 0; x < kMaxRanks; ++x) {
                    part[x] = make_int4(0, 0, 0, 0);
                    if (x < ranks) part[x] = *reinterpret_cast<const int4 *>(p + x * quads * g.pitch);
                }
                int4 sum = part[0];
#pragma unroll
                for (int x = 1; x < kMaxRanks; ++x) { sum.x += part[x].x; sum.y += part[x].y; sum.z += part[x].z; sum.w += part[x].w; }
                const size_t o = (size_t)mm * a.ldy + n;
                if (a.out_kind == 2) {
                    *reinterpret_cast<int4 *>(reinterpret_cast<int32_t *>(a.Y) + o) = sum;
                    continue;
                }
                const float sx = a.per_vec ? s_scale[mm] : s;
                const float4 sw = a.per_vec ? __ldg(reinterpret_cast<const float4 *>(a.s_w + n)) : make_float4(sw0, sw0, sw0, sw0);
                float4 y = make_float4(__fmul_rn(__fmul_rn(sx, sw.x), __int2float_rn(sum.x)), __fmul_rn(__fmul_rn(sx, sw.y), __int2float_rn(sum.y)),
                                       __fmul_rn(__fmul_rn(sx, sw.z), __int2float_rn(sum.z)), __fmul_rn(__fmul_rn(sx, sw.w), __int2float_rn(sum.w)));
                if (a.bias) {
                    const float4 b = __ldcg(reinterpret_cast<const float4 *>(a.bias + n));
                    y = make_float4(__fadd_rn(y.x, b.x), __fadd_rn(y.y, b.y), __fadd_rn(y.z, b.z), __fadd_rn(y.w, b.w));
                }
                if (a.out_kind == 1) {
                    *reinterpret_cast<float4 *>(reinterpret_cast<float *>(a.Y) + o) = y;
                } else {
                    const __half2 h0 = __floats2half2_rn(y.x, y.y), h1 = __floats2half2_rn(y.z, y.w);
                    *reinterpret_cast<uint2 *>(reinterpret_cast<__half *>(a.Y) + o) =
                        make_uint2(*reinterpret_cast<const uint32_t *>(&h0), *reinterpret_cast<const uint32_t *>(&h1));
                }
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    // A CTA whose waits have all come true has received all that the others store into it and may go.  One that gave up stays until
    // the others have gone or given up as well: the barrier counts those that have not exited.
    if (!ok) {
        if (lane == 0 && a.dev_status) atomicMax(a.dev_status, kStatusTimeout);
        // the weights on their way land first, and products read shared memory and write tensor memory to the end
        if (warp == 0 && steps && !side && !mbar_wait_warp(issued ? &bar_acc : &bar_w, 0u, abort_flag, a.spin))
            for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    tc_fence_before();
    if (__syncthreads_or(!ok)) {
        cluster_arrive();
        cluster_wait();
    }
    if (warp == 1 && !side) {
        tc_fence_after();
        tmem_dealloc(tmem, (uint32_t)g.cols);
    }
}

}  // namespace shorts
}  // namespace muxq
