// K4, list form for independent layers: the decode-shaped MUXQ layers of a list (M <= 16 token rows each; Section
// III-C, Eq. 1, Eq. 4-5, Eq. 7, Eq. 3 per layer) as two launches, a preparation of every X and one persistent
// stream over all weights on the 5th-generation tensor cores.
//
//   k_list_prep    One cluster of four CTAs per layer.  The CTAs split the channels; a warp takes slices of 64 channels,
//                  derives their maxima and outlier flags, the CTAs exchange the maxima of Body through distributed
//                  shared memory, and each quantizes its share.  The codes go to the plan's device memory as the
//                  B operand of the products: per 128 channels a block of 2R rows x 128 bytes in the 128-byte-swizzled
//                  layout, rows 0..R-1 the codes of the token rows, rows R..2R-1 the same codes masked to the outlier
//                  channels (Aux_q == Body_q[:, O], Eq. 5), R = 8 or 16.
//   k_list_stream  One CTA per SM, launched as a programmatic dependent: its weight stream starts while X is still being
//                  prepared.  The weights are the A operand: D[128 output channels][2R] = W_q[128 rows] . codes, so that
//                  Body's product and the Aux term (Eq. 7) for all token rows come out of one pass of
//                  tcgen05.mma kind::i8 over each weight tile, whatever M and however many outlier channels.
//
// The work of a list is a line of K blocks (128 rows x 128 bytes of W_q, 16 KB), layer after layer, tile after tile; CTA
// b takes the b-th of `grid` equal pieces.  A tile cut by the end of a piece is finished by whoever comes last: its
// CTAs add their integer partial sums (exact in any order) into a slot of the plan's memory and count themselves in; the
// last one reads the total and stores Y.  Nobody waits for another CTA.
//
// Bound by HBM (W_q once).  A loader warp keeps 11 or 12 stages (about 200 KB per SM) in flight, one thread issues four
// MMAs per stage, four warps read the accumulators; nothing else runs, whereas the streaming kernel for dependent lists
// (k4s_decode_stream.cu) does the products in warps, which costs it more than the stream from M = 4 on.  Measured against
// that kernel (it keeps the dependent lists, where a layer's tiles of 128 rows would leave most SMs idle), weights of
// width-1280 / 1024 / 1280 models: 144 layers at M = 1 132.8 -> 122 us (708 MB: 5.8 TB/s), 96 at M = 4 153.7 -> 60.6 us
// (302 MB: 5.0 TB/s), 144 at M = 16 293 -> 137 us (5.3 TB/s).  The preparation is launched programmatically too (its wait comes first, the
// weights' stream is let go behind it, so nothing is read that a launch before the list still writes), which shows where lists follow one another, 121.5 -> 120.5,
// 60.7 -> 58.5, 136.1 -> 134.6 us, and not in a first pass by itself; with the stream letting the next launch start early as well 122.4, 59.9, 135.6.  What is left over HBM
// time is the start: the stages are full some 6 us after the launch and the preparation ends at 7 (M = 1) to 12 us (M = 16, K = 5120; eight smaller CTAs per layer
// instead of four: 11 to 16 us, no gain).
#include <cuda.h>
#include <string.h>

#include "gemm_common.cuh"
#include "quant.cuh"

namespace muxq {

namespace {

using gemm::kStatusTimeout;
constexpr int kStatusCapacity = 5;  // MUXQ_ERR_CAPACITY
constexpr int kPrepCtas = 4;        // CTAs (one cluster) that prepare one layer
constexpr int kPrepThreads = 256;
constexpr int kPrepWarps = kPrepThreads / 32;
constexpr int kTileN = 128;         // output channels per tile
constexpr int kBK = 128;            // bytes of K per stage
constexpr int kThreads = 192;       // loader, MMA, four epilogue warps

constexpr int kHeaderBytes = 128;   // a layer's scales, in front of its codes
__host__ __device__ constexpr int code_rows(int M) { return M <= 8 ? 8 : 16; }
__host__ __device__ inline size_t layer_scratch_bytes(int R, int K) {
    return (size_t)kHeaderBytes + (size_t)((K + kBK - 1) / kBK) * (2 * R * kBK);
}

// ---------------------------------------------------------------- preparation of X
// U: 4-row groups of token rows (M <= 4 U).  Lane (rg, cg): rows rg, rg + 4, ..., channels 8 cg .. 8 cg + 7 of a slice.
// (Registers are bounded so that four of these CTAs and one of the stream's fit an SM together.)
template <int U>
__global__ void __launch_bounds__(kPrepThreads, 5) k_list_prep(const ListArgs a) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    constexpr int R = U == 4 ? 16 : 8;
    __shared__ float s_max[kPrepWarps][16];
    __shared__ int s_cnt[kPrepWarps];
    __shared__ float s_ex[16];  // this CTA's row maxima of Body (per tensor: entry 0) and outlier count, read by the cluster
    __shared__ int s_exr;
    __shared__ float s_scale[16];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rg = lane >> 3, cg = lane & 7;
    const int l = blockIdx.y, rank = blockIdx.x, M = a.M;
    const ChainLayer &ly = a.layers[l];
    const __half *X = ly.X;
    const int ldx = ly.ldx, ns = ly.K >> 6;
    const int per = (ns + kPrepCtas - 1) / kPrepCtas;
    const int s_begin = rank * per, s_end = min(ns, s_begin + per);
    const float down = __int_as_float((127 - a.exp_factor) << 23);  // 2^-e
    const float qf = (float)a.qmax;

    auto load = [&](int s, int u) {
        const int m = rg + 4 * u;
        return m < M ? ld_plain_v4(X + (size_t)m * ldx + s * 64 + cg * 8) : make_uint4(0u, 0u, 0u, 0u);
    };
    // all of a warp's slices are requested now, ahead of the weights, so that the rounds below find them in L2
    for (int s = s_begin + warp; s < s_end; s += kPrepWarps)
        if (lane < M) asm volatile("prefetch.global.L2 [%0];" ::"l"(X + (size_t)lane * ldx + s * 64));

    // the weight stream needs nothing from here for its first stages; it waits for this grid before it reads codes
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint32_t masks = 0;  // the lane's 8 flag bits of up to four rounds
    float rm[U];
#pragma unroll
    for (int u = 0; u < U; ++u) rm[u] = 0.0f;
    int cnt = 0, round = 0, s = s_begin + warp;
    uint4 v[U];
    for (; s < s_end; s += kPrepWarps, ++round) {
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = load(s, u);
        __half2 cm[4];
        cm[0] = cm[1] = cm[2] = cm[3] = __float2half2_rn(0.f);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const __half2 *h = reinterpret_cast<const __half2 *>(&v[u]);
#pragma unroll
            for (int i = 0; i < 4; ++i) cm[i] = __hmax2(cm[i], __habs2(h[i]));
        }
        uint32_t mask = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t w = *reinterpret_cast<uint32_t *>(&cm[i]);
            uint32_t o = __shfl_xor_sync(0xffffffffu, w, 8);
            cm[i] = __hmax2(cm[i], *reinterpret_cast<__half2 *>(&o));
            w = *reinterpret_cast<uint32_t *>(&cm[i]);
            o = __shfl_xor_sync(0xffffffffu, w, 16);
            cm[i] = __hmax2(cm[i], *reinterpret_cast<__half2 *>(&o));
            if (__low2float(cm[i]) > a.tau) mask |= 1u << (2 * i);  // strict (Section III-C)
            if (__high2float(cm[i]) > a.tau) mask |= 2u << (2 * i);
        }
        masks |= mask << (8 * round);
        if (rg == 0) cnt += __popc(mask);
        // Row maxima of Body (Eq. 4), in fp16 where nothing is scaled: the channels outside O as they are; those in O
        // (few) in fp32 times 2^-e.  Both exact.
        uint32_t keep[4];  // |.| of the channels outside O
#pragma unroll
        for (int i = 0; i < 4; ++i)
            keep[i] = 0x7FFF7FFFu & ~(((mask >> (2 * i)) & 1u ? 0xFFFFu : 0u) | ((mask >> (2 * i)) & 2u ? 0xFFFF0000u : 0u));
#pragma unroll
        for (int u = 0; u < U; ++u) {
            uint32_t x[4] = {v[u].x & keep[0], v[u].y & keep[1], v[u].z & keep[2], v[u].w & keep[3]};
            const __half2 *h = reinterpret_cast<const __half2 *>(x);
            const __half2 hm = __hmax2(__hmax2(h[0], h[1]), __hmax2(h[2], h[3]));
            rm[u] = fmaxf(rm[u], fmaxf(__low2float(hm), __high2float(hm)));
        }
        if (mask) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float f[8];
                unpack8(v[u], f);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if ((mask >> i) & 1u) rm[u] = fmaxf(rm[u], fabsf(f[i] * down));
            }
        }
    }
    if (!a.per_vec) {
#pragma unroll
        for (int u = 1; u < U; ++u) rm[0] = fmaxf(rm[0], rm[u]);
        rm[0] = warp_max(rm[0]);
        if (lane == 0) s_max[warp][0] = rm[0];
    } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            rm[u] = fmaxf(rm[u], __shfl_xor_sync(0xffffffffu, rm[u], 1));
            rm[u] = fmaxf(rm[u], __shfl_xor_sync(0xffffffffu, rm[u], 2));
            rm[u] = fmaxf(rm[u], __shfl_xor_sync(0xffffffffu, rm[u], 4));
            if (cg == 0) s_max[warp][rg + 4 * u] = rm[u];
        }
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) s_cnt[warp] = cnt;
    __syncthreads();
    if (t < 16) {
        float mx = 0.0f;
        const bool have = a.per_vec ? t < 4 * U : t == 0;
#pragma unroll
        for (int w = 0; w < kPrepWarps; ++w)
            if (have) mx = fmaxf(mx, s_max[w][t]);
        s_ex[t] = mx;
    } else if (t == 32) {
        int r = 0;
#pragma unroll
        for (int w = 0; w < kPrepWarps; ++w) r += s_cnt[w];
        s_exr = r;
    }
    cluster_sync_all();
    uint8_t *head = a.scratch + (size_t)ly.codes_off * 128;
    if (t < 16) {
        float mx = 0.0f;
#pragma unroll
        for (int c = 0; c < kPrepCtas; ++c) {
            float v;
            asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(map_to_cta(smem_u32(&s_ex[a.per_vec ? t : 0]), c)));
            mx = fmaxf(mx, v);
        }
        const float sc = mx > 0.0f ? __fdiv_rn(mx, qf) : 1.0f;  // Eq. 1
        s_scale[t] = sc;
        if (rank == 0) reinterpret_cast<float *>(head)[t] = sc;
        if (rank == 0 && t == 0) {
            int r = 0;
#pragma unroll
            for (int c = 0; c < kPrepCtas; ++c) {
                int v;
                asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(map_to_cta(smem_u32(&s_exr), c)));
                r += v;
            }
            const bool over = r > a.cap;  // MUXQ_ERR_CAPACITY: Y of this layer is unspecified
            if (over && a.dev_status) atomicMax(a.dev_status, kStatusCapacity);
            if (a.results) {
                ChainResult rr;
                rr.n_outliers = r;
                rr.status = over ? kStatusCapacity : 0;
                rr.s_x = sc;
                rr.reserved = 0;
                a.results[l] = rr;
            }
        }
    }
    // this CTA has read the others' words; nobody leaves before everybody has (waited for at the end)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    __syncthreads();
    float sc[U], inv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        sc[u] = s_scale[rg + 4 * u];
        inv[u] = __frcp_rn(sc[u]);
    }
    // the rounds again, last one first: its values are still in registers
    for (bool held = true; round > 0; held = false) {
        --round;
        s -= kPrepWarps;
        if (!held)
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = load(s, u);
        const uint32_t mask = (masks >> (8 * round)) & 0xFFu;
        const int ch = s * 64 + cg * 8;
        uint8_t *block = head + kHeaderBytes + (size_t)(ch >> 7) * (2 * R * kBK);
        const int chunk = (ch & 127) >> 4, half = ch & 8;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int m = rg + 4 * u;
            if (m >= M) break;
            float f[8];
            unpack8(v[u], f);
            if (mask)
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if ((mask >> i) & 1u) f[i] *= down;  // exact
            const uint2 code = quotient8(f, inv[u], sc[u]);
            uint8_t *q = block + m * kBK + ((chunk ^ (m & 7)) << 4) + half;
            *reinterpret_cast<uint2 *>(q) = code;
            // 0xFF at the outlier channels of this lane's eight (bit i of a nibble to byte i)
            const uint32_t m0 = ((mask & 15u) * 0x00204081u & 0x01010101u) * 0xFFu, m1 = ((mask >> 4) * 0x00204081u & 0x01010101u) * 0xFFu;
            *reinterpret_cast<uint2 *>(q + R * kBK) = make_uint2(code.x & m0, code.y & m1);  // (R is a multiple of 8: same swizzle)
        }
    }
    // the slots of cut tiles start the run at zero
    {
        const int words4 = a.grid * M * (kTileN / 4);
        const int nthr = gridDim.x * gridDim.y * kPrepThreads, me = (l * kPrepCtas + rank) * kPrepThreads + t;
        for (int i = me; i < words4; i += nthr) reinterpret_cast<uint4 *>(a.fix)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (int i = me; i < 4 * a.grid; i += nthr) a.fix_count[i] = 0u;
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---------------------------------------------------------------- the weight stream
template <int R>
struct Cfg {
    static constexpr int kStageW = kTileN * kBK;
    static constexpr int kStageX = 2 * R * kBK;
    static constexpr int kStageBytes = kStageW + kStageX;
    static constexpr int kStages = (227 * 1024 - 2048) / kStageBytes;
    static constexpr int kSmemBytes = kStages * kStageBytes + 1024;
    static constexpr int kAccCols = 2 * R;               // accumulator columns of one tile
    static constexpr int kTmemCols = R == 16 ? 64 : 32;  // two buffers
    static_assert(kStageBytes % 1024 == 0, "swizzled operand blocks start at multiples of 1024 bytes");
};

// Position on the line of K blocks.
struct Walk {
    int l, tile, kb, nkb, tiles;
    const ChainLayer *tab;
    __device__ __forceinline__ void layer() {
        const int K = __ldg(&tab[l].K), N = __ldg(&tab[l].N);
        nkb = (K + kBK - 1) / kBK;
        tiles = (N + kTileN - 1) / kTileN;
    }
    __device__ __forceinline__ void start(const ChainLayer *t, int first_layer, uint32_t pos) {
        tab = t;
        l = first_layer;
        layer();
        const uint32_t rel = pos - __ldg(&tab[l].kb_first);
        tile = (int)(rel / (uint32_t)nkb);
        kb = (int)(rel - (uint32_t)tile * nkb);
    }
    // true when the next block belongs to another layer (the caller knows that there is a next block)
    __device__ __forceinline__ bool next_tile() {
        kb = 0;
        if (++tile < tiles) return false;
        tile = 0;
        ++l;
        layer();
        return true;
    }
};

__device__ __forceinline__ void bulk_load_elect(void *smem_dst, const void *gsrc, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n\t}\n" ::"r"(
            smem_u32(smem_dst)),
        "l"(gsrc), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

template <int R>
__global__ void __launch_bounds__(kThreads, 1) k_list_stream(const ListArgs a) {
    using C = Cfg<R>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_full[C::kStages], bar_empty[C::kStages], bar_acc_full[2], bar_acc_empty[2];
    __shared__ uint32_t s_tmem_base, s_abort;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // warp-uniform by construction
    const int lane = threadIdx.x & 31;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_al = smem_raw + (smem_base - smem_u32(smem_raw));

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kStages; ++s) {
            mbar_init(&bar_full[s], 1);
            mbar_init(&bar_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bar_acc_full[b], 1);
            mbar_init(&bar_acc_empty[b], 4);
        }
        s_abort = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(&s_tmem_base, C::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, s_tmem_base, 0);
    volatile uint32_t *abort_flag = &s_abort;

    // this CTA's piece of the line, and the layer it starts in
    const uint32_t grid = gridDim.x, cta = blockIdx.x;
    const uint32_t begin = (uint32_t)((uint64_t)a.total_kb * cta / grid);
    const uint32_t end = (uint32_t)((uint64_t)a.total_kb * (cta + 1) / grid);
    int first_layer = -1;
    for (int b = 0; b < a.n_layers; b += 32)
        first_layer += __popc(__ballot_sync(0xffffffffu, b + lane < a.n_layers && __ldg(&a.layers[b + lane].kb_first) <= begin));

    if (warp == 0) {
        // ------------------------------------------------------------ loader: W_q tiles by tensor map, codes block by block
        const uint32_t count = end - begin, pre = min(count, (uint32_t)C::kStages);
        Walk w;
        auto map_of = [&](int l) {
            const CUtensorMap *m = a.maps + l;
            // the maps were written by a copy before this launch; no older content of these addresses may be used
            asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(m) : "memory");
            return m;
        };
        // the weights of the first stages need nothing from the preparation of X
        w.start(a.layers, first_layer, begin);
        const CUtensorMap *map = map_of(w.l);
        for (uint32_t it = 0; it < pre; ++it) {
            mbar_expect_tx_elect(&bar_full[it], C::kStageBytes);
            tma_load_2d_elect(smem_al + it * C::kStageBytes, map, &bar_full[it], w.kb * kBK, w.tile * kTileN);
            if (++w.kb == w.nkb && it + 1 < count && w.next_tile()) map = map_of(w.l);
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("fence.proxy.async;" ::: "memory");  // the codes were written by ordinary stores
        auto codes_of = [&](int l) { return a.scratch + (size_t)__ldg(&a.layers[l].codes_off) * 128 + kHeaderBytes; };
        {
            Walk x;
            x.start(a.layers, first_layer, begin);
            const uint8_t *codes = codes_of(x.l);
            for (uint32_t it = 0; it < pre; ++it) {
                bulk_load_elect(smem_al + it * C::kStageBytes + C::kStageW, codes + (size_t)x.kb * C::kStageX, C::kStageX, &bar_full[it]);
                if (++x.kb == x.nkb && it + 1 < count && x.next_tile()) codes = codes_of(x.l);
            }
        }
        const uint8_t *codes = count > pre ? codes_of(w.l) : nullptr;
        uint32_t s = 0, ph = 0, it = pre;  // ph: parity of the use of stage s that has to be over
        bool ok = true;
        for (; it < count; ++it) {
            if (!mbar_wait_warp(&bar_empty[s], ph, abort_flag, a.spin)) { ok = false; break; }
            uint8_t *dst = smem_al + s * C::kStageBytes;
            mbar_expect_tx_elect(&bar_full[s], C::kStageBytes);
            tma_load_2d_elect(dst, map, &bar_full[s], w.kb * kBK, w.tile * kTileN);
            bulk_load_elect(dst + C::kStageW, codes + (size_t)w.kb * C::kStageX, C::kStageX, &bar_full[s]);
            if (++w.kb == w.nkb && it + 1 < count && w.next_tile()) {
                map = map_of(w.l);
                codes = codes_of(w.l);
            }
            if (++s == C::kStages) { s = 0; ph ^= 1u; }
        }
        if (!ok) {  // time-out: wait (bounded) until the copies issued so far have landed
            for (uint32_t j = it > (uint32_t)C::kStages ? it - C::kStages : 0u; j < it; ++j)
                for (uint32_t i = 0; i < a.spin; ++i)
                    if (__any_sync(0xffffffffu, mbar_try_wait(&bar_full[j % C::kStages], (j / C::kStages) & 1u))) break;
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        constexpr uint32_t idesc = idesc_i8(kTileN, 2 * R);
        const uint64_t w_desc0 = smem_desc_sw128(smem_base), x_desc0 = smem_desc_sw128(smem_base + C::kStageW);
        Walk w;
        w.start(a.layers, first_layer, begin);
        uint32_t s = 0, ph = 0, tiles_done = 0;
        bool ok = true;
        for (uint32_t pos = begin; pos < end && ok;) {
            const uint32_t buf = tiles_done & 1u;
            if (!mbar_wait_warp(&bar_acc_empty[buf], ((tiles_done >> 1) & 1u) ^ 1u, abort_flag, a.spin)) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + buf * C::kAccCols;
            const uint32_t n = min((uint32_t)(w.nkb - w.kb), end - pos);
            for (uint32_t i = 0; i < n; ++i) {
                if (!mbar_wait_warp(&bar_full[s], ph, abort_flag, a.spin)) { ok = false; break; }
                tc_fence_after();
                const uint64_t wd = w_desc0 + (uint64_t)(s * (C::kStageBytes >> 4)), xd = x_desc0 + (uint64_t)(s * (C::kStageBytes >> 4));
                mma_i8_ss_elect(d_tmem, wd, xd, idesc, i > 0 ? 1u : 0u);
                mma_i8_ss_elect(d_tmem, wd + 2, xd + 2, idesc, 1u);
                mma_i8_ss_elect(d_tmem, wd + 4, xd + 4, idesc, 1u);
                mma_i8_ss_elect(d_tmem, wd + 6, xd + 6, idesc, 1u);
                mma_commit_elect(&bar_empty[s]);
                if (++s == C::kStages) { s = 0; ph ^= 1u; }
            }
            if (!ok) break;
            mma_commit_elect(&bar_acc_full[buf]);
            ++tiles_done;
            pos += n;
            if (pos < end) w.next_tile();
        }
    } else {
        // ------------------------------------------------------------ epilogue: lane = output channel
        asm volatile("griddepcontrol.wait;" ::: "memory");  // scales and the cleared slots
        const int quad = warp & 3, row = quad * 32 + lane, M = a.M;
        Walk w;
        w.start(a.layers, first_layer, begin);
        uint32_t tiles_done = 0;
        for (uint32_t pos = begin; pos < end;) {
            const uint32_t buf = tiles_done & 1u;
            const uint32_t tile_begin = pos - (uint32_t)w.kb, tile_end = tile_begin + (uint32_t)w.nkb;
            const uint32_t n = min(tile_end, end) - pos;
            const ChainLayer *ly = a.layers + w.l;
            const float *scale = reinterpret_cast<const float *>(a.scratch + (size_t)__ldg(&ly->codes_off) * 128);
            const int ncol = w.tile * kTileN + row, N = __ldg(&ly->N), ldy = __ldg(&ly->ldy);
            void *Y = ly->Y;
            const bool live = ncol < N;
            const float *bias = ly->bias;
            const float sw = a.out_kind != gemm::kOutI32 ? __ldg(ly->s_w + (a.per_vec && live ? ncol : 0)) : 0.0f;
            const float bv = bias && live ? __ldg(bias + ncol) : 0.0f;
            // lane m mod 16 holds the scale of token row m: loads in the rows' own order would wait for the stores between them
            const float sx = a.out_kind != gemm::kOutI32 ? __ldcg(scale + (lane & 15)) : 0.0f;
            auto emit = [&](int m, int acc) {
                const float ss = __fmul_rn(__shfl_sync(0xffffffffu, sx, m), sw);  // Eq. 3
                if (!live) return;
                const size_t o = (size_t)m * ldy + ncol;
                if (a.out_kind == gemm::kOutI32) {
                    reinterpret_cast<int32_t *>(Y)[o] = acc;
                    return;
                }
                float y = __fmul_rn(ss, __int2float_rn(acc));
                if (bias) y = __fadd_rn(y, bv);
                if (a.out_kind == gemm::kOutF32) reinterpret_cast<float *>(Y)[o] = y;
                else reinterpret_cast<__half *>(Y)[o] = __float2half_rn(y);
            };
            if (!mbar_wait_warp(&bar_acc_full[buf], (tiles_done >> 1) & 1u, abort_flag, a.spin)) break;
            tc_fence_after();
            uint32_t v[2 * R];
            const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + buf * C::kAccCols;
            tmem_ld_32x16(taddr, v);
            if constexpr (R == 16) tmem_ld_32x16(taddr + 16, v + 16);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_acc_empty[buf]);
            if (tile_begin >= begin && tile_end <= end) {
#pragma unroll
                for (int m = 0; m < R; ++m)
                    if (m < M) emit(m, (int)v[m] + a.c * (int)v[R + m]);  // Eq. 7
            } else {
                // A tile shared with other CTAs; its slot is named after the first of them.  CTA x holds position p when
                // total * x / grid <= p < total * (x + 1) / grid (both rounded down).  Each of the four warps counts
                // itself in for its own 32 output channels, so that no warp waits for another one here.
                const uint32_t c0 = (uint32_t)((((uint64_t)tile_begin + 1) * grid - 1) / a.total_kb);
                const uint32_t c1 = (uint32_t)(((uint64_t)tile_end * grid - 1) / a.total_kb);
                int32_t *slot = a.fix + (size_t)c0 * M * kTileN + row;
#pragma unroll
                for (int m = 0; m < R; ++m)
                    if (m < M) atomicAdd(slot + m * kTileN, (int)v[m] + a.c * (int)v[R + m]);
                __threadfence();
                __syncwarp();
                uint32_t before = 0;
                if (lane == 0) before = atomicAdd(a.fix_count + 4 * c0 + quad, 1u);
                if (__shfl_sync(0xffffffffu, before, 0) == c1 - c0) {  // every part is in
                    __threadfence();
                    int32_t acc[R];
#pragma unroll
                    for (int m = 0; m < R; ++m) acc[m] = m < M ? __ldcg(slot + m * kTileN) : 0;
#pragma unroll
                    for (int m = 0; m < R; ++m)
                        if (m < M) emit(m, acc[m]);
                }
            }
            ++tiles_done;
            pos += n;
            if (pos < end) w.next_tile();
        }
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, C::kTmemCols);
    }
    if (threadIdx.x == 0 && s_abort && a.dev_status) atomicMax(a.dev_status, kStatusTimeout);
}

template <int R, int U>
cudaError_t launch_list_inst(const ListArgs &a, cudaStream_t s) {
    using C = Cfg<R>;
    static PerDevice<int> attr_set;
    const int dev = current_device();
    if (dev < 0) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(device_mutex());
        if (!attr_set.have[dev]) {
            cudaError_t e = cudaFuncSetAttribute(k_list_stream<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
            if (e != cudaSuccess) return e;
            attr_set.have[dev] = true;
        }
    }
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg{};
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(kPrepCtas, a.n_layers);
    cfg.blockDim = dim3(kPrepThreads);
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = kPrepCtas; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_list_prep<U>, a);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3(a.grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = C::kSmemBytes;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_list_stream<R>, a);
}

}  // namespace

size_t list_layer_bytes(int M, int K) { return layer_scratch_bytes(code_rows(M), K); }

size_t list_sync_bytes(int M) { return (size_t)kListMaxCtas * (16 + (size_t)M * kTileN * 4); }

bool list_map(void *map128, const int8_t *w_q, int N, int K, int ldw) {
    CUtensorMap m;
    if (!gemm::make_map_i8(&m, w_q, (uint64_t)N, (uint64_t)K, (uint64_t)ldw, kTileN)) return false;
    static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
    memcpy(map128, &m, sizeof m);
    return true;
}

uint32_t list_plan(ChainLayer *layers, int n_layers, int M) {
    uint64_t kb = 0, off = 0;
    for (int l = 0; l < n_layers; ++l) {
        layers[l].kb_first = (uint32_t)kb;
        layers[l].codes_off = (uint32_t)(off / 128);
        kb += (uint64_t)((layers[l].K + kBK - 1) / kBK) * ((layers[l].N + (uint64_t)kTileN - 1) / kTileN);
        off += list_layer_bytes(M, layers[l].K);
        if (kb > 0x7FFFFFFFu) return 0;
    }
    return (uint32_t)kb;
}

cudaError_t launch_decode_list(const ListArgs &a, cudaStream_t s) {
    if (a.M <= 4) return launch_list_inst<8, 1>(a, s);
    if (a.M <= 8) return launch_list_inst<8, 2>(a, s);
    return launch_list_inst<16, 4>(a, s);
}

}  // namespace muxq
