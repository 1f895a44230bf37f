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
#include "k9_prep_rows.cuh"

namespace muxq {

using namespace prep_rows;

namespace {

__global__ void __launch_bounds__(kT, 2) k_channel_max(const PrepArgs a, int stripes, int width, int slices, int first_rows) {
    __shared__ uint4 s_part[kWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int stripe = blockIdx.x % stripes, slice = blockIdx.x / stripes;
    const int g = stripe * width + lane, G = a.K >> 3;
    const bool on = lane < width && g < G;
    const int step = slices * kWarps;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // behind the wait: the dependent may read X at once
    uint32_t mark = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) mark = __ldcg(&a.ctrl->arrived) & kPrepPoisonBit;
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
    // An earlier call on this workspace timed out and left half-merged maxima: said to every CTA of k_quant_rows by a maximum that
    // no input has (reading the mark there, 300 CTAs of 16 warps beside the tickets, cost 0.7 us per call).
    if (mark) atomicMax(a.colmax_rep, kMarkedMaximum);
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
