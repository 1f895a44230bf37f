// Choice of the clusters and launch of k_short (k10_short.cuh).
#include "k10_short.cuh"

namespace muxq {

using namespace shorts;

namespace {

using Fn = void (*)(const CUtensorMap, const Args, const Plan);

constexpr int kMaxSmem = 216 * 1024;
// beyond 16 rows as many chunks a thread as there are, or eight at a time; up to 16 rows no more than four
const Fn fns[6] = {k_short<2, true, true>, k_short<4, true, true>, k_short<8, true, true>, k_short<8, false, true>,
                   k_short<2, true, false>, k_short<4, true, false>};

cudaError_t set_up_form(int i, int dev) {
    static PerDevice<int> done[6];
    std::lock_guard<std::mutex> lock(device_mutex());
    if (done[i].have[dev]) return cudaSuccess;
    // (one split of L1 for every layer kernel: k4f_common.cuh)
    cudaError_t e = cudaFuncSetAttribute(fns[i], cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fns[i], cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    done[i].have[dev] = e == cudaSuccess;
    return e;
}

// Shared memory, threads and tensor memory for clusters of `ranks` CTAs, of which `most` fit on the device, one of them for the
// reports; false: does not fit.
bool make_plan(Plan *g, int M, int K, int N, int ranks, int most) {
    const int steps = (K + 31) / 32;
    if (ranks > steps || most < 2) return false;
    g->ranks = ranks;
    g->kc = (steps + ranks - 1) / ranks * 32;
    g->kb = (g->kc + 127) / 128;
    g->bn = ((N + most - 2) / (most - 1) + 15) & ~15;
    if (g->kc > kMaxKc || g->bn > 256) return false;
    g->clusters = (N + g->bn - 1) / g->bn;
    g->mr = (M + 7) & ~7;
    g->rows = (M + ranks - 1) / ranks;
    g->pitch = (g->rows | 1) * 16;
    g->chunks = g->kc / 8;
    g->groups = kT / g->chunks < M ? kT / g->chunks : M;
    const int block = g->mr * 128, codes = g->kb * block;  // the copy stands behind the rows of a block (M <= 16), else behind all blocks
    g->a_block = M <= 16 ? 2 * block : block;
    g->off_m = M <= 16 ? block : codes;
    g->off_w = 2 * codes > kT * 16 ? 2 * codes : kT * 16;
    g->off_p = g->off_w + g->kb * g->bn * 128;
    g->total = g->off_p + ranks * (g->bn / 4) * g->pitch;
    const int read = (M <= 16 ? 0 : g->off_m) + (g->kb - 1) * g->a_block + gemm::BM * 128;  // the products read 128 rows whatever M is
    if (g->total < read) g->total = read;
    g->total += 1024;
    for (g->line_shift = 5; (1 << g->line_shift) < M; ++g->line_shift) {}
    for (g->cols = 32; g->cols < g->bn; g->cols *= 2) {}
    return g->total <= kMaxSmem;
}

// Clusters of `ranks` CTAs that fit on the device, one CTA per SM.
int most_clusters(int ranks, int dev) {
    static PerDevice<int> cache[kMaxRanks + 1];
    std::lock_guard<std::mutex> lock(device_mutex());
    PerDevice<int> &c = cache[ranks];
    if (!c.have[dev]) {
        cudaLaunchConfig_t q{};
        q.gridDim = dim3(ranks * 64);
        q.blockDim = dim3(kT);
        q.dynamicSmemBytes = 120 * 1024;
        cudaLaunchAttribute qa[1];
        qa[0].id = cudaLaunchAttributeClusterDimension;
        qa[0].val.clusterDim.x = ranks; qa[0].val.clusterDim.y = 1; qa[0].val.clusterDim.z = 1;
        q.attrs = qa;
        q.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, fns[0], &q) != cudaSuccess) return 0;
        c.v[dev] = n;
        c.have[dev] = true;
    }
    return c.v[dev];
}

// Microseconds of a layer in a row of layers, fitted to 780 measured forms (M = 2..128, K = 400..6144, N = 400..5120, both
// granularities): a clear chain of latencies, quantization by rows x channels of a CTA, the partial sums' way through the
// cluster, the products.  5.5 % rms for the clusters it chooses, 9 % over 2284 forms of 968 layers (M = 17..128, K = 64..8192, N =
// 192..16384) with clusters of every size, of which it misses the best size by 0.7 % of the time on average.
double cost(const Plan &g, int M, bool per_vec) {
    const double slice = 1e-4 * M * g.kc, sums = 1e-4 * M * g.bn * (g.ranks - 1) / g.ranks;
    return 3.5 + (M > 16 ? 0.8 : 0.0) + 0.0065 * M + 1.1 * slice + 2.0 * sums + 0.0025 * g.kc + 0.0095 * g.bn + (per_vec ? 1.3 + 0.65 * slice : 0.0);
}

// The same for the three launches beyond 16 rows (7.6 % rms).
double cost_without(int M, int K, int N, bool per_vec) {
    const double k = 1e-3 * K, n = 1e-3 * N;
    return 7.4 + 1.5 * k + 0.85 * n + 0.005 * M + 1.2e-3 * M * k - 1.5e-3 * M * n + (per_vec ? 0.45 : 0.0);
}

// Clusters of 8, 4 or 2: larger ones have less to quantize per CTA and more partial sums to send.  Rows of one layer, us, without ->
// here (clusters of): 16 x 3072 x 768 8.7 -> 5.0 (8), 16 x 5120 x 1280 13.9 -> 6.4 (8), 32 x 768 x 768 9.1 -> 5.5 (8), 32 x 1280 x 5120
// 13.3 -> 8.7 (4), 64 x 1280 x 1280 10.6 -> 7.9 (8), 128 x 768 x 768 9.6 -> 8.6 (8); left to the others: 128 x 1280 x 3840 13.4 against
// 13.9, 128 x 768 x 768 per token 9.8 against 10.8.
bool choose(Plan *best, int M, int K, int N, bool per_vec, int dev, double *us) {
    bool found = false;
    for (const int ranks : {8, 4, 2}) {
        Plan g;
        if (!make_plan(&g, M, K, N, ranks, most_clusters(ranks, dev))) continue;
        const double c = cost(g, M, per_vec);
        if (found && c >= *us) continue;
        *best = g;
        *us = c;
        found = true;
    }
    return found;
}

}  // namespace

// Beyond 16 rows by the two estimates; one launch instead of three is the better one for the host too, so it is taken where both are
// even, but for two kinds of layers whose estimates are off: per token with three or four chunks a thread in clusters of four (of 35
// such layers next to the line 18 were slower here, us, three launches / here: 96 x 640 -> 2560 9.8 / 11.6, 80 x 768 -> 2304 9.8 / 11.2), and few
// output channels behind many input channels, which leaves most of the device idle (113 x 4688 -> 616 per token 17.5 / 22.0, 72 x 6288 -> 280
// 14.5 / 17.5).  Of 968 layers (M = 17..128, K = 64..8192, N = 192..16384) 858 are taken, 19 of them slower here, by 6 % on average (42 of 895 without these two lines).  Up to 16 rows it is the blocks of a model that count, not rows of one layer: launches of clusters and of k_decode_fused in turn
// cost more than either alone (a step of 12 blocks of width 768 at M = 16, us a layer: all of them here 5.1, the long-K layers only
// 5.9, none 5.7), so the line is drawn by the smaller side of the layer, which is the same for all four of a block.  A layer in such
// steps, captured (as plain calls), without -> here, us: per tensor width 1280 M = 16 8.1 -> 5.6 (8.5 -> 6.2), M = 5 6.4 -> 5.0 (6.7 -> 5.7), 1024 M = 16
// 6.6 -> 4.8 (6.9 -> 5.4), 768 M = 12 5.5 -> 4.5 (5.8 -> 5.0); per token 1280 M = 12 8.4 -> 6.9 (8.7 -> 7.4).  The lines were drawn when outlier
// channels cost c more products here; since they do not, layers left to k_decode_fused next to the lines would gain as well: 1024 M = 8 5.25 -> 4.5,
// 768 M = 8 4.7 -> 4.3, 512 M = 12 4.4 -> 3.9, per token 1280 M = 8 6.9 -> 6.4, 1024 M = 16 7.1 -> 6.7.
// Fewer than 192 output channels stay out: most of the device would be idle (100 x 5120 -> 136: 13.5 us either way, 128 rows 13.7 and 15.1).
bool short_preferred(int M, int K, int N, bool per_vec) {
    if (M < 5 || M > kMaxM || K > kPrepMaxK || N < 192) return false;
    const int width = K < N ? K : N;
    if (M <= 16 && (per_vec ? M <= 8 || width < 1152 : width < (M > 8 ? 640 : 1152))) return false;
    const int dev = current_device();
    if (dev < 0 || set_up_form(0, dev) != cudaSuccess) return false;
    Plan g;
    double us = 0.0;
    if (!choose(&g, M, K, N, per_vec, dev, &us)) return false;
    if (M <= 16) return true;
    const int iters = (M + g.groups - 1) / g.groups;
    const double line = per_vec && g.ranks == 4 && iters > 2 && iters <= 4 ? 0.935 : K >= 8 * N && iters > 4 ? 0.9 : 1.03;
    return us < line * cost_without(M, K, N, per_vec);
}

cudaError_t launch_short(const DecodeFusedArgs &a, const ShortOut &out, cudaStream_t s) {
    const int dev = current_device();
    if (dev < 0) return cudaErrorInvalidDevice;
    Plan g;
    double us = 0.0;
    if (!choose(&g, a.M, a.K, a.N, a.per_vec, dev, &us)) return cudaErrorInvalidValue;
    g.skip = test_hooks().gemm_skip_kb - 1;
    g.late = test_hooks().short_late_warps;
    Args arg{a, out};
    arg.d.spin = test_hooks().spin_limit ? test_hooks().spin_limit : kSpinLimit;
    CUtensorMap map;
    if (!gemm::make_map_i8(&map, a.w_q, a.N, a.K, a.ldw, g.bn)) return cudaErrorInvalidValue;
    const int iters = (a.M + g.groups - 1) / g.groups, i = a.M <= 16 ? (iters <= 2 ? 4 : 5) : iters <= 2 ? 0 : iters <= 4 ? 1 : iters <= 8 ? 2 : 3;
    const cudaError_t e = set_up_form(i, dev);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((g.clusters + 1) * g.ranks);
    cfg.blockDim = dim3(kT);
    cfg.dynamicSmemBytes = (size_t)(g.total < decode::kMinSmem ? decode::kMinSmem : g.total);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = g.ranks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, fns[i], map, arg, g);
}

}  // namespace muxq
