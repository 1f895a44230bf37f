// K4, fused form: shared-memory layout and choice of the kernel (k4f_decode_fused.cuh, k4r_decode_row.cu) for a layer.
#include "k4f_common.cuh"
#include "ptx.cuh"

namespace muxq {

using namespace decode;

namespace {

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
    // 14.6 us with one from 64 KB on, 12.6 without); else a ring
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
    // One CTA per SM, the reporting one included: a grid of more would put two CTAs of the same layer on some SM (the next
    // layer's take every SM's second place) and that SM would set the pace.
    const int workers = a.N < sms ? a.N : sms - 1, rows = (a.N + workers - 1) / workers;
    // Token rows of the instantiation.  M = 9..12 have a form of their own where X is wide and the layer fills an SM: it saves a quarter
    // of what is read twice (8192 x 2048 at M = 12 21.4 -> 19.2 us; with all of X in registers the form for 16 rows is as fast or
    // faster, 768 x 768 4.2 against 4.4 us).
    int MT = a.M <= 2 ? a.M : a.M <= 4 ? 4 : a.M <= 8 ? 8 : 16;
    Geometry geo = geometry(MT, a.K, rows);
    // (the forms with more registers keep other layers' CTAs away, so they are for layers that do so anyway: a step of 12 blocks of width
    // 1280 at M = 16 469 us with them at 5120 -> 1280, 416 with the form of two slices before)
    const bool alone = geo.total > kBesideSmem;
    if (MT == 16 && a.M <= 12 && alone && a.K > channels_of(16, 2)) {
        MT = 12;
        geo = geometry(MT, a.K, rows);
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
        return launch_row(a, cfg, dev);
    }
    // lanes per row of W_q: as many as let every row of the CTA (of a chunk) be worked on at once
    const int r = geo.rows < rows ? geo.rows : rows, lanes = r <= kWarps ? 2 : r <= 2 * kWarps ? 1 : 0;
    switch (MT) {
        case 1: return launch_rows<1>(a, geo, cfg, lanes, alone, dev);
        case 2: return launch_rows<2>(a, geo, cfg, lanes, alone, dev);
        case 4: return launch_rows<4>(a, geo, cfg, lanes, alone, dev);
        case 8: return launch_rows<8>(a, geo, cfg, lanes, alone, dev);
        case 12: return launch_rows<12>(a, geo, cfg, lanes, alone, dev);
        default: return launch_rows<16>(a, geo, cfg, lanes, alone, dev);
    }
}

}  // namespace muxq
