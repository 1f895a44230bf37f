"""GPU parity: every stage of the CUDA path (through the C-ABI binding) against the CPU oracle on
the same seeded inputs.  Integer results (codes, accumulators, outlier sets) and fp32 scales must
match bit for bit; fp32 outputs within 1e-5 relative; fp16 outputs within 1 ulp."""
import numpy as np
import pytest

import muxq_synth as synth
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2604_04701_b200 as m
    m.lib()
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def f16_ulp_diff(a, b):
    """Distance in units of fp16 spacing between two float16 arrays (as ordered integers)."""
    def key(x):
        u = x.view(np.uint16).astype(np.int32)
        return np.where(u & 0x8000, -(u & 0x7FFF), u)
    return np.abs(key(a) - key(b))


def rel_err32(y, ref):
    den = np.maximum(np.abs(ref), 1e-6 * np.abs(ref).max())
    return (np.abs(y.astype(np.float64) - ref.astype(np.float64)) / den).max()


def make_case(seed, M, K, N, n_out=4, mult=50.0, bulk="normal", bulk_scale=1.0):
    x, ch = synth.make_x(seed, 3, M, K, n_out, mult, mult, bulk, bulk_scale)
    w = synth.make_w(seed, 3, K, N)
    return x, w, ch


def run_linear(mx, x, w, p, out_kind, rows=None):
    """GPU: quantize W, run the layer; returns (Y, workspace tensors) and oracle result."""
    M, K = x.shape
    N = w.shape[1]
    wsw = mx.Workspace(mx.muxq_small_workspace_bytes(N))
    w_q, s_w = mx.muxq_quantize(dev(w), p, True, wsw)
    ws = mx.Workspace(mx.muxq_workspace_bytes(M, K, N, p))
    ws.buf.fill_(0xA5)  # everything but the words muxq_workspace_init prepares may hold garbage
    ws.init()
    y = mx.muxq_linear(dev(x), w_q, s_w, p, ws, out_kind)
    st = mx.muxq_read_status(ws)
    return y, ws, st, w_q, s_w


def oracle_linear(x, w, p, rows=None):
    per_vec = p.gran == 1
    wq, sw = oracle.quantize_weight(w, bits=p.w_bits, per_channel=per_vec)
    res = oracle.linear(x, wq, sw, tau=p.threshold, e=p.exp_factor, act_bits=p.act_bits, per_vector=per_vec,
                        cap=p.max_outliers, rows=rows)
    return wq, sw, res


def ws_views(mx, ws, M, K, N, p):
    v = mx.muxq_workspace_view(M, K, N, p)
    b = ws.buf.cpu().numpy()
    cap = p.max_outliers
    out = {
        "col_absmax": b[v.col_absmax: v.col_absmax + 4 * K].view(np.float32),
        "outlier_idx": b[v.outlier_idx: v.outlier_idx + 4 * cap].view(np.int32),
        "n_outliers": int(b[v.n_outliers: v.n_outliers + 4].view(np.int32)[0]),
        "s_x": b[v.s_x: v.s_x + 4 * (M if p.gran == 1 else 1)].view(np.float32),
        "body_q": b[v.body_q: v.body_q + M * v.ld_body_q].view(np.int8).reshape(M, v.ld_body_q)[:, :K],
        "aux_q": b[v.aux_q: v.aux_q + M * v.aux_cols].view(np.int8).reshape(M, v.aux_cols),
        "w_aux": b[v.w_aux: v.w_aux + N * v.aux_cols].view(np.int8).reshape(N, v.aux_cols),
    }
    return out


# ------------------------------------------------------------------ K1
@pytest.mark.parametrize("M,K", [(128, 768), (1, 1280), (333, 1040), (4096, 3072), (37, 16)])
def test_detect_matches_oracle(mx, M, K):
    x, _, ch = make_case(10 + M, M, K, 8, n_out=min(5, K // 4))
    x[0, 0] = 6.0  # exactly the threshold somewhere: must not flag by itself
    cap = 64
    ws = mx.Workspace(mx.muxq_small_workspace_bytes(K))
    ws.buf.fill_(0x5A)
    cm, idx, n = mx.muxq_detect_outliers(dev(x), 6.0, cap, ws)
    cm_o = oracle.colmax(x)
    O, r, _ = oracle.detect(cm_o, 6.0, cap)
    assert np.array_equal(cm.cpu().numpy().view(np.uint32), cm_o.view(np.uint32))
    assert int(n.item()) == r
    assert np.array_equal(idx.cpu().numpy()[:min(r, cap)], O)


def test_detect_pitched_input_and_capacity_overflow(mx):
    M, K, ld = 64, 256, 320
    x, _, _ = make_case(5, M, K, 8, n_out=12)
    xp = torch.zeros(M, ld, dtype=torch.float16, device="cuda")
    xp[:, :K] = dev(x)
    xp[:, K:] = 1000.0  # padding beyond K must be ignored
    ws = mx.Workspace(mx.muxq_small_workspace_bytes(K))
    cm, idx, n = mx.muxq_detect_outliers(xp[:, :K], 6.0, 4, ws)
    cm_o = oracle.colmax(x)
    O, r, rc = oracle.detect(cm_o, 6.0, 4)
    assert rc == oracle.ERR_CAPACITY and r >= 12
    assert int(n.item()) == r and np.array_equal(idx.cpu().numpy(), O)
    assert np.array_equal(cm.cpu().numpy(), cm_o)


# ------------------------------------------------------------------ Eq. 4-5 in the real domain
def test_build_aux_reconstructs_x(mx):
    x, _, _ = make_case(6, 200, 512, 8, n_out=6, mult=70.0)
    ws = mx.Workspace(mx.muxq_small_workspace_bytes(512))
    xd = dev(x)
    cm, idx, n = mx.muxq_detect_outliers(xd, 6.0, 16, ws)
    for e in (1, 2, 3):
        aux, body = mx.muxq_build_aux(xd, idx, n, e)
        O, r, _ = oracle.detect(oracle.colmax(x), 6.0, 16)
        body_o, aux_o = oracle.decompose(x, O, e)
        assert np.array_equal(body.cpu().numpy(), body_o)
        a = aux.cpu().numpy()
        assert np.array_equal(a[:, :r], aux_o) and not a[:, r:].any()
        recon = body_o.copy()
        recon[:, O] = body.cpu().numpy()[:, O] + np.float32(2 ** e - 1) * a[:, :r]   # Eq. 6
        assert np.array_equal(recon, x.astype(np.float32))


# ------------------------------------------------------------------ K5 / K2
@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("K,N,bits", [(768, 768, 8), (1040, 200, 8), (512, 264, 5)])
def test_weight_quantization_matches_oracle(mx, gran, K, N, bits):
    w = synth.make_w(7, K * 3 + N, K, N)
    p = mx.MuxqParams(gran=gran, w_bits=bits)
    ws = mx.Workspace(mx.muxq_small_workspace_bytes(N))
    ws.buf.fill_(0x33)
    w_q, s_w = mx.muxq_quantize(dev(w), p, True, ws)
    wq_o, sw_o = oracle.quantize_weight(w, bits=bits, per_channel=bool(gran))
    assert np.array_equal(s_w.cpu().numpy().view(np.uint32), sw_o.view(np.uint32))
    assert np.array_equal(w_q.cpu().numpy(), wq_o.T)


@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("K,N,ld,zero_col", [
    (1, 8, 8, False), (16, 64, 64, True), (33, 72, 80, False), (128, 8, 8, False), (136, 200, 200, True),
    (1280, 1288, 1296, True), (5120, 136, 136, False), (12800, 8, 8, False), (12816, 72, 72, False)])
def test_weight_quantization_tile_edges(mx, gran, K, N, ld, zero_col):
    """One output channel group, K tails below 16, stripes and slices that end inside a tile, pitched W, rows of W_q that
    are not 16-byte aligned, an all-zero output channel, and K on both sides of what a cluster's shared memory holds."""
    w = np.zeros((K, ld), np.float16)
    w[:, :N] = synth.make_w(8, K * 5 + N, K, N)
    w[:, N:] = 100.0   # behind the matrix: must not be read
    if zero_col:
        w[:, N - 3] = 0
    p = mx.MuxqParams(gran=gran)
    ws = mx.Workspace(mx.muxq_small_workspace_bytes(N))
    ws.buf.fill_(0x77)
    w_q, s_w = mx.muxq_quantize(dev(w)[:, :N], p, True, ws)
    wq_o, sw_o = oracle.quantize_weight(np.ascontiguousarray(w[:, :N]), bits=8, per_channel=bool(gran))
    assert np.array_equal(s_w.cpu().numpy().view(np.uint32), sw_o.view(np.uint32))
    assert np.array_equal(w_q.cpu().numpy(), wq_o.T)


@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("M,K,e,bits", [(128, 768, 2, 8), (77, 1040, 2, 8), (300, 512, 3, 6), (64, 256, 1, 8)])
def test_activation_quantization_matches_oracle(mx, gran, M, K, e, bits):
    x, _, _ = make_case(20 + M, M, K, 8, n_out=5, mult=60.0)
    x[3] = 0  # an all-zero token row (per-token scale must become 1)
    p = mx.MuxqParams(gran=gran, exp_factor=e, act_bits=bits, max_outliers=16)
    ws = mx.Workspace(mx.muxq_small_workspace_bytes(K))
    xd = dev(x)
    cm, idx, n = mx.muxq_detect_outliers(xd, p.threshold, p.max_outliers, ws)
    body_q, aux_q, s_x = mx.muxq_quantize(xd, p, False, ws, cm, idx, n)
    O, r, _ = oracle.detect(oracle.colmax(x), 6.0, 16)
    body, aux = oracle.decompose(x, O, e)
    sx_o, sa_o, bq_o, aq_o = oracle.quantize_act(body, aux, bits, bool(gran), False)
    assert np.array_equal(s_x.cpu().numpy().view(np.uint32), sx_o.view(np.uint32))
    assert np.array_equal(body_q.cpu().numpy(), bq_o)
    c = 2 ** e - 1
    a = aux_q.cpu().numpy()
    assert a.shape[1] == mx.muxq_aux_cols(p)
    for j in range(r):
        for t in range(c):
            assert np.array_equal(a[:, c * j + t], aq_o[:, j])
    assert not a[:, c * r:].any()
    # naive quantization (no outlier handling): Eq. 1 alone
    nq, _, ns = mx.muxq_quantize(xd, p, False, ws, cm, None, None, want_aux=False)
    sx_n, _, bq_n, _ = oracle.quantize_act(x.astype(np.float32), np.zeros((M, 0), np.float32), bits, bool(gran), False)
    assert np.array_equal(ns.cpu().numpy(), sx_n) and np.array_equal(nq.cpu().numpy(), bq_n)


def test_quantization_ties_round_half_even(mx):
    """Scale 0.25 exactly and inputs on multiples of 0.125: every other value is an exact .5 tie."""
    M, K = 64, 256
    rng = np.random.default_rng(3)
    x = (rng.integers(-100, 101, (M, K)) * 0.125).astype(np.float16)
    x[0, 7] = 31.75  # abs-max -> s = 31.75 / 127 = 0.25
    p = mx.MuxqParams(threshold=1e4)
    ws = mx.Workspace(mx.muxq_small_workspace_bytes(K))
    xd = dev(x)
    cm, idx, n = mx.muxq_detect_outliers(xd, p.threshold, p.max_outliers, ws)
    body_q, _, s_x = mx.muxq_quantize(xd, p, False, ws, cm, idx, n, want_aux=False)
    assert s_x.item() == 0.25
    ref = np.rint(x.astype(np.float32) / np.float32(0.25)).astype(np.int8)  # numpy rint is half-to-even
    assert (np.abs(x.astype(np.float32) / 0.25 % 1.0) == 0.5).sum() > 1000
    assert np.array_equal(body_q.cpu().numpy(), ref)
    for gran in (0, 1):
        sx_o, _, bq_o, _ = oracle.quantize_act(x.astype(np.float32), np.zeros((M, 0), np.float32), 8, bool(gran), False)
        pq = mx.MuxqParams(threshold=1e4, gran=gran)
        bq, _, sx = mx.muxq_quantize(xd, pq, False, ws, cm, idx, n, want_aux=False)
        assert np.array_equal(sx.cpu().numpy(), sx_o) and np.array_equal(bq.cpu().numpy(), bq_o)


# ------------------------------------------------------------------ K3 alone
@pytest.mark.parametrize("M,K,N", [(128, 128, 128), (128, 256, 256), (256, 768, 768), (300, 1040, 520),
                                   (1000, 512, 1288), (128, 32, 64), (129, 4096, 264)])
def test_gemm_accumulators_bit_exact(mx, M, K, N):
    rng = np.random.default_rng(M * 7 + K + N)
    a = rng.integers(-127, 128, (M, K), dtype=np.int8)
    b = rng.integers(-127, 128, (N, K), dtype=np.int8)
    p = mx.MuxqParams()
    ws = mx.Workspace(256)
    acc = mx.muxq_gemm(dev(a), None, dev(b), None, None, p, None, None, mx.MUXQ_OUT_ACC_I32, ws)
    assert mx.muxq_read_status(ws) == 0
    ref = a.astype(np.int32) @ b.astype(np.int32).T
    assert np.array_equal(acc.cpu().numpy(), ref)


def test_gemm_worst_case_magnitudes(mx):
    M, K, N = 128, 5120, 256
    a = np.full((M, K), 127, np.int8)
    b = np.full((N, K), -127, np.int8)
    b[::2] = 127
    acc = mx.muxq_gemm(dev(a), None, dev(b), None, None, mx.MuxqParams(), None, None, 2, mx.Workspace(256))
    ref = a.astype(np.int32) @ b.astype(np.int32).T
    assert np.array_equal(acc.cpu().numpy(), ref)
    assert np.abs(ref).max() > 2 ** 24  # int32 -> fp32 must round (to nearest even) here
    sx = np.array([0.0123], np.float32); sw = np.array([0.00071], np.float32)
    y = mx.muxq_gemm(dev(a), None, dev(b), None, None, mx.MuxqParams(), dev(sx), dev(sw), 1, mx.Workspace(256))
    assert np.array_equal(y.cpu().numpy(), (sx * sw) * ref.astype(np.float32))
    # odd magnitudes above 2^24 exercise the rounding itself
    a[:, :7] = 1; b[:, :7] = 1
    b[1::2, 7] = 3
    ref = a.astype(np.int32) @ b.astype(np.int32).T
    y = mx.muxq_gemm(dev(a), None, dev(b), None, None, mx.MuxqParams(), dev(sx), dev(sw), 1, mx.Workspace(256))
    assert np.array_equal(y.cpu().numpy(), (sx * sw) * ref.astype(np.float32))
    y16 = mx.muxq_gemm(dev(a), None, dev(b), None, None, mx.MuxqParams(), dev(sx), dev(sw), 0, mx.Workspace(256))
    with np.errstate(over="ignore"):
        assert np.array_equal(y16.cpu().numpy(), ((sx * sw) * ref.astype(np.float32)).astype(np.float16))


@pytest.mark.parametrize("M,K,N", [(8192, 128, 2304), (8192, 256, 768), (8192, 128, 2048)])
def test_gemm_several_tiles_per_cta_pair_full_matrix(mx, M, K, N):
    """Full-matrix check of the persistent loop beyond its first tile: 288 / 128 / 256 output tiles over 74 CTA
    pairs give every pair 2 to 4 tiles, so the flip between the two TMEM accumulator buffers, the phase wrap of
    their barriers and the operand ring running on across tiles all decide values that are compared here.  The
    reference is a float32 matrix product: every partial sum stays below 2^24, so it is exact."""
    rng = np.random.default_rng(M + 3 * K + N)
    a = rng.integers(-127, 128, (M, K), dtype=np.int8)
    b = rng.integers(-127, 128, (N, K), dtype=np.int8)
    assert 127 * 127 * K < 2 ** 24
    ref = (a.astype(np.float32) @ b.astype(np.float32).T).astype(np.int32)
    ws = mx.Workspace(256)
    acc = mx.muxq_gemm(dev(a), None, dev(b), None, None, mx.MuxqParams(), None, None, mx.MUXQ_OUT_ACC_I32, ws)
    assert mx.muxq_read_status(ws) == 0
    assert np.array_equal(acc.cpu().numpy(), ref)


@pytest.mark.parametrize("gran", [0, 1])
def test_linear_several_tiles_per_cta_pair_full_matrix(mx, gran):
    """The same through the whole layer with an Aux block (K = 256, 6 outlier channels, 288 output tiles):
    every accumulator and every output of the 8192 x 2304 result against the oracle."""
    M, K, N = 8192, 256, 2304
    x, w, _ = make_case(77, M, K, N, n_out=6, mult=50.0)
    p = mx.MuxqParams(gran=gran, max_outliers=32)
    _, _, res = oracle_linear(x, w, p)
    assert res.r >= 6
    acc, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0 and np.array_equal(acc.cpu().numpy(), res.acc)
    y16, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F16)
    assert st == 0 and f16_ulp_diff(y16.cpu().numpy(), res.y16).max() <= 1
    y32, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F32)
    assert st == 0 and np.array_equal(y32.cpu().numpy(), res.y32)


# ------------------------------------------------------------------ whole layer
@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("M,K,N,n_out", [(128, 768, 768, 4), (300, 1040, 520, 7), (512, 256, 1288, 0),
                                         (1024, 1280, 1280, 21)])
def test_linear_matches_oracle(mx, gran, M, K, N, n_out):
    x, w, ch = make_case(40 + M, M, K, N, n_out=n_out, mult=50.0)
    p = mx.MuxqParams(gran=gran, max_outliers=32)
    wq_o, sw_o, res = oracle_linear(x, w, p)
    assert res.r >= n_out
    # raw accumulators
    acc, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0
    v = ws_views(mx, ws, M, K, N, p)
    assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O)
    assert np.array_equal(v["col_absmax"].view(np.uint32), res.colmax.view(np.uint32))
    assert np.array_equal(v["s_x"].view(np.uint32), res.s_x.view(np.uint32))
    assert np.array_equal(v["body_q"], res.body_q)
    assert np.array_equal(w_q.cpu().numpy(), wq_o.T)
    c = 3
    for j in range(res.r):
        assert np.array_equal(v["w_aux"][:, c * j], wq_o[res.O[j]])
        assert np.array_equal(v["aux_q"][:, c * j + 2], res.aux_q[:, j])
    assert np.array_equal(acc.cpu().numpy(), res.acc)
    # fp32 and fp16 outputs
    y32, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F32)
    assert st == 0 and rel_err32(y32.cpu().numpy(), res.y32) <= 1e-5
    assert np.array_equal(y32.cpu().numpy(), res.y32)  # same operands, same two roundings
    y16, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F16)
    assert st == 0 and f16_ulp_diff(y16.cpu().numpy(), res.y16).max() <= 1


@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("M,K,N,n_out,cap", [
    (17, 16, 24, 1, 4), (33, 256, 136, 3, 8), (47, 528, 64, 0, 8), (35, 1024, 64, 5, 8), (40, 1280, 72, 8, 16),   # a warp per row, up to its last chunk
    (40, 1296, 72, 8, 16), (60, 2048, 72, 4, 16), (300, 2560, 136, 9, 16),                                         # two warps
    (20, 2576, 72, 5, 16), (33, 3088, 64, 3, 16), (700, 5120, 64, 8, 16), (33, 5136, 64, 8, 16), (19, 8192, 64, 20, 64),   # four
    (50, 1040, 72, 100, 128), (21, 5120, 72, 150, 256)])                                    # more Aux codes than a row stages
def test_preparation_row_groups(mx, gran, M, K, N, n_out, cap):
    """Codes, Aux block, W_aux, O, scales and accumulators at the edges of the row kernel's warps-per-row choice; the
    workspace's accumulators are zero again (a second call gives the same bits)."""
    x, w, _ = make_case(90 + M + K, M, K, N, n_out=n_out, mult=60.0)
    x[M // 2] = 0
    p = mx.MuxqParams(gran=gran, max_outliers=cap)
    wq_o, sw_o, res = oracle_linear(x, w, p)
    assert res.r <= cap
    acc, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0
    for _ in range(2):
        v = ws_views(mx, ws, M, K, N, p)
        assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O)
        assert np.array_equal(v["col_absmax"].view(np.uint32), res.colmax.view(np.uint32))
        assert np.array_equal(v["s_x"].view(np.uint32), res.s_x.view(np.uint32))
        assert np.array_equal(v["body_q"], res.body_q)
        pad = (3 * res.r + 31) // 32 * 32
        assert np.array_equal(v["aux_q"][:, :3 * res.r], np.repeat(res.aux_q[:, :res.r], 3, axis=1))
        assert not v["aux_q"][:, 3 * res.r:pad].any()
        assert np.array_equal(v["w_aux"][:, :3 * res.r], np.repeat(wq_o[res.O].T, 3, axis=1))
        assert np.array_equal(acc.cpu().numpy(), res.acc)
        acc = mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32)
        assert mx.muxq_read_status(ws) == 0


@pytest.mark.parametrize("gran,tau", [(0, 6.0), (1, 6.0), (0, 2.0 ** -15), (1, 2.0 ** -15)])
@pytest.mark.parametrize("M,K", [(1040, 240), (600, 1296), (300, 2576), (5200, 528)])
def test_preparation_ties_and_small_scales(mx, gran, tau, M, K):
    """Codes where the quotient is next to or on a tie, for scales of every significand (a row whose maximum is b has its
    structural ties at odd multiples of b / 254), and rows so small that a value times 2^-e is no normal fp16 number."""
    x, w, _ = make_case(110 + M, M, K, 8, n_out=0)
    x = x.astype(np.float64)
    rng = np.random.default_rng(M + K)
    top = (1024 + np.arange(M) % 1024) / 512.0                                          # row maxima 2 .. 4
    ties = np.round(rng.integers(0, 127, (M, K)) + 0.5) * top[:, None] / 127.0
    odd = (2 * rng.integers(0, 127, (M, K)) + 1) * top[:, None] / 254.0
    x = np.where(rng.random((M, K)) < 0.5, odd, np.where(rng.random((M, K)) < 0.5, ties, x)).clip(-top[:, None], top[:, None])
    x *= rng.choice([-1.0, 1.0], (M, K))
    x[np.arange(M), rng.integers(0, K, M)] = top
    x[M // 2:] *= 2.0 ** -(np.arange(M - M // 2) % 26)[:, None]                          # down to subnormal rows and zeros
    if tau < 1:
        x *= 2.0 ** -13                                                                  # the whole input, per tensor as well
    out = rng.permutation(K)[:5]
    x[3, out] = 50.0 if tau > 1 else 2.0 ** -11
    x = x.astype(np.float16)
    p = mx.MuxqParams(gran=gran, threshold=tau, max_outliers=K if tau < 1 else 16)
    wq_o, sw_o, res = oracle_linear(x, w, p)
    acc, ws, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    v = ws_views(mx, ws, M, K, 8, p)
    assert st == 0 and v["n_outliers"] == res.r
    assert np.array_equal(v["s_x"].view(np.uint32), res.s_x.view(np.uint32))
    assert np.array_equal(v["body_q"], res.body_q)
    assert np.array_equal(v["aux_q"][:, :3 * res.r], np.repeat(res.aux_q[:, :res.r], 3, axis=1))
    assert np.array_equal(acc.cpu().numpy(), res.acc)


@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("M,K,N,n_out", [
    (100, 5120, 136, 5), (129, 3072, 1288, 0), (200, 5120, 1288, 40), (129, 3088, 1312, 3),  # one row of tiles, all cut
    (17, 2048, 1288, 0), (128, 1040, 1280, 40),                        # in one launch, without a GEMM (128 rows: per tensor)
    (300, 4112, 264, 6), (1003, 2064, 1040, 7),                        # all tiles cut, ragged edges, K tail
    (2600, 1280, 2304, 8)])                                            # whole tiles and cut ones (99 tiles)
def test_gemm_tiles_cut_along_k(mx, gran, M, K, N, n_out):
    """Tiles whose K blocks are divided among CTA pairs: accumulators and outputs of the full matrix, twice on one workspace."""
    x, w, _ = make_case(120 + M, M, K, N, n_out=n_out, mult=60.0)
    p = mx.MuxqParams(gran=gran, max_outliers=64)
    _, _, res = oracle_linear(x, w, p)
    acc, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0 and np.array_equal(acc.cpu().numpy(), res.acc)
    xd, bias = dev(x), (synth.normal(120, 1, N) * 0.5).astype(np.float32)
    y32 = mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_F32, bias=dev(bias))
    y16 = mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_F16)
    assert mx.muxq_read_status(ws) == 0
    assert np.array_equal(y32.cpu().numpy(), res.y32 + bias[None, :])
    assert f16_ulp_diff(y16.cpu().numpy(), res.y16).max() <= 1


@pytest.mark.parametrize("M,K,N,parts", [(300, 4096, 776, 4), (800, 8192, 776, 4), (4700, 3072, 776, 8), (100, 5120, 136, 20), (129, 3088, 1312, 5), (200, 5120, 1288, 5)])
def test_gemm_tiles_that_are_cut(mx, M, K, N, parts):
    """Tiles 128, 256, 256 (74 whole ones before two cut ones), 64, 192 and 128 columns wide on 148 SMs, cut into `parts` along K, which the first
    counter behind W_aux shows; ragged edges, outlier channels."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the plan is that of 148 SMs")
    x, w, _ = make_case(140 + M, M, K, N, n_out=5, mult=60.0)
    p = mx.MuxqParams(max_outliers=64)
    _, _, res = oracle_linear(x, w, p)
    acc, ws, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0 and np.array_equal(acc.cpu().numpy(), res.acc)
    v = mx.muxq_workspace_view(M, K, N, p)
    at = (v.w_aux + N * v.aux_cols + 1023) // 1024 * 1024
    assert int(ws.buf[at: at + 4].cpu().numpy().view(np.int32)[0]) == parts


@pytest.mark.parametrize("pairs", [1, 9])
@pytest.mark.parametrize("M,K,N,bias", [(100, 5120, 136, False), (300, 4112, 264, True)])
def test_gemm_on_a_device_that_holds_fewer_cta_pairs(mx, M, K, N, bias, pairs):
    """Where the parts of cut tiles do not all fit at once the tiles are done whole: the same results, in more rounds."""
    x, w, _ = make_case(130 + M, M, K, N, n_out=5, mult=60.0)
    p = mx.MuxqParams(max_outliers=64)
    b = (synth.normal(130, 1, N) * 0.5).astype(np.float32) if bias else None
    _, _, res = oracle_linear(x, w, p)
    w_q, s_w = mx.muxq_quantize(dev(w), p, True, mx.Workspace(mx.muxq_small_workspace_bytes(N)))
    ws = mx.Workspace(mx.muxq_workspace_bytes(M, K, N, p))
    try:
        mx.muxq_test_hooks(gemm_pairs=pairs)
        acc = mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32)
        y32 = mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_F32, bias=dev(b) if bias else None)
        y16 = mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_F16)
        assert mx.muxq_read_status(ws) == 0
    finally:
        mx.muxq_test_hooks()
    assert np.array_equal(acc.cpu().numpy(), res.acc)
    assert np.array_equal(y32.cpu().numpy(), res.y32 + b[None, :] if bias else res.y32)
    assert f16_ulp_diff(y16.cpu().numpy(), res.y16).max() <= 1


def test_handworked_example_on_gpu(mx):
    from conftest import load_golden
    g = load_golden("handworked_exp2.txt")
    K, N = 16, 8  # the 2x4 / 4x2 example embedded in zero padding
    x = np.zeros((2, K), np.float16); x[:, :4] = g["X"]
    w = np.zeros((K, N), np.float16); w[:4, :2] = g["W"]
    p = mx.MuxqParams(max_outliers=4)
    # decode path (M = 2)
    y, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_F32)
    assert st == 0 and np.array_equal(y.cpu().numpy()[:, :2].astype(np.float64), g["Y"])
    # tensor-core path: repeat the two rows to M = 32
    xx = np.tile(x, (16, 1))
    acc, ws, st, _, _ = run_linear(mx, xx, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0 and np.array_equal(acc.cpu().numpy()[:2, :2], g["acc"].astype(np.int32))
    y16, _, _, _, _ = run_linear(mx, xx, w, p, mx.MUXQ_OUT_F16)
    assert np.array_equal(y16.cpu().numpy()[:2, :2].astype(np.float64), g["Y16"])


@pytest.mark.parametrize("M", [1, 2, 4, 7, 16])
@pytest.mark.parametrize("K,N", [(1280, 1280), (1280, 3840), (5120, 1280), (256, 72)])
def test_decode_matches_oracle(mx, M, K, N):
    x, w, _ = make_case(60 + M + K, M, K, N, n_out=8, mult=60.0)
    for gran in (0, 1):
        p = mx.MuxqParams(gran=gran, max_outliers=32)
        _, _, res = oracle_linear(x, w, p)
        acc, ws, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
        assert st == 0 and np.array_equal(acc.cpu().numpy(), res.acc)
        y32, _, _, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F32)
        assert np.array_equal(y32.cpu().numpy(), res.y32)
        y16, _, _, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F16)
        assert f16_ulp_diff(y16.cpu().numpy(), res.y16).max() <= 1


# ------------------------------------------------------------------ edge cases
@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("K,N,pad,n_out", [
    (16, 8, 0, 1), (48, 136, 16, 0), (528, 2304, 0, 3), (1040, 1288, 0, 33),   # one group of channels, K tails, fewer rows than CTAs
    (5136, 264, 48, 8), (8192, 72, 0, 70),                                     # X read twice, pitched W_q
    (1296, 10240, 0, 8), (8192, 2400, 0, 4)])                                  # W_q through the ring of chunks
def test_decode_layer_edges(mx, M, K, N, pad, n_out):
    x, w, _ = make_case(160 + M + K, M, K, N, n_out=n_out, mult=60.0)
    for gran in (0, 1):
        p = mx.MuxqParams(gran=gran, max_outliers=512)
        wq_o, sw_o, res = oracle_linear(x, w, p)
        w_q, s_w = mx.muxq_quantize(dev(w), p, True, mx.Workspace(mx.muxq_small_workspace_bytes(N)))
        wide = torch.full((N, K + pad), 77, dtype=torch.int8, device="cuda")
        wide[:, :K] = w_q
        ws = mx.Workspace(mx.muxq_workspace_bytes(M, K, N, p))
        xd = dev(x)
        for out_kind, ref in ((mx.MUXQ_OUT_ACC_I32, res.acc), (mx.MUXQ_OUT_F32, res.y32)):
            y = mx.muxq_linear(xd, wide[:, :K], s_w, p, ws, out_kind)
            assert mx.muxq_read_status(ws) == 0
            assert np.array_equal(y.cpu().numpy(), ref)
        v = ws_views(mx, ws, M, K, N, p)
        assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O)
        assert np.array_equal(v["col_absmax"].view(np.uint32), res.colmax.view(np.uint32))
        assert np.array_equal(v["s_x"].view(np.uint32), res.s_x.view(np.uint32))


def test_decode_call_does_not_clear_the_status_word(mx):
    """The status word is sticky: an over-capacity decode call raises it, the ordinary call behind it leaves it raised."""
    M, K, N = 2, 768, 264
    p = mx.MuxqParams(max_outliers=4)
    x, w, _ = make_case(170, M, K, N, n_out=3, mult=200.0)
    bad, _, _ = make_case(171, M, K, N, n_out=40, mult=200.0)
    w_q, s_w = mx.muxq_quantize(dev(w), p, True, mx.Workspace(mx.muxq_small_workspace_bytes(N)))
    ws = mx.Workspace(mx.muxq_workspace_bytes(M, K, N, p))
    mx.muxq_linear(dev(bad), w_q, s_w, p, ws)
    assert mx.muxq_read_status(ws) == mx.MUXQ_ERR_CAPACITY
    mx.muxq_linear(dev(x), w_q, s_w, p, ws)
    assert mx.muxq_read_status(ws) == mx.MUXQ_ERR_CAPACITY
    ws.clear_status()
    mx.muxq_linear(dev(x), w_q, s_w, p, ws)
    assert mx.muxq_read_status(ws) == mx.MUXQ_OK


@pytest.mark.parametrize("M", [1, 4, 16, 64, 200])
def test_layer_call_directly_after_its_weights_were_rewritten(mx, M):
    """W_q and s_w are rewritten by ordinary kernels (the library's weight quantization, then a device copy into the
    very buffers the layer reads) directly before the layer call on the same stream.  The layer kernels fetch weight
    tiles ahead of their programmatic wait; predecessors that do not release their dependents early -- these -- must
    still be seen in full.  Decode (M <= 16), one launch (M = 64) and GEMM path (M = 200)."""
    K, N = 1280, 1280
    p = mx.MuxqParams(max_outliers=32)
    x, _ = synth.make_x(21, 1, M, K, 6, 50.0, 50.0)
    xd = dev(x)
    ws = mx.Workspace(mx.muxq_workspace_bytes(M, K, N, p))
    w1, w2 = synth.make_w(21, 1, K, N), synth.make_w(22, 2, K, N, sigma=0.05)
    wsw = mx.Workspace(mx.muxq_small_workspace_bytes(N))
    w_q, s_w = mx.muxq_quantize(dev(w1), p, True, wsw)
    y1 = mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_F32)           # quantize -> layer, back to back
    wq2, sw2 = mx.muxq_quantize(dev(w2), p, True, wsw)
    for _ in range(3):
        w_q.copy_(wq2); s_w.copy_(sw2)                                   # device copies into the buffers in use ...
        y2 = mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_F32)       # ... directly followed by the layer
    assert mx.muxq_read_status(ws) == 0
    for w, y in ((w1, y1), (w2, y2)):
        _, _, res = oracle_linear(x, w, p)
        assert np.array_equal(y.cpu().numpy(), res.y32)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("K,N", [(768, 768), (1280, 3840), (1536, 136), (2064, 1280), (5120, 64)])
def test_decode_call_whose_bias_is_the_result_of_the_call_before_it(mx, K, N, graph):
    """y_l = x_l W + y_(l-1) with one token row and fp32 results: every call's bias is what the call before it stores, so it
    must not be read ahead of the stream's order (the weights are).  One fp32 addition each: exact against the same sum."""
    p, L = mx.MuxqParams(max_outliers=32), 24
    x = synth.make_x(23, 1, L, K, 6, 50.0, 50.0)[0]
    w = synth.make_w(23, 1, K, N)
    w_q, s_w = mx.muxq_quantize(dev(w), p, True, mx.Workspace(mx.muxq_small_workspace_bytes(N)))
    ws = mx.Workspace(mx.muxq_workspace_bytes(1, K, N, p))
    xd, first = dev(x), dev(synth.normal(24, 1, N).astype(np.float32))
    ys = torch.empty(L, N, device="cuda")
    wq_o, sw_o = oracle.quantize_weight(w)
    want, acc = np.empty((L, N), np.float32), first.cpu().numpy()
    for l in range(L):
        acc = oracle.linear(x[l:l + 1], wq_o, sw_o, cap=32, want_codes=False).y32[0] + acc
        want[l] = acc

    def calls():
        ys.fill_(1e6)  # what a bias read too early would add
        for l in range(L):
            mx.muxq_linear(xd[l:l + 1], w_q, s_w, p, ws, mx.MUXQ_OUT_F32, out=ys[l:l + 1], bias=ys[l - 1] if l else first)

    run = calls
    if graph:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            calls()
            side.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side):
                calls()
        torch.cuda.synchronize()
        run = g.replay
    for _ in range(5):
        run()
        assert mx.muxq_read_status(ws) == 0
        assert np.array_equal(ys.cpu().numpy(), want)


@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("M,d", [(1, 64), (1, 768), (4, 64), (7, 64), (16, 64), (16, 528), (16, 1280), (33, 256), (300, 1296)])
def test_layer_calls_that_pass_their_results_back_and_forth(mx, M, d, gran):
    """Two buffers, each layer reads what the one before it wrote and overwrites what that one read, with as many launches in
    flight as the device takes: the same bits as one launch at a time."""
    p, L = mx.MuxqParams(gran=gran, max_outliers=d), 40
    ws = mx.Workspace(mx.muxq_workspace_bytes(M, d, d, p))
    small = mx.Workspace(mx.muxq_small_workspace_bytes(d))
    w = [mx.muxq_quantize(dev(synth.make_w(25, l, d, d, sigma=1.2 * d ** -0.5)), p, True, small) for l in range(4)]
    x0 = dev(synth.make_x(25, 1, M, d, 3, 20.0, 20.0)[0])

    def steps(a, b, wait):
        for l in range(L):
            mx.muxq_linear(a, w[l % 4][0], w[l % 4][1], p, ws, out=b)
            if wait:
                torch.cuda.synchronize()
            a, b = b, a
        return a

    want = steps(x0.clone(), torch.empty_like(x0), True).clone()
    assert torch.isfinite(want).all() and want.abs().max() > 0
    side = torch.cuda.Stream()
    a, b = x0.clone(), torch.empty_like(x0)
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            last = steps(a, b, False)
    torch.cuda.synchronize()
    for _ in range(3):
        a.copy_(x0)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(last, want)
        assert torch.equal(steps(x0.clone(), torch.empty_like(x0), False), want)
    assert mx.muxq_read_status(ws) == 0


def test_zero_outliers_equals_naive_int8(mx):
    x, w, _ = make_case(70, 256, 512, 256, n_out=0)
    p = mx.MuxqParams(threshold=1e4)
    _, _, res = oracle_linear(x, w, p)
    assert res.r == 0
    acc, ws, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0 and np.array_equal(acc.cpu().numpy(), res.acc)


def test_capacity_overflow_sets_status_and_stays_in_bounds(mx):
    M, K, N = 256, 512, 256
    x, w, _ = make_case(71, M, K, N, n_out=12)
    p = mx.MuxqParams(max_outliers=4)
    wsw = mx.Workspace(mx.muxq_small_workspace_bytes(N))
    w_q, s_w = mx.muxq_quantize(dev(w), p, True, wsw)
    nbytes = mx.muxq_workspace_bytes(M, K, N, p)
    ws = mx.Workspace(nbytes + 4096)
    ws.buf.fill_(0x77)  # canary behind the workspace proper
    ybuf = torch.full((M + 2, N), 1234.0, dtype=torch.float16, device="cuda")
    ws_use = mx.Workspace(0)
    ws_use.buf = ws.buf[:nbytes]
    ws_use.init()
    y = mx.muxq_linear(dev(x), w_q, s_w, p, ws_use, mx.MUXQ_OUT_F16, out=ybuf[1:M + 1])
    assert mx.muxq_read_status(ws_use) == mx.MUXQ_ERR_CAPACITY
    assert (ws.buf[nbytes:] == 0x77).all()
    assert (ybuf[0] == 1234.0).all() and (ybuf[M + 1] == 1234.0).all()
    v = ws_views(mx, ws_use, M, K, N, p)
    O, r, _ = oracle.detect(oracle.colmax(x), 6.0, 4)
    assert v["n_outliers"] == r and np.array_equal(v["outlier_idx"][:4], O)


def test_all_zero_activations(mx):
    x = np.zeros((128, 256), np.float16)
    w = synth.make_w(1, 1, 256, 128)
    for gran in (0, 1):
        y, ws, st, _, _ = run_linear(mx, x, w, mx.MuxqParams(gran=gran), mx.MUXQ_OUT_F32)
        assert st == 0 and not y.cpu().numpy().any()


def test_argument_errors(mx):
    p = mx.MuxqParams()
    ws = mx.Workspace(1 << 20)
    x = torch.zeros(32, 24, dtype=torch.float16, device="cuda")   # K % 16 != 0
    w_q = torch.zeros(64, 24, dtype=torch.int8, device="cuda")
    s_w = torch.ones(1, device="cuda")
    with pytest.raises(mx.MuxqError) as ei:
        mx.muxq_linear(x, w_q, s_w, p, ws)
    assert ei.value.status == mx.MUXQ_ERR_UNSUPPORTED
    x = torch.zeros(32, 32, dtype=torch.float16, device="cuda")
    w_q = torch.zeros(64, 32, dtype=torch.int8, device="cuda")
    small = mx.Workspace(256)
    with pytest.raises(mx.MuxqError) as ei:
        mx.muxq_linear(x, w_q, s_w, p, small)
    assert ei.value.status == mx.MUXQ_ERR_WORKSPACE
    with pytest.raises(mx.MuxqError) as ei:
        mx.muxq_linear(x, w_q, s_w, mx.MuxqParams(exp_factor=5), ws)
    assert ei.value.status == mx.MUXQ_ERR_INVALID_ARG
    with pytest.raises(mx.MuxqError) as ei:
        mx.muxq_linear(x, w_q, s_w, mx.MuxqParams(aux_scale=1), ws, mx.MUXQ_OUT_ACC_I32)
    assert ei.value.status == mx.MUXQ_ERR_UNSUPPORTED


def test_host_buffer_entry_point(mx):
    M, K, N = 256, 512, 264
    x, w, _ = make_case(80, M, K, N, n_out=3)
    p = mx.MuxqParams()
    wsw = mx.Workspace(mx.muxq_small_workspace_bytes(N))
    w_q, s_w = mx.muxq_quantize(dev(w), p, True, wsw)
    ws = mx.Workspace(mx.muxq_host_workspace_bytes(M, K, N, p, mx.MUXQ_OUT_F16))
    xh = torch.from_numpy(x).pin_memory()
    yh = torch.empty(M, N, dtype=torch.float16).pin_memory()
    mx.muxq_linear_host(xh, w_q, s_w, p, ws, yh, mx.MUXQ_OUT_F16)
    assert mx.muxq_read_status(ws) == 0
    _, _, res = oracle_linear(x, w, p)
    assert f16_ulp_diff(yh.numpy(), res.y16).max() <= 1


# ------------------------------------------------------------------ full benchmark sizes
def _full_size_check(mx, spec, gran, n_rows=32, cap=32, full=False):
    """One layer at its full size through muxq_linear (the launch configuration bench.py times);
    detection results, scales and every code of the full matrix are compared.  The products are compared
    on every row (full=True) or on sample rows: one row of every 128-row block of X (so that every
    output tile of the persistent GEMM loop, whichever CTA of a pair owns it, is hit) at an offset that
    walks through the block, the edges, and seeded random rows.  Each row of the layer is independent
    once O and the scales are fixed, so the oracle computes them one by one."""
    x, _ = spec.x()
    w = spec.w()
    p = mx.MuxqParams(gran=gran, max_outliers=cap)
    rows = None
    if not full:
        rng = np.random.default_rng(spec.seed * 1000 + spec.tensor_id)
        blocks = np.arange(0, spec.M, 128)
        per_block = blocks + (blocks // 128 * 37) % 128
        rows = np.unique(np.concatenate([[0, spec.M - 1, 127, 128, spec.M // 2], per_block,
                                         rng.integers(0, spec.M, n_rows)])).astype(np.int32)
        rows = rows[rows < spec.M]
    sel = slice(None) if rows is None else rows
    wq_o, sw_o, res = oracle_linear(x, w, p, rows=rows)
    assert res.rc == 0 and res.r >= spec.n_outliers
    y16, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_F16)
    assert st == 0
    v = ws_views(mx, ws, spec.M, spec.K, spec.N, p)
    assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O)
    assert np.array_equal(v["col_absmax"].view(np.uint32), res.colmax.view(np.uint32))
    assert np.array_equal(v["s_x"].view(np.uint32), res.s_x.view(np.uint32))
    assert np.array_equal(v["body_q"], res.body_q)          # every code of the full matrix
    assert np.array_equal(w_q.cpu().numpy(), wq_o.T)
    assert f16_ulp_diff(y16.cpu().numpy()[sel], res.y16).max() <= 1
    acc, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0 and np.array_equal(acc.cpu().numpy()[sel], res.acc)
    y32, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F32)
    assert st == 0 and rel_err32(y32.cpu().numpy()[sel], res.y32) <= 1e-5


def test_config0_full_matrix(mx):
    _full_size_check(mx, synth.config_layers(0)[0], 0, full=True)


@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("layer", [0, 1, 2, 3])
def test_config1_full_matrix(mx, layer, gran):
    _full_size_check(mx, synth.config_layers(1)[layer], gran, full=True)


@pytest.mark.parametrize("layer", [0, 1, 2, 3])
def test_config2_heavy_tailed_full_size_sampled_rows(mx, layer):
    _full_size_check(mx, synth.config_layers(2)[layer], 0, cap=64)


@pytest.mark.parametrize("layer", [0, 1, 2, 3])
def test_config3_prefill_full_size_sampled_rows(mx, layer):
    _full_size_check(mx, synth.config_layers(3)[layer], 0)


@pytest.mark.parametrize("M", [1, 4, 16])
def test_config3_decode_full_size(mx, M):
    for spec in synth.config_layers(3, M=M):
        x, _ = spec.x()
        w = spec.w()
        p = mx.MuxqParams(max_outliers=32)
        _, _, res = oracle_linear(x, w, p)
        y32, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F32)
        assert st == 0 and np.array_equal(y32.cpu().numpy(), res.y32)
        y16, ws, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F16)
        assert st == 0 and f16_ulp_diff(y16.cpu().numpy(), res.y16).max() <= 1
        v = ws_views(mx, ws, spec.M, spec.K, spec.N, p)
        assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O)


@pytest.mark.parametrize("n_out", [0, 2, 8, 32])
def test_config4_outlier_sweep_full_size_sampled_rows(mx, n_out):
    spec = synth.config_layers(4, n_outliers=n_out, layers=36)[35 * 4 + 2]   # last layer's c_fc, 8192 x 1280 -> 5120
    _full_size_check(mx, spec, 0, cap=64)


@pytest.mark.parametrize("linear", [0, 1, 2, 3])
@pytest.mark.parametrize("layer", [0, 17, 35])
def test_config4_first_middle_last_layer(mx, layer, linear):
    """Layers 0, 17 and 35 of the 36-layer stack, all four linears (8 outlier channels): the layers are
    independent problems (fresh X per layer), so three of them with every linear shape cover the stack's shapes
    and seeds at both ends and in the middle."""
    spec = synth.config_layers(4, n_outliers=8, layers=36)[layer * 4 + linear]
    _full_size_check(mx, spec, 0, cap=64, full=(layer == 0 and linear == 1))


@pytest.mark.parametrize("e,act_bits,w_bits,gran", [(1, 8, 8, 0), (3, 6, 5, 0), (3, 7, 4, 1), (2, 5, 8, 1)])
def test_linear_other_exp_factors_and_bit_widths(mx, e, act_bits, w_bits, gran):
    """exp factor 1 / 3 and the reduced bit widths of Tables 1-2 through the whole layer (tensor-core path
    and decode path): the Aux block then repeats each column 2^e - 1 = 1 or 7 times."""
    for M, K, N in ((384, 768, 520), (5, 1280, 264)):
        x, w, _ = make_case(300 + e + act_bits, M, K, N, n_out=5, mult=50.0)
        p = mx.MuxqParams(exp_factor=e, act_bits=act_bits, w_bits=w_bits, gran=gran, max_outliers=16)
        wq_o, sw_o, res = oracle_linear(x, w, p)
        acc, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
        assert st == 0 and np.array_equal(w_q.cpu().numpy(), wq_o.T)
        assert np.array_equal(acc.cpu().numpy(), res.acc)
        y32, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F32)
        assert st == 0 and np.array_equal(y32.cpu().numpy(), res.y32)
        y16, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F16)
        assert st == 0 and f16_ulp_diff(y16.cpu().numpy(), res.y16).max() <= 1


@pytest.mark.parametrize("M", [3, 40])
@pytest.mark.parametrize("gran", [0, 1])
def test_wide_k_takes_the_separate_kernels(mx, M, gran):
    """K beyond what the fused preparation / fused decode kernels hold (8192 channels) falls back to the
    stand-alone detect and quantize kernels; same results."""
    K, N = 8320, 136
    x, w, _ = make_case(500 + M, M, K, N, n_out=9, mult=50.0)
    p = mx.MuxqParams(gran=gran, max_outliers=32)
    _, _, res = oracle_linear(x, w, p)
    acc, ws, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0 and np.array_equal(acc.cpu().numpy(), res.acc)
    v = ws_views(mx, ws, M, K, N, p)
    assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O)
    assert np.array_equal(v["body_q"], res.body_q)
    y32, _, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F32)
    assert st == 0 and np.array_equal(y32.cpu().numpy(), res.y32)


def test_one_workspace_serves_a_sequence_of_shapes(mx):
    """The layer kernels leave the prepared words of the workspace as they found them: one
    muxq_workspace_init, then different shapes, granularities and repeats, each checked against the oracle."""
    shapes = [(300, 768, 256, 0), (300, 768, 256, 0), (64, 256, 136, 1), (520, 3072, 128, 0), (8, 512, 128, 0),
              (40, 8320, 136, 0), (300, 768, 256, 1), (1000, 1024, 264, 0)]
    big = 0
    for M, K, N, gran in shapes:
        big = max(big, mx.muxq_workspace_bytes(M, K, N, mx.MuxqParams(gran=gran)))
    ws = mx.Workspace(big)
    ws.buf.fill_(0x3C)
    ws.init()
    for i, (M, K, N, gran) in enumerate(shapes):
        p = mx.MuxqParams(gran=gran)
        x, w, _ = make_case(900 + i, M, K, N, n_out=5)
        w_q, s_w = mx.muxq_quantize(dev(w), p, True, mx.Workspace(mx.muxq_small_workspace_bytes(N)))
        y = mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_F32)
        assert mx.muxq_read_status(ws) == 0
        _, _, res = oracle_linear(x, w, p)
        v = ws_views(mx, ws, M, K, N, p)
        assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O), (i, M, K, N)
        assert rel_err32(y.cpu().numpy(), res.y32) <= 1e-5, (i, M, K, N)


# ------------------------------------------------------------------ own-scale reading of the Aux quantization
@pytest.mark.parametrize("M,K,N,gran,e,n_out", [(300, 768, 256, 0, 2, 5), (300, 768, 256, 1, 2, 5), (8, 512, 128, 0, 2, 3),
                                                 (1000, 1024, 264, 0, 3, 9), (520, 3072, 128, 1, 1, 6), (64, 256, 136, 0, 2, 0)])
def test_aux_own_scale_layer_matches_oracle(mx, M, K, N, gran, e, n_out):
    """Aux quantized with its own abs-max scale (the other reading of Eq. 1 for Aux): scales, Aux codes and
    outputs against the oracle's aux_own path."""
    p = mx.MuxqParams(gran=gran, exp_factor=e, aux_scale=mx.MUXQ_AUX_OWN)
    x, w, _ = make_case(1200 + M + e, M, K, N, n_out=n_out)
    wq, sw = oracle.quantize_weight(w, bits=p.w_bits, per_channel=gran == 1)
    res = oracle.linear(x, wq, sw, tau=p.threshold, e=e, act_bits=p.act_bits, per_vector=gran == 1, aux_own=True,
                        cap=p.max_outliers)
    for out_kind in (mx.MUXQ_OUT_F32, mx.MUXQ_OUT_F16):
        y, ws, st, _, _ = run_linear(mx, x, w, p, out_kind)
        assert st == 0
        v = ws_views(mx, ws, M, K, N, p)
        view = mx.muxq_workspace_view(M, K, N, p)
        b = ws.buf.cpu().numpy()
        s_a = b[view.s_a: view.s_a + 4 * (M if gran == 1 else 1)].view(np.float32)
        assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O)
        assert np.array_equal(v["s_x"], res.s_x) and np.array_equal(s_a, res.s_a)
        assert np.array_equal(v["body_q"], res.body_q)
        assert np.array_equal(v["aux_q"][:, :res.r], res.aux_q) and not v["aux_q"][:, res.r:].any()
        if out_kind == mx.MUXQ_OUT_F32:
            assert rel_err32(y.cpu().numpy(), res.y32) <= 1e-5
        else:
            assert f16_ulp_diff(y.cpu().numpy(), res.y16).max() <= 1


# ------------------------------------------------------------------ the layer's additive term (muxq_linear_bias)
@pytest.mark.parametrize("M,K,N,gran", [(300, 768, 256, 0), (1000, 1024, 264, 1), (2600, 256, 776, 0), (1, 1280, 264, 0),
                                        (7, 768, 136, 1), (16, 8320, 128, 0)])
@pytest.mark.parametrize("out_kind", [0, 1])
def test_linear_with_bias(mx, M, K, N, gran, out_kind):
    """Prefill shapes (both GEMM kernels' epilogues, ragged tiles) and decode shapes (fused and two-kernel form):
    fp32 outputs bit-equal to the oracle's one-addition reading, fp16 within 1 ulp."""
    p = mx.MuxqParams(gran=gran)
    x, w, _ = make_case(1800 + M + gran, M, K, N, n_out=5, mult=50.0)
    bias = (synth.normal(1800 + M, 9, N) * 0.5).astype(np.float32)
    wq, sw = oracle.quantize_weight(w, bits=p.w_bits, per_channel=gran == 1)
    res = oracle.linear(x, wq, sw, per_vector=gran == 1, bias=bias, want_codes=False)
    w_q, s_w = mx.muxq_quantize(dev(w), p, True, mx.Workspace(mx.muxq_small_workspace_bytes(N)))
    ws = mx.Workspace(mx.muxq_workspace_bytes(M, K, N, p))
    y = mx.muxq_linear(dev(x), w_q, s_w, p, ws, out_kind, bias=dev(bias))
    assert mx.muxq_read_status(ws) == 0
    g = y.cpu().numpy()
    if out_kind == 1:
        assert np.array_equal(g, res.y32)
    else:
        assert f16_ulp_diff(g, res.y16).max() <= 1
    # without the term the same call gives the plain layer (the epilogue's branch is off, not stale)
    y0 = mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_F32)
    assert np.array_equal(y0.cpu().numpy(), oracle.linear(x, wq, sw, per_vector=gran == 1, want_codes=False).y32)


def test_linear_bias_argument_errors(mx):
    p = mx.MuxqParams()
    x = torch.zeros(32, 256, dtype=torch.float16, device="cuda")
    w_q = torch.zeros(128, 256, dtype=torch.int8, device="cuda")
    s_w = torch.ones(1, device="cuda")
    bias = torch.zeros(128, device="cuda")
    ws = mx.Workspace(mx.muxq_workspace_bytes(32, 256, 128, p))
    with pytest.raises(mx.MuxqError) as ei:
        mx.muxq_linear(x, w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32, bias=bias)
    assert ei.value.status == mx.MUXQ_ERR_INVALID_ARG
    pown = mx.MuxqParams(aux_scale=mx.MUXQ_AUX_OWN)
    with pytest.raises(mx.MuxqError) as ei:
        mx.muxq_linear(x, w_q, s_w, pown, mx.Workspace(mx.muxq_workspace_bytes(32, 256, 128, pown)), mx.MUXQ_OUT_F32, bias=bias)
    assert ei.value.status == mx.MUXQ_ERR_UNSUPPORTED


# ------------------------------------------------------------------ an outlier set as large as K
@pytest.mark.parametrize("M,K,N,gran", [(300, 1280, 256, 0), (300, 1280, 256, 1), (260, 5120, 136, 0), (4, 1280, 264, 0),
                                        (16, 5120, 128, 1)])
def test_every_channel_an_outlier_channel(mx, M, K, N, gran):
    """A bulk wide enough that every channel holds an element above the threshold: O is all of K (beyond 1024
    channels), Aux mirrors the whole of Body, and the layer still matches the oracle code for code."""
    p = mx.MuxqParams(gran=gran, max_outliers=K)
    x, w, _ = make_case(1700 + M + gran, M, K, N, n_out=8, mult=60.0, bulk="t4", bulk_scale=6.0 if M > 16 else 40.0)
    wq, sw = oracle.quantize_weight(w, bits=p.w_bits, per_channel=gran == 1)
    res = oracle.linear(x, wq, sw, tau=p.threshold, e=p.exp_factor, act_bits=p.act_bits, per_vector=gran == 1, cap=K)
    assert res.r > 1024 and res.r >= 0.97 * K
    y, ws, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F32)
    assert st == 0
    v = ws_views(mx, ws, M, K, N, p)
    assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O)
    assert np.array_equal(v["s_x"], res.s_x)
    if M > 16:
        assert np.array_equal(v["body_q"], res.body_q)
        c = (1 << p.exp_factor) - 1
        assert np.array_equal(v["aux_q"][:, 0:c * res.r:c], res.aux_q)
    assert rel_err32(y.cpu().numpy(), res.y32) <= 1e-5
    acc = mx.muxq_linear(dev(x), *mx.muxq_quantize(dev(w), p, True, mx.Workspace(mx.muxq_small_workspace_bytes(N))),
                         p, mx.Workspace(mx.muxq_workspace_bytes(M, K, N, p)), mx.MUXQ_OUT_ACC_I32)
    assert np.array_equal(acc.cpu().numpy(), res.acc)


# ------------------------------------------------------------------ many outlier channels (capacity up to 1024)
@pytest.mark.parametrize("M,K,N,gran,own", [(300, 1024, 256, 0, 0), (300, 1024, 256, 1, 0), (8, 1024, 128, 0, 0),
                                             (200, 512, 136, 0, 1)])
def test_many_outlier_channels(mx, M, K, N, gran, own):
    """Heavy-tailed activations at unit scale flag most channels (Section III-C detection on a Student-t bulk):
    with max_outliers = 1024 the layer still matches the oracle code for code."""
    p = mx.MuxqParams(gran=gran, max_outliers=1024, aux_scale=own)
    # (a few rows need a wider bulk to push most channels over the threshold)
    x, w, _ = make_case(1500 + M + gran, M, K, N, n_out=8, mult=60.0, bulk="t4", bulk_scale=1.0 if M > 16 else 4.0)
    wq, sw = oracle.quantize_weight(w, bits=p.w_bits, per_channel=gran == 1)
    res = oracle.linear(x, wq, sw, tau=p.threshold, e=p.exp_factor, act_bits=p.act_bits, per_vector=gran == 1,
                        aux_own=bool(own), cap=1024)
    assert res.r > 64  # beyond the default capacity
    y, ws, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_F32)
    assert st == 0
    v = ws_views(mx, ws, M, K, N, p)
    assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O)
    assert np.array_equal(v["s_x"], res.s_x)
    if M > 16:
        assert np.array_equal(v["body_q"], res.body_q)
        c = 1 if own else (1 << p.exp_factor) - 1
        assert np.array_equal(v["aux_q"][:, 0:c * res.r:c], res.aux_q)
    assert rel_err32(y.cpu().numpy(), res.y32) <= 1e-5
    if not own:
        acc = mx.muxq_linear(dev(x), *mx.muxq_quantize(dev(w), p, True, mx.Workspace(mx.muxq_small_workspace_bytes(N))),
                             p, mx.Workspace(mx.muxq_workspace_bytes(M, K, N, p)), mx.MUXQ_OUT_ACC_I32)
        assert np.array_equal(acc.cpu().numpy(), res.acc)
    # the default capacity reports the overflow instead
    p64 = mx.MuxqParams(gran=gran, aux_scale=own)
    _, ws64, st64, _, _ = run_linear(mx, x, w, p64, mx.MUXQ_OUT_F32)
    assert st64 == mx.MUXQ_ERR_CAPACITY
