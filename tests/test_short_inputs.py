"""Layers of short inputs in one launch, shared along K between the CTAs of a cluster (k_short), against the oracle: every code and
accumulator, what is left in the workspace, outputs bit for bit (fp32) and within 1 ulp (fp16)."""
import numpy as np
import pytest

from conftest import kernels_launched
from test_gpu_parity import dev, f16_ulp_diff, make_case, mx, oracle_linear, run_linear, ws_views  # noqa: F401  (mx: fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def check_workspace(v, M, res, wq_o, c=3):
    assert v["n_outliers"] == res.r and np.array_equal(v["outlier_idx"][:res.r], res.O)
    assert np.array_equal(v["col_absmax"].view(np.uint32), res.colmax.view(np.uint32))
    assert np.array_equal(v["s_x"].view(np.uint32), res.s_x.view(np.uint32))
    if M <= 16:
        return
    used, pad = c * res.r, (c * res.r + 31) // 32 * 32
    assert np.array_equal(v["body_q"], res.body_q)
    assert np.array_equal(v["aux_q"][:, :used], np.repeat(res.aux_q[:, :res.r], c, axis=1)) and not v["aux_q"][:, used:pad].any()
    assert np.array_equal(v["w_aux"][:, :used], np.repeat(wq_o[res.O].T, c, axis=1)) and not v["w_aux"][:, used:pad].any()


# one row and one column more or less than a tile, slices that end inside a block of 128 or 32 channels or are empty, rows that no CTA
# finishes, several reads of X per thread (fewer than 192 output channels, narrow decode layers and some per token take other kernels:
# test_forms_of_short_inputs says which forms of this one run)
@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("M,K,N,n_out,cap", [
    (17, 16, 24, 1, 4), (17, 48, 8, 2, 8), (31, 272, 136, 3, 8), (33, 400, 400, 0, 8), (64, 768, 776, 6, 64), (65, 1040, 264, 7, 64),
    (128, 768, 768, 4, 64), (127, 1296, 520, 8, 16), (96, 3088, 768, 8, 64), (40, 5120, 1280, 8, 64), (17, 8192, 72, 20, 64),
    (20, 1280, 5120, 8, 64), (24, 2048, 4096, 40, 64), (50, 1040, 72, 100, 128), (16, 5120, 1280, 8, 64), (9, 3072, 768, 5, 64),
    (16, 8192, 520, 70, 128), (5, 4112, 264, 3, 8), (4, 5120, 1280, 8, 64)])
def test_layers_of_short_inputs(mx, gran, M, K, N, n_out, cap):
    x, w, _ = make_case(200 + M + K, M, K, N, n_out=n_out, mult=60.0)
    x[M // 2] = 0
    p = mx.MuxqParams(gran=gran, max_outliers=cap)
    wq_o, sw_o, res = oracle_linear(x, w, p)
    assert res.r <= cap
    acc, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0
    for _ in range(2):
        check_workspace(ws_views(mx, ws, M, K, N, p), M, res, wq_o)
        assert np.array_equal(acc.cpu().numpy(), res.acc)
        acc = mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32)
    b = np.linspace(-2.0, 2.0, N, dtype=np.float32)
    y32 = mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_F32, bias=dev(b)).cpu().numpy()
    y16 = mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_F16).cpu().numpy()
    assert mx.muxq_read_status(ws) == 0
    assert np.array_equal(y32, res.y32 + b) and f16_ulp_diff(y16, res.y16).max() <= 1


# Clusters of 8, 4 and 2; two, four and eight chunks of X per thread, and more than stay in registers (read again for the codes, per token
# for the row maxima too); the smallest layer, the widest X
@pytest.mark.parametrize("M,K,N,gran,ctas,form", [
    (17, 48, 192, 0, 2, "2,1,1"), (17, 48, 192, 1, 2, "2,1,1"), (33, 512, 5120, 0, 2, "4,1,1"), (20, 1280, 5120, 0, 4, "2,1,1"),
    (20, 1280, 5120, 1, 4, "2,1,1"), (24, 2048, 4096, 0, 4, "4,1,1"), (31, 1040, 264, 1, 8, "2,1,1"), (128, 768, 768, 0, 8, "4,1,1"),
    (65, 1040, 264, 1, 8, "4,1,1"), (40, 5120, 1280, 1, 8, "8,1,1"), (127, 1296, 520, 0, 8, "8,1,1"), (100, 3088, 768, 0, 8, "8,0,1"),
    (48, 6144, 1536, 1, 8, "8,0,1"), (64, 8192, 512, 0, 8, "8,0,1"), (16, 768, 5120, 0, 2, "2,1,0"), (5, 1280, 1288, 0, 4, "2,1,0"),
    (9, 3072, 768, 0, 8, "2,1,0"), (16, 5120, 1280, 0, 8, "4,1,0"), (16, 5120, 1280, 1, 8, "4,1,0"), (16, 8192, 1152, 0, 8, "4,1,0")])
def test_forms_of_short_inputs(mx, M, K, N, gran, ctas, form):
    x, w, _ = make_case(500 + M + K, M, K, N, n_out=7, mult=60.0)
    p = mx.MuxqParams(gran=gran)
    wq_o, _, res = oracle_linear(x, w, p)
    acc, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0 and np.array_equal(acc.cpu().numpy(), res.acc)
    check_workspace(ws_views(mx, ws, M, K, N, p), M, res, wq_o)
    xd, b = dev(x), np.linspace(-2.0, 2.0, N, dtype=np.float32)
    y32 = mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_F32, bias=dev(b))
    y16 = mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_F16)
    assert mx.muxq_read_status(ws) == 0
    assert np.array_equal(y32.cpu().numpy(), res.y32 + b) and f16_ulp_diff(y16.cpu().numpy(), res.y16).max() <= 1
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:  # (the choice is that of 148 SMs)
        hold, keeps, full = form.split(",")
        (name, size), = kernels_launched(lambda: mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_F16, out=y16))
        assert size == ctas and f"k_shortILi{hold}ELb{keeps}ELb{full}E" in name


@pytest.mark.parametrize("gran", [0, 1])
def test_marked_workspace_is_left_alone_by_the_one_launch(mx, gran):
    """After a time-out of the preparation (which the switch makes this call take) ordinary calls, in one launch again, report it and leave
    everything as it is until the workspace is prepared anew."""
    M, K, N = 48, 1280, 776
    x, w, _ = make_case(37, M, K, N, n_out=5, mult=60.0)
    p = mx.MuxqParams(gran=gran)
    wq_o, _, res = oracle_linear(x, w, p)
    _, ws, _, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    xd, y = dev(x), torch.full((M, N), 0x5A5A5A5A, dtype=torch.int32, device="cuda")
    call = lambda: mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32, out=y)  # noqa: E731
    try:
        mx.muxq_test_hooks(spin_limit=4096, prep_extra_arrivals=1)
        call()
        assert mx.muxq_read_status(ws) == mx.MUXQ_ERR_TIMEOUT
    finally:
        mx.muxq_test_hooks()
    assert [k for k, _ in kernels_launched(call) if "k_short" not in k] == []
    v = mx.muxq_workspace_view(M, K, N, p)
    written = [(v.col_absmax, 4 * K), (v.outlier_idx, 4 * p.max_outliers), (v.body_q, M * v.ld_body_q), (v.aux_q, M * v.aux_cols),
               (v.w_aux, N * v.aux_cols)] + ([(v.s_x, 4 * M)] if gran else [])
    for off, n in written:
        ws.buf[off: off + n] = 0x5A
    y.fill_(0x5A5A5A5A)
    for _ in range(2):
        ws.clear_status()
        call()
        assert mx.muxq_read_status(ws) == mx.MUXQ_ERR_TIMEOUT and bool((y == 0x5A5A5A5A).all())
        for off, n in written:
            assert bool((ws.buf[off: off + n] == 0x5A).all()), off
    ws.init()
    call()
    assert mx.muxq_read_status(ws) == 0 and np.array_equal(y.cpu().numpy(), res.acc)
    check_workspace(ws_views(mx, ws, M, K, N, p), M, res, wq_o)


@pytest.mark.parametrize("exp_factor,bits", [(1, 8), (3, 8), (2, 5)])
def test_exponents_and_widths_of_short_inputs(mx, exp_factor, bits):
    M, K, N = 48, 1024, 1024
    x, w, _ = make_case(31, M, K, N, n_out=9, mult=60.0)
    p = mx.MuxqParams(exp_factor=exp_factor, act_bits=bits, w_bits=bits, max_outliers=16)
    wq_o, sw_o, res = oracle_linear(x, w, p)
    acc, ws, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0 and np.array_equal(acc.cpu().numpy(), res.acc)
    check_workspace(ws_views(mx, ws, M, K, N, p), M, res, wq_o, c=(1 << exp_factor) - 1)


def launched(mx, M, K, N, gran):
    """[(kernel, CTAs per cluster)] of a layer call on data that do not matter."""
    p = mx.MuxqParams(gran=gran)
    ws = mx.Workspace(mx.muxq_workspace_bytes(M, K, N, p))
    x, y = torch.zeros(M, K, dtype=torch.float16, device="cuda"), torch.zeros(M, N, dtype=torch.float16, device="cuda")
    w_q, s_w = torch.zeros(N, K, dtype=torch.int8, device="cuda"), torch.ones(N, device="cuda")
    mx.muxq_linear(x, w_q, s_w, p, ws, out=y)
    return kernels_launched(lambda: mx.muxq_linear(x, w_q, s_w, p, ws, out=y))


@pytest.mark.parametrize("M,K,N,gran", [(96, 640, 2560, 1), (80, 768, 2304, 1), (112, 512, 2048, 1), (113, 4688, 616, 1), (72, 6288, 280, 1)])
def test_layers_that_the_one_launch_would_slow_down(mx, M, K, N, gran):
    """Layers that three launches do faster by 10 to 25 % take the three."""
    assert torch.cuda.get_device_properties(0).multi_processor_count != 148 or len(launched(mx, M, K, N, gran)) == 3


# Words of Aux and W_aux that two CTAs share, for c = 1, 3 and 7; more outlier channels than lanes, than a list of default length, and
# all of some steps of 32 channels; slices without any
@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("M,K,N,n_out,cap,exp_factor", [
    (50, 1040, 264, 100, 160, 2), (20, 768, 768, 200, 256, 3), (64, 1280, 1288, 64, 128, 1), (128, 768, 264, 37, 64, 3),
    (33, 512, 5120, 130, 256, 2), (24, 2048, 4096, 1, 1, 3),
    (16, 1280, 1280, 100, 160, 3), (9, 1296, 1288, 64, 128, 2), (12, 1296, 1296, 3, 8, 1), (16, 5120, 1288, 300, 512, 3)])
def test_many_outlier_channels_of_short_inputs(mx, gran, M, K, N, n_out, cap, exp_factor):
    x, w, _ = make_case(400 + M + K, M, K, N, n_out=n_out, mult=60.0)
    x[:, 32:64] *= np.float16(8.0 if n_out > 60 else 1.0)
    p = mx.MuxqParams(gran=gran, max_outliers=cap, exp_factor=exp_factor)
    wq_o, _, res = oracle_linear(x, w, p)
    assert 0 < res.r <= cap
    acc, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    xd = dev(x)
    names = [k for k, _ in kernels_launched(lambda: mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32, out=acc))]
    assert len(names) == 1 and "k_short" in names[0]
    for _ in range(2):
        assert st == 0 and np.array_equal(acc.cpu().numpy(), res.acc)
        check_workspace(ws_views(mx, ws, M, K, N, p), M, res, wq_o, c=(1 << exp_factor) - 1)
        acc = mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32)
        st = mx.muxq_read_status(ws)


def test_pitched_operands_and_more_outliers_than_room(mx):
    M, K, N = 32, 768, 768
    x, w, _ = make_case(32, M, K, N, n_out=12, mult=60.0)
    p = mx.MuxqParams()
    _, _, res = oracle_linear(x, w, p)
    wide = torch.zeros(M, K + 24, dtype=torch.float16, device="cuda")
    wide[:, :K] = dev(x)
    _, ws, _, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_F16)
    out = torch.zeros(M, N + 16, dtype=torch.float16, device="cuda")
    mx.muxq_linear(wide[:, :K], w_q, s_w, p, ws, mx.MUXQ_OUT_F16, out=out[:, :N])
    assert mx.muxq_read_status(ws) == 0 and not out[:, N:].any()
    assert f16_ulp_diff(out[:, :N].cpu().numpy(), res.y16).max() <= 1
    few = mx.MuxqParams(max_outliers=8)
    ws = mx.Workspace(mx.muxq_workspace_bytes(M, K, N, few))
    mx.muxq_linear(dev(x), w_q, s_w, few, ws, mx.MUXQ_OUT_F16)
    assert mx.muxq_read_status(ws) == mx.MUXQ_ERR_CAPACITY


def test_output_in_the_place_of_the_input(mx):
    """Beyond 16 rows Y may stand where X does: such a call takes the way that has read X when it writes."""
    M, K = 64, 1024
    x, w, _ = make_case(33, M, K, K, n_out=5, mult=60.0)
    p = mx.MuxqParams()
    _, _, res = oracle_linear(x, w, p)
    _, ws, _, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_F16)
    xy = dev(x)
    mx.muxq_linear(xy, w_q, s_w, p, ws, mx.MUXQ_OUT_F16, out=xy)
    assert mx.muxq_read_status(ws) == 0 and f16_ulp_diff(xy.cpu().numpy(), res.y16).max() <= 1


@pytest.mark.parametrize("M", [16, 64])
def test_weights_that_never_arrive_time_out(mx, M):
    K, N = 5120, 1288
    x, w, _ = make_case(34, M, K, N, n_out=5, mult=60.0)
    p = mx.MuxqParams()
    _, _, res = oracle_linear(x, w, p)
    acc, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0
    raw = torch.full((M + 2, N), 0x5A5A5A5A, dtype=torch.int32, device="cuda")
    try:
        mx.muxq_test_hooks(spin_limit=20000, gemm_skip_k_block=2)
        mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32, out=raw[1:-1])
        assert mx.muxq_read_status(ws) == mx.MUXQ_ERR_TIMEOUT
    finally:
        mx.muxq_test_hooks()
    assert bool((raw[0] == 0x5A5A5A5A).all()) and bool((raw[-1] == 0x5A5A5A5A).all())
    for _ in range(3):
        ws.clear_status()
        acc = mx.muxq_linear(dev(x), w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32)
        assert mx.muxq_read_status(ws) == 0 and np.array_equal(acc.cpu().numpy(), res.acc)


# the first warp of every CTA, the one that lists the outlier channels, some, all but the first, all
@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("late", [0x0001, 0x0002, 0x5A5A, 0xFFFE, 0xFFFF])
@pytest.mark.parametrize("M", [16, 64])
def test_exchange_that_only_some_warps_give_up_on(mx, M, late, gran):
    """Warps poll the exchange between the CTAs each for itself.  Where the limit runs out for some of them only, the reporting CTAs
    give up as a whole and store nothing, W_aux gets its own bytes or none, the call ends with a time-out, and the next one is right."""
    K, N = 5120, 1288
    x, w, _ = make_case(35, M, K, N, n_out=5, mult=60.0)
    p = mx.MuxqParams(gran=gran)
    wq_o, _, res = oracle_linear(x, w, p)
    acc, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0
    v = mx.muxq_workspace_view(M, K, N, p)
    written = [(v.col_absmax, 4 * K), (v.outlier_idx, 4 * p.max_outliers)] + ([(v.s_x, 4 * M)] if gran else [])
    if M > 16:
        written += [(v.body_q, M * v.ld_body_q), (v.aux_q, M * v.aux_cols)]
    for off, n in written + [(v.w_aux, N * v.aux_cols)]:
        ws.buf[off: off + n] = 0x5A
    xd, raw = dev(x), torch.full((M + 2, N), 0x5A5A5A5A, dtype=torch.int32, device="cuda")
    call = lambda: mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32, out=raw[1:-1])  # noqa: E731
    assert [k for k, _ in kernels_launched(call) if "k_short" not in k] == []
    try:
        mx.muxq_test_late_warps(late)
        call()
        assert mx.muxq_read_status(ws) == mx.MUXQ_ERR_TIMEOUT
    finally:
        mx.muxq_test_hooks()
    assert bool((raw[0] == 0x5A5A5A5A).all()) and bool((raw[-1] == 0x5A5A5A5A).all())
    w_aux, pad = ws_views(mx, ws, M, K, N, p)["w_aux"].view(np.uint8), (3 * res.r + 31) // 32 * 32
    want = np.zeros((N, pad), np.uint8)
    want[:, :3 * res.r] = np.repeat(wq_o[res.O].T, 3, axis=1).view(np.uint8)
    assert ((w_aux[:, :pad] == want) | (w_aux[:, :pad] == 0x5A)).all() and (w_aux[:, pad:] == 0x5A).all()
    for off, n in written:
        assert bool((ws.buf[off: off + n] == 0x5A).all()), off
    for _ in range(3):
        ws.clear_status()
        call()
        assert mx.muxq_read_status(ws) == 0 and np.array_equal(raw[1:-1].cpu().numpy(), res.acc)
        check_workspace(ws_views(mx, ws, M, K, N, p), M, res, wq_o)


@pytest.mark.parametrize("late", [0x00010000, 0x00020000, 0x5A5A0000, 0xFFFF0000])
@pytest.mark.parametrize("M", [16, 64])
def test_products_that_some_warps_give_up_on(mx, M, late):
    """A limit that runs out while products are on their way: they end before tensor memory is freed, CTAs that wait for sums that
    are never sent give up too, and the next calls find everything free and are right."""
    K, N = 5120, 1288
    x, w, _ = make_case(36, M, K, N, n_out=12, mult=60.0)
    p = mx.MuxqParams()
    wq_o, _, res = oracle_linear(x, w, p)
    acc, ws, st, w_q, s_w = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0
    xd, raw = dev(x), torch.full((M + 2, N), 0x5A5A5A5A, dtype=torch.int32, device="cuda")
    call = lambda: mx.muxq_linear(xd, w_q, s_w, p, ws, mx.MUXQ_OUT_ACC_I32, out=raw[1:-1])  # noqa: E731
    assert [k for k, _ in kernels_launched(call) if "k_short" not in k] == []
    try:
        mx.muxq_test_hooks(spin_limit=20000)
        mx.muxq_test_late_warps(late)
        call()
        assert mx.muxq_read_status(ws) == mx.MUXQ_ERR_TIMEOUT
    finally:
        mx.muxq_test_hooks()
    assert bool((raw[0] == 0x5A5A5A5A).all()) and bool((raw[-1] == 0x5A5A5A5A).all())
    for _ in range(3):
        ws.clear_status()
        call()
        assert mx.muxq_read_status(ws) == 0 and np.array_equal(raw[1:-1].cpu().numpy(), res.acc)
        check_workspace(ws_views(mx, ws, M, K, N, p), M, res, wq_o)


@pytest.mark.parametrize("gran", [0, 1])
@pytest.mark.parametrize("K,n_out,cap", [(16, 1, 4), (528, 0, 8), (1024, 5, 8), (1280, 8, 16), (1296, 8, 16), (2560, 9, 16), (2576, 5, 16), (5120, 8, 16),
                                         (5136, 8, 16), (8192, 20, 64), (1040, 100, 128)])
def test_row_kernel_edges_behind_short_inputs(mx, gran, K, n_out, cap):
    """One row more than k_short takes: the edges of the row kernel's warps per row."""
    M, N = 129, 72
    x, w, _ = make_case(300 + K, M, K, N, n_out=n_out, mult=60.0)
    p = mx.MuxqParams(gran=gran, max_outliers=cap)
    wq_o, _, res = oracle_linear(x, w, p)
    acc, ws, st, _, _ = run_linear(mx, x, w, p, mx.MUXQ_OUT_ACC_I32)
    assert st == 0 and np.array_equal(acc.cpu().numpy(), res.acc)
    check_workspace(ws_views(mx, ws, M, K, N, p), M, res, wq_o)
