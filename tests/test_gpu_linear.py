"""GPU parity: the group-quantized linear / conv layer against the oracle (int64 accumulate, fp64 de-quantize)."""
import numpy as np
import pytest

from oracle import calibration as oc
from oracle import linear as ol
from paper_2501_04304_b200 import synth
from dgq_testlib import gpu, to_dev, unpermute_codes, layer_case, check_output

pytestmark = pytest.mark.gpu

REL = 1e-3   # max|delta| <= 1e-3 * max|ref|


def _run_linear(torch, b, X, W, bias, gr, g, mode, w_bits):
    wq_ref, sw_ref = ol.weight_rtn(W, w_bits)
    w = b.weight_prepare(g, to_dev(torch, W), w_bits)
    wq, sw = w.export()
    assert np.array_equal(wq, wq_ref) and np.array_equal(sw, sw_ref)
    Xd = to_dev(torch, X)
    bd = to_dev(torch, bias) if bias is not None else None
    if mode == "static":
        codes, s_rows, z_rows = ol.quantize_static(X, gr, 0)
        Xq, ds, dz = b.quantize_act(g, Xd)
        Y = b.linear(g, w, Xq, bias=bd)
    else:
        codes, s_rows, z_rows = ol.quantize_dynamic_token(X, gr.col_group, gr.G, gr.bits)
        Xq, ds, dz = b.quantize_act(g, Xd, mode=b.MODE_DYNAMIC_TOKEN)
        Y = b.linear(g, w, Xq, mode=b.MODE_DYNAMIC_TOKEN, dyn_scale=ds, dyn_zp=dz, bias=bd)
    assert np.array_equal(unpermute_codes(Xq, g.export()["perm"], X.shape[1]), codes)
    Yref = ol.group_linear(codes, s_rows, z_rows, gr.col_group, wq_ref, sw_ref, bias)
    assert b.device_status() == 0
    return check_output(Y, Yref, REL)


@pytest.mark.parametrize("mode", ["static", "dynamic"])
def test_config1_w8a8(mode):
    """256 tokens x 320 channels, 4 channel groups + outlier group, both outlier types, W8A8."""
    torch, b = gpu()
    Xcal, X, W, bias, gr = layer_case(0, 1, 256, 320, 320, 4, 8, oc.DIM_BOTH, oc.OUTLIER_EXPLICIT, 4, 2)
    g = b.calibrate_groups(to_dev(torch, Xcal), 256, 8, 4, b.DIM_BOTH, b.OUTLIER_EXPLICIT, 5.0)
    assert g.G == 5
    _run_linear(torch, b, X, W, bias, gr, g, mode, 8)


@pytest.mark.parametrize("M,C,N,K,w_bits,mode", [
    (128, 32, 16, 1, 8, "static"),          # one tile, one atom, one group
    (128, 32, 16, 1, 4, "static"),
    (1000, 320, 320, 8, 8, "dynamic"),      # ragged M tail, BN = 160
    (1000, 320, 320, 8, 4, "dynamic"),
    (616, 768, 640, 8, 4, "dynamic"),       # cross-attention k/v projection shape, M = 8 x 77
    (384, 1280, 320, 8, 8, "static"),       # FF2-like: long K, several stages per group
    (300, 320, 2560, 8, 8, "dynamic"),      # FF1-like: many N tiles
    (260, 328, 72, 16, 8, "dynamic"),       # N not a tile multiple (BN = 128 with tail), G = 16
    (130, 64, 48, 3, 4, "static"),          # BN = 64 path
])
def test_linear_shapes(M, C, N, K, w_bits, mode):
    torch, b = gpu()
    Xcal, X, W, bias, gr = layer_case(7, 1, M, C, N, K, 8, oc.DIM_CHANNEL)
    g = b.calibrate_groups(to_dev(torch, Xcal), M, 8, K, b.DIM_CHANNEL)
    _run_linear(torch, b, X, W, bias, gr, g, mode, w_bits)


def test_static_grid_with_pixel_groups_and_no_bias():
    torch, b = gpu()
    Xcal, X, W, bias, gr = layer_case(8, 2, 256, 320, 320, 4, 8, oc.DIM_BOTH)
    g = b.calibrate_groups(to_dev(torch, Xcal), 256, 8, 4, b.DIM_BOTH)
    assert g.R > 1 and g.G > 1
    _run_linear(torch, b, X, W, None, gr, g, "static", 8)


def test_a6_codes_and_centred_linear():
    """6-bit activations; zero-centred signed codes give the same layer output with no zero-point term."""
    torch, b = gpu()
    Xcal, X, W, bias, gr = layer_case(9, 1, 512, 320, 320, 8, 6, oc.DIM_CHANNEL, token_outliers=False)
    g = b.calibrate_groups(to_dev(torch, Xcal), 512, 6, 8, b.DIM_CHANNEL)
    wq, sw = ol.weight_rtn(W, 4)
    w = b.weight_prepare(g, to_dev(torch, W), 4)
    codes, s_rows, z_rows = ol.quantize_static(X, gr, 0)
    Yref = ol.group_linear(codes, s_rows, z_rows, gr.col_group, wq, sw, bias)
    Xd, bd = to_dev(torch, X), to_dev(torch, bias)
    Xq, _, _ = b.quantize_act(g, Xd, layout=b.CODES_S8_CENTRED)
    Y = b.linear(g, w, Xq, layout=b.CODES_S8_CENTRED, bias=bd)
    check_output(Y, Yref, REL)
    Xq2, _, _ = b.quantize_act(g, Xd)
    Y2 = b.linear(g, w, Xq2, bias=bd)
    check_output(Y2, Yref, REL)
    assert b.device_status() == 0


@pytest.mark.parametrize("n,H,W,C,N,K", [
    (2, 8, 8, 64, 64, 4),        # two images per row tile
    (1, 16, 16, 96, 160, 8),     # 8 image rows per tile
    (2, 32, 32, 320, 320, 16),   # 4 image rows per tile, G = 16
    (1, 64, 64, 64, 128, 3),     # 2 image rows per tile
])
def test_conv3x3_w4a6(n, H, W, C, N, K):
    torch, b = gpu()
    P = H * W
    Xcal = synth.activations(11, 100, 2 * n, P, C, None, None, token_outliers=False)
    X = synth.activations(11, 1, n, P, C, None, None, token_outliers=False)
    Wt = synth.conv_weights(11, 2, N, C)
    bias = synth.bias(11, 3, N)
    gr = oc.calibrate(Xcal, P, 6, K, dim_select=oc.DIM_CHANNEL)
    g = b.calibrate_groups(to_dev(torch, Xcal), P, 6, K, b.DIM_CHANNEL)
    wq, sw = ol.weight_rtn(Wt, 4)
    codes, s_rows, z_rows = ol.quantize_static(X, gr, 0)
    Yref = ol.group_conv3x3(codes.reshape(n, H, W, C), gr.scale[0][0], gr.zp[0][0], gr.col_group, wq, sw, bias)
    conv = (n, H, W, C)
    w = b.weight_prepare(g, to_dev(torch, Wt), 4, conv=conv)
    Xq, _, _ = b.quantize_act(g, to_dev(torch, X), layout=b.CODES_S8_CENTRED)
    Y = b.linear(g, w, Xq, layout=b.CODES_S8_CENTRED, bias=to_dev(torch, bias), conv=conv)
    assert b.device_status() == 0
    check_output(Y, Yref.reshape(n * P, N), REL)


@pytest.mark.parametrize("w_bits", [8, 4])
@pytest.mark.parametrize("M,N", [
    (128, 9440),      # 59 blocks of 160 columns, 148 of 64: as many narrow tiles as the GPU has SMs
    (128, 9472),      # the same from blocks of 128
    (77, 9600),       # 150 narrow blocks: one too many, wide tiles
    (77, 10240), (128, 10240),   # the feed-forward of the 8 x 8 level, batch 1 and 2
    (128, 11840),     # the last width whose wide blocks leave half of the SMs free
    (256, 5120),      # two row blocks: 160 narrow tiles
])
def test_narrow_tile_rule(M, N, w_bits):
    torch, b = gpu()
    rng = np.random.default_rng(N + M)
    C = 72
    cg = (np.arange(C) % 2).astype(np.int32)
    g = b.groups_from_host(C, 1, 8, cg, np.zeros(1, np.int32), np.full((1, 1, 2), 0.03, np.float32),
                           np.full((1, 1, 2), 120, np.int32))
    W = rng.normal(0, 0.02, (N, C)).astype(np.float16)
    bias = rng.normal(0, 0.01, N).astype(np.float16)
    wq, sw = ol.weight_rtn(W, w_bits)
    w = b.weight_prepare(g, to_dev(torch, W), w_bits)
    X = rng.normal(0, 1, (M, C)).astype(np.float16)
    codes, s_rows, z_rows = ol.quantize_dynamic_token(X, cg, 2, 8)
    Xq, ds, dz = b.quantize_act(g, to_dev(torch, X), mode=b.MODE_DYNAMIC_TOKEN)
    Y = torch.full((M, N), float("nan"), dtype=torch.float16, device="cuda")
    b.linear(g, w, Xq, mode=b.MODE_DYNAMIC_TOKEN, dyn_scale=ds, dyn_zp=dz, bias=to_dev(torch, bias), out=Y)
    check_output(Y, ol.group_linear(codes, s_rows, z_rows, cg, wq, sw, bias), REL)
    assert b.device_status() == 0


def test_linear_argument_errors():
    torch, b = gpu()
    Xcal, X, W, bias, gr = layer_case(12, 1, 128, 64, 64, 2, 8, oc.DIM_CHANNEL)
    g = b.calibrate_groups(to_dev(torch, Xcal), 128, 8, 2, b.DIM_CHANNEL)
    w = b.weight_prepare(g, to_dev(torch, W), 8)
    Xq, _, _ = b.quantize_act(g, to_dev(torch, X))
    with pytest.raises(b.DgqError) as e:          # dynamic mode without its parameter arrays
        b.linear(g, w, Xq, mode=b.MODE_DYNAMIC_TOKEN)
    assert e.value.status == 1
    with pytest.raises(b.DgqError) as e:          # conv descriptor on a linear weight
        b.linear(g, w, Xq, conv=(1, 8, 16, 64))
    assert e.value.status == 1
    Y = torch.empty((128, 72), dtype=torch.float16, device="cuda")[:, 4:68]
    with pytest.raises(b.DgqError) as e:          # output not 16-byte aligned
        b.linear(g, w, Xq, out=Y)
    assert e.value.status == 2


@pytest.mark.parametrize("w_bits", [8, 4])
def test_objects_rebuilt_from_exports_give_identical_results(w_bits):
    """dgq_groups_export -> dgq_groups_from_host and dgq_weight_export -> dgq_weight_from_codes: the rebuilt
    grouping has the same layout and tables, the rebuilt weight the same codes, and the layer output is bit for
    bit the same (static grid with pixel and channel groups)."""
    torch, b = gpu()
    P, C, N, K = 256, 320, 320, 4
    Xcal, X, W, bias, gr = layer_case(14, 2, P, C, N, K, 8, oc.DIM_BOTH)
    g = b.calibrate_groups(to_dev(torch, Xcal), P, 8, K, b.DIM_BOTH)
    ex = g.export()
    g2 = b.groups_from_host(C, P, 8, ex["col_group"], ex["row_group"], ex["scale"], ex["zp"])
    ex2 = g2.export()
    assert (g2.G, g2.R, g2.T, g2.K_pad, g2.bits) == (g.G, g.R, g.T, g.K_pad, g.bits)
    for k in ("perm", "col_group", "group_off", "row_group", "scale", "zp"):
        assert np.array_equal(ex[k], ex2[k]), k
    w = b.weight_prepare(g, to_dev(torch, W), w_bits)
    wq, sw = w.export()
    w2 = b.weight_from_codes(g2, wq, sw, w_bits)
    wq2, sw2 = w2.export()
    assert np.array_equal(wq, wq2) and np.array_equal(sw, sw2)
    Xd, bd = to_dev(torch, X), to_dev(torch, bias)
    Xq, _, _ = b.quantize_act(g, Xd)
    Xq2, _, _ = b.quantize_act(g2, Xd)
    assert torch.equal(Xq, Xq2)
    Y = b.linear(g, w, Xq, bias=bd)
    Y2 = b.linear(g2, w2, Xq2, bias=bd)
    assert torch.equal(Y, Y2)
    codes, s_rows, z_rows = ol.quantize_static(X, gr, 0)
    check_output(Y2, ol.group_linear(codes, s_rows, z_rows, gr.col_group, *ol.weight_rtn(W, w_bits), bias), REL)
    assert b.device_status() == 0


def test_four_bit_weights_with_and_without_workspace():
    """4-bit weights take two routes: expanded once per call into the caller's workspace in front of the GEMM, or,
    without a workspace, expanded stage by stage inside it.  Same integers either way: identical outputs."""
    torch, b = gpu()
    M, C, N, K = 1000, 640, 640, 8
    Xcal, X, W, bias, gr = layer_case(15, 1, M, C, N, K, 8, oc.DIM_CHANNEL)
    g = b.calibrate_groups(to_dev(torch, Xcal), M, 8, K, b.DIM_CHANNEL)
    w = b.weight_prepare(g, to_dev(torch, W), 4)
    need = b.linear_workspace_bytes(g, w, M)
    assert need > 0
    Xq, ds, dz = b.quantize_act(g, to_dev(torch, X), mode=b.MODE_DYNAMIC_TOKEN)
    kw = dict(mode=b.MODE_DYNAMIC_TOKEN, dyn_scale=ds, dyn_zp=dz, bias=to_dev(torch, bias))
    Y_ws = b.linear(g, w, Xq, workspace=torch.empty(need, dtype=torch.uint8, device="cuda"), **kw)
    Y_in = b.linear(g, w, Xq, workspace=False, **kw)
    assert torch.equal(Y_ws, Y_in)
    with pytest.raises(b.DgqError) as e:          # a workspace that is too small is refused
        b.linear(g, w, Xq, workspace=torch.empty(need // 2, dtype=torch.uint8, device="cuda"), **kw)
    assert e.value.status == 4
    codes, s_rows, z_rows = ol.quantize_dynamic_token(X, gr.col_group, gr.G, gr.bits)
    check_output(Y_ws, ol.group_linear(codes, s_rows, z_rows, gr.col_group, *ol.weight_rtn(W, 4), bias), REL)
    assert b.device_status() == 0


@pytest.mark.parametrize("w_bits,M", [(8, 1), (4, 200)])
def test_bias_may_come_from_a_kernel_still_running(w_bits, M):
    """A layer whose bias is a row of another layer's output (as a time embedding added per channel is), with a tiny
    quantizer in between that lets the second GEMM start while the first still runs: the bias is read after the wait."""
    torch, b = gpu()
    C, N = 320, 328
    Xcal, X, W, bias, gr = layer_case(19, 1, 512, C, N, 8, 8, oc.DIM_CHANNEL)
    g = b.calibrate_groups(to_dev(torch, Xcal), 512, 8, 8, b.DIM_CHANNEL)
    w1, w2 = b.weight_prepare(g, to_dev(torch, W), 8), b.weight_prepare(g, to_dev(torch, W), w_bits)
    big = to_dev(torch, np.tile(X, (64, 1)))
    x = to_dev(torch, X[:M])
    kw = dict(mode=b.MODE_DYNAMIC_TOKEN)
    xq, ds, dz = b.quantize_act(g, big, **kw)
    xq2, ds2, dz2 = b.quantize_act(g, x, **kw)
    y1 = b.linear(g, w1, xq, dyn_scale=ds, dyn_zp=dz, **kw)
    torch.cuda.synchronize()
    ref = b.linear(g, w2, xq2, dyn_scale=ds2, dyn_zp=dz2, bias=y1[-1], **kw)
    for _ in range(5):
        y1.fill_(float("nan"))
        b.linear(g, w1, xq, dyn_scale=ds, dyn_zp=dz, out=y1, **kw)
        b.quantize_act_into(g, x, xq2, ds2, dz2, **kw)
        y2 = b.linear(g, w2, xq2, dyn_scale=ds2, dyn_zp=dz2, bias=y1[-1], **kw)
        torch.cuda.synchronize()
        assert torch.equal(y2, ref)
    assert b.device_status() == 0


def test_workspace_belongs_to_the_stream_of_the_call():
    """A call on another stream than the current one, still waiting there when it returns: its workspace is not given to
    the next allocation on the current stream."""
    torch, b = gpu()
    M, C, N = 2500, 640, 1280
    Xcal, X, W, bias, gr = layer_case(17, 1, M, C, N, 8, 8, oc.DIM_CHANNEL)
    g = b.calibrate_groups(to_dev(torch, Xcal), M, 8, 8, b.DIM_CHANNEL)
    w = b.weight_prepare(g, to_dev(torch, W), 4)
    Xq, ds, dz = b.quantize_act(g, to_dev(torch, X), mode=b.MODE_DYNAMIC_TOKEN)
    kw = dict(mode=b.MODE_DYNAMIC_TOKEN, dyn_scale=ds, dyn_zp=dz)
    Y_ref = b.linear(g, w, Xq, **kw)
    Q, K, V = [to_dev(torch, x) for x in synth.attention_inputs(18, 8, 16, 260, 77, 80, ctx_dim=16)]
    O_ref, _, _ = b.cross_attn_logq(Q, K, V, 8)
    Y, O = torch.empty_like(Y_ref), torch.empty_like(O_ref)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)
    b.linear(g, w, Xq, out=Y, stream=side, **kw)
    b.cross_attn_logq(Q, K, V, 8, out=O, stream=side)
    need = [b.linear_workspace_bytes(g, w, M), b.cross_attn_workspace_bytes(8, 16, 260, 77, 80)]
    taken = [torch.full((n,), 0x77, dtype=torch.uint8, device="cuda") for n in need]
    torch.cuda.current_stream().synchronize()
    side.synchronize()
    assert torch.equal(Y, Y_ref) and torch.equal(O, O_ref) and b.device_status() == 0
    assert all(bool((t == 0x77).all()) for t in taken)    # and the other way round


def test_a_wait_that_runs_out_is_reported_and_leaves_the_device_usable():
    """Every device-side wait is bounded.  The library's self-test kernel runs both of the kernels' wait functions, with
    a short limit (2000 x 1024 clocks, about a millisecond), on a barrier nobody arrives at, each beside a warp that waits
    with the usual limit of a second and has to leave with it: the kernel is over long before that second, the status
    word reads DGQ_ERR_TIMEOUT once, is clear afterwards, and a layer call right after it gives the right result."""
    torch, b = gpu()
    assert b.device_status() == 0
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record()
    b.selftest_wait_timeout(2000)
    end.record()
    end.synchronize()
    assert 1.0 <= start.elapsed_time(end) < 500.0    # 2 048 000 clocks at up to 1965 MHz
    assert b.device_status() == 6
    assert b.device_status() == 0
    Xcal, X, W, bias, gr = layer_case(16, 1, 256, 320, 320, 4, 8, oc.DIM_CHANNEL)
    g = b.calibrate_groups(to_dev(torch, Xcal), 256, 8, 4, b.DIM_CHANNEL)
    _run_linear(torch, b, X, W, bias, gr, g, "dynamic", 8)
