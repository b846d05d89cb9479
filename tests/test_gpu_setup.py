"""GPU parity of the set-up kernels at the edges of their ranges: calibration reductions on ragged recordings and
weight preparation on group sizes around the 32-position atom."""
import numpy as np
import pytest

from oracle import calibration as oc
from oracle import linear as ol
from paper_2501_04304_b200 import synth
from dgq_testlib import gpu, to_dev, oracle_grouping_matches, check_output

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,n,C,ld,dim,K", [
    (1, 1, 8, 8, oc.DIM_CHANNEL, 2),          # one row, one vector
    (31, 1, 13, 16, oc.DIM_BOTH, 3),          # a last vector of five columns, fewer rows than a block takes
    (33, 3, 2056, 2064, oc.DIM_BOTH, 4),      # more vectors than threads, ragged blocks, row groups change inside one
    (96, 1, 320, 320, oc.DIM_PIXEL, 8),
])
def test_calibration_edges(P, n, C, ld, dim, K):
    torch, b = gpu()
    X = synth.activations(31, 1, n, P, C)
    X1 = synth.activations(31, 2, n, P, C)
    buf = torch.zeros((n * P, ld), dtype=torch.float16, device="cuda")
    gr = oc.calibrate(X, P, 8, K, dim_select=dim)
    oc.fill_timestep(gr, X1, 1)
    buf[:, :C] = to_dev(torch, X)
    g = b.calibrate_groups(buf[:, :C], P, 8, K, dim, n_timesteps=2)
    buf[:, :C] = to_dev(torch, X1)
    b.calibrate_groups(buf[:, :C], P, 8, K, dim, n_timesteps=2, timestep=1, groups=g)
    oracle_grouping_matches(gr, g.export())


@pytest.mark.parametrize("w_bits", [8, 4])
@pytest.mark.parametrize("sizes,N", [
    ((8,), 8),                      # one word of members
    ((24, 25, 1, 30), 16),          # padding that just fits the atom, spills into the next, fills one alone
    ((32, 64, 7, 9), 264),          # whole atoms of padding, rows beyond N in the last tile
    ((400, 8), 72),                 # sums that eight padding positions cannot absorb at 4 bits
])
def test_weight_layout_edges(sizes, N, w_bits):
    torch, b = gpu()
    C = sum(sizes)
    rng = np.random.default_rng(C)
    cg = rng.permutation(np.repeat(np.arange(len(sizes)), sizes)).astype(np.int32)
    G, M = len(sizes), 40
    scale = rng.uniform(0.01, 0.05, (1, 1, G)).astype(np.float32)
    zp = rng.integers(100, 140, (1, 1, G)).astype(np.int32)
    g = b.groups_from_host(C, 1, 8, cg, np.zeros(1, np.int32), scale, zp)
    W = (rng.normal(0.01, 0.02, (N, C))).astype(np.float16)   # biased, so that a group's sum outgrows its padding
    W[N - 1] = 0
    wq, sw = ol.weight_rtn(W, w_bits)
    w = b.weight_prepare(g, to_dev(torch, W), w_bits)
    got, got_sw = w.export()
    assert np.array_equal(got, wq) and np.array_equal(got_sw, sw)
    w2 = b.weight_from_codes(g, wq, sw, w_bits)
    X = rng.normal(0, 1, (M, C)).astype(np.float16)
    codes = np.clip(np.rint(X.astype(np.float32) * (np.float32(1) / scale[0, 0, cg])) + zp[0, 0, cg], 0, 255).astype(np.int64)
    Xq, _, _ = b.quantize_act(g, to_dev(torch, X))
    Y, Y2 = b.linear(g, w, Xq), b.linear(g, w2, Xq)
    assert torch.equal(Y, Y2) and b.device_status() == 0
    s_rows, z_rows = np.broadcast_to(scale[0], (M, G)), np.broadcast_to(zp[0], (M, G))
    check_output(Y, ol.group_linear(codes, s_rows, z_rows, cg, wq, sw, None))


@pytest.mark.parametrize("mode", ["static", "dynamic"])
@pytest.mark.parametrize("M,sizes,bits", [
    (1, (8,), 8),                    # one row, two chunks: a block of 64 pairs with one of them real
    (3, (1, 31, 33, 255), 6),        # odd row count, groups that end inside a chunk, 6-bit clamp
    (257, (320,), 8),                # a cell that covers a whole warp
    (2601, (300, 188), 8),           # 32 chunks: a warp per row pair, several batches, odd row count
    (9, (5112, 8), 8),               # one pair per block, more chunks than a small block has threads
    (4100, (8184, 8), 4),            # the widest layer, several batches per block, rows asked for two batches ahead
    (2367, (1500, 36), 8),           # 100 chunks, one round of the device with two pairs per block
    (3551, (1100, 20), 8),           # 72 chunks, one round with three
    (18947, (512, 512, 512), 8),     # two pairs per block and rows asked for ahead, odd row count, no group of more than half
])
def test_quantizer_edges(M, sizes, bits, mode):
    torch, b = gpu()
    C, G = sum(sizes), len(sizes)
    rng = np.random.default_rng(M)
    cg = rng.permutation(np.repeat(np.arange(G), sizes)).astype(np.int32)
    scale = rng.uniform(0.01, 0.05, (1, 1, G)).astype(np.float32)
    zp = rng.integers(0, 2 ** bits, (1, 1, G)).astype(np.int32)
    g = b.groups_from_host(C, 1, bits, cg, np.zeros(1, np.int32), scale, zp)
    X = rng.normal(0, 1, (M, C)).astype(np.float16)
    ex = g.export()
    L = 2 ** bits - 1
    Xq, ds, dz = b.quantize_act(g, to_dev(torch, X), mode=b.MODE_DYNAMIC_TOKEN if mode == "dynamic" else b.MODE_STATIC)
    if mode == "dynamic":
        codes, s_rows, z_rows = ol.quantize_dynamic_token(X, cg, G, bits)
        assert np.array_equal(ds.cpu().numpy(), s_rows) and np.array_equal(dz.cpu().numpy(), z_rows)
    else:
        inv = (np.float32(1) / scale[0, 0]).astype(np.float32)
        codes = np.clip(np.rint(X.astype(np.float32) * inv[cg]) + zp[0, 0, cg], 0, L).astype(np.int64)
        z_rows = np.broadcast_to(zp[0], (M, G))
    full = Xq.cpu().numpy().astype(np.int64)
    valid = ex["perm"] >= 0
    assert np.array_equal(full[:, valid], codes[:, ex["perm"][valid]])
    group_of = np.repeat(np.arange(G), np.diff(ex["group_off"]))
    assert np.array_equal(full[:, ~valid], np.clip(z_rows, 0, L)[:, group_of[~valid]])   # padding = clamped zero-point
    assert b.device_status() == 0


@pytest.mark.parametrize("M,N,sizes", [
    (130, 64, (856,)),                       # 27 atoms: the longest reduction of one producer
    (130, 64, (24, 856)),                    # 28 atoms, a group that ends inside a stage
    (130, 64, (24, 880, 8)),                 # 30 atoms: the shortest of two producers, ragged last stage
    (300, 320, (56, 2000, 24, 24, 88, 600)),  # long reduction whose groups begin at every atom of a stage
    (2500, 1280, (120, 1000, 24)),           # more tiles than half the SMs: wide tiles, several per block
])
def test_linear_reduction_lengths(M, N, sizes):
    torch, b = gpu()
    C, G = sum(sizes), len(sizes)
    rng = np.random.default_rng(C)
    cg = rng.permutation(np.repeat(np.arange(G), sizes)).astype(np.int32)
    scale = rng.uniform(0.01, 0.05, (1, 1, G)).astype(np.float32)
    zp = rng.integers(100, 140, (1, 1, G)).astype(np.int32)
    g = b.groups_from_host(C, 1, 8, cg, np.zeros(1, np.int32), scale, zp)
    W = rng.normal(0, 0.02, (N, C)).astype(np.float16)
    bias = rng.normal(0, 0.01, N).astype(np.float16)
    wq, sw = ol.weight_rtn(W, 8)
    w = b.weight_prepare(g, to_dev(torch, W), 8)
    X = rng.normal(0, 1, (M, C)).astype(np.float16)
    codes, s_rows, z_rows = ol.quantize_dynamic_token(X, cg, G, 8)
    Xq, ds, dz = b.quantize_act(g, to_dev(torch, X), mode=b.MODE_DYNAMIC_TOKEN)
    Y = torch.full((M, N), float("nan"), dtype=torch.float16, device="cuda")
    b.linear(g, w, Xq, mode=b.MODE_DYNAMIC_TOKEN, dyn_scale=ds, dyn_zp=dz, bias=to_dev(torch, bias), out=Y)
    rows = np.unique(np.r_[0:3, M // 2, M - 3:M])
    ref = ol.group_linear(codes[rows], s_rows[rows], z_rows[rows], cg, wq, sw, bias)
    check_output(Y[torch.from_numpy(rows).cuda()], ref)
    assert torch.isfinite(Y).all() and b.device_status() == 0


@pytest.mark.parametrize("M,C,N", [
    (130, 320, 64),          # few pieces: unpacked inside the GEMM although there is a workspace
    (128, 4000, 64),         # 64 pieces of 64-column tiles: the last reduction unpacked inside
    (128, 4160, 64),         # the first expanded in front
    (2500, 640, 1280),       # several tiles per block, expanded in front
    (6300, 1016, 160), (6300, 1024, 160),    # a single wide tile per block: 8 stages inside, 9 in front
    (1000, 1400, 2560), (1000, 1408, 2560),  # the same with 3 MiB of weights: 11 stages inside, 12 in front
    (20000, 792, 160),                       # two tiles on some blocks: 70 pieces in front
    (20000, 744, 160),                       # 60 inside
])
def test_four_bit_routes(M, C, N):
    torch, b = gpu()
    rng = np.random.default_rng(M + C)
    g = b.groups_from_host(C, 1, 8, np.zeros(C, np.int32), np.zeros(1, np.int32), np.full((1, 1, 1), 0.03, np.float32),
                           np.full((1, 1, 1), 120, np.int32))
    W = rng.normal(0, 0.02, (N, C)).astype(np.float16)
    wq, sw = ol.weight_rtn(W, 4)
    w = b.weight_prepare(g, to_dev(torch, W), 4)
    X = rng.normal(0, 1, (M, C)).astype(np.float16)
    Xq, ds, dz = b.quantize_act(g, to_dev(torch, X), mode=b.MODE_DYNAMIC_TOKEN)
    kw = dict(mode=b.MODE_DYNAMIC_TOKEN, dyn_scale=ds, dyn_zp=dz)
    Y = b.linear(g, w, Xq, **kw)
    assert torch.equal(Y, b.linear(g, w, Xq, workspace=False, **kw))
    rows = np.unique(np.r_[0:3, M // 2, M - 2:M])
    codes, s_rows, z_rows = ol.quantize_dynamic_token(X[rows], np.zeros(C, np.int32), 1, 8)
    check_output(Y[torch.from_numpy(rows).cuda()], ol.group_linear(codes, s_rows, z_rows, np.zeros(C, np.int32), wq, sw, None))
    assert b.device_status() == 0


def _weight(torch, b, rng, N, C, w_bits, conv):
    """A prepared weight of two channel groups and its codes and scales."""
    g = b.groups_from_host(C, 1, 8 if not conv else 6, (np.arange(C) % 2).astype(np.int32), np.zeros(1, np.int32),
                           np.full((1, 1, 2), 0.03, np.float32), np.full((1, 1, 2), 31, np.int32))
    W = rng.normal(0, 0.02, (N, (9 if conv else 1) * C)).astype(np.float16)
    wq, sw = ol.weight_rtn(W, w_bits)
    return g, W, wq, sw


@pytest.mark.parametrize("w_bits", [8, 4])
@pytest.mark.parametrize("N,C,conv", [
    (8, 256, False),         # 2^11 codes: the last weight put in order on the host
    (8, 264, False),         # the first on the device
    (8, 24, True), (264, 24, True),
])
def test_weight_export_routes_and_during_a_capture(N, C, conv, w_bits):
    """An export copies host memory as far as its caller can tell: also while the caller captures a graph."""
    torch, b = gpu()
    g, W, wq, sw = _weight(torch, b, np.random.default_rng(N + C), N, C, w_bits, conv)
    w = b.weight_prepare(g, to_dev(torch, W), w_bits, conv=(1, 16, 8, C) if conv else None)
    x = torch.arange(64.0, device="cuda")
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        y = x + 1
        got, got_sw = w.export()
        z = y * 2
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(got, wq) and np.array_equal(got_sw, sw)
    assert torch.equal(z, (x + 1) * 2)
    again, _ = w.export()
    assert np.array_equal(again, wq) and b.device_status() == 0


def test_weight_of_another_device_than_the_current_one():
    """Building a weight from groups and fp16 weights of another device, and exporting it while a third party's device is
    current, read each array where it lies."""
    torch, b = gpu()
    if torch.cuda.device_count() < 2:
        pytest.skip("one GPU")
    g, W, wq, sw = _weight(torch, b, np.random.default_rng(3), 264, 320, 4, False)
    Wd = to_dev(torch, W)
    with torch.cuda.device(1):
        w = b.weight_prepare(g, Wd, 4)
    got, got_sw = w.export()
    assert np.array_equal(got, wq) and np.array_equal(got_sw, sw)


@pytest.mark.parametrize("w_bits", [8, 4])
def test_weights_that_are_not_finite(w_bits):
    """A NaN gets code 0 and does not count for its row's scale; an infinity makes the row's scale infinite and its codes
    0 (the fp32 sequence with NaN -> 0, as for activations)."""
    torch, b = gpu()
    rng = np.random.default_rng(9)
    g, W, _, _ = _weight(torch, b, rng, 16, 72, w_bits, False)
    finite = W.copy()
    finite[2, 5] = finite[2, 70] = 0
    wq, sw = ol.weight_rtn(finite, w_bits)
    W[2, 5], W[2, 70] = np.nan, -np.nan
    W[7, 0] = np.inf
    wq[7], sw[7] = 0, np.inf
    got, got_sw = b.weight_prepare(g, to_dev(torch, W), w_bits).export()
    assert np.array_equal(got, wq) and np.array_equal(got_sw, sw)
