"""GPU parity: attention with log2-quantized scores over all keys (self-attention) against the fp64 oracle."""
import numpy as np
import pytest

from oracle import attention as oa
from paper_2501_04304_b200 import synth
from dgq_testlib import gpu, to_dev, check_output, check_codes, flipped_output_bound

pytestmark = pytest.mark.gpu


def _compare(torch, b, Q, K, V, bits, fixed=None, out_rel=1e-3):
    O_ref, codes_ref, s_ref, A = oa.self_attn_logq(Q, K, V, bits, fixed)
    fx = to_dev(torch, np.asarray(fixed, np.float32)) if fixed is not None else None
    O, codes = b.self_attn_logq(to_dev(torch, Q), to_dev(torch, K), to_dev(torch, V), bits, fx, want_codes=True)
    torch.cuda.synchronize()
    assert b.device_status() == 0
    c = codes.cpu().numpy().astype(np.int64)
    diff = check_codes(c, codes_ref)
    # a score on a rounding boundary may take either neighbouring level: every row is held to the oracle's
    # output with the allowance its flipped codes (if any) explain, and to the product evaluated with the
    # codes the kernel chose
    Og = O.float().cpu().numpy().astype(np.float64)
    bound = out_rel * np.max(np.abs(O_ref)) + flipped_output_bound(diff, c, codes_ref, s_ref, V)
    assert np.all(np.abs(Og - O_ref) <= bound), f"max excess {np.max(np.abs(Og - O_ref) - bound):.3e}"
    check_output(O, oa.self_product(c, s_ref, V), out_rel)
    # the variant that writes no codes gives the same output
    O2, _ = b.self_attn_logq(to_dev(torch, Q), to_dev(torch, K), to_dev(torch, V), bits, fx)
    assert torch.equal(O, O2)


def _qkv(seed, B, H, n, d, nk=None):
    """Self-attention inputs: queries, keys and values of the same n tokens (seeded normal fp16)."""
    rng = np.random.default_rng((seed, 77))
    nk = n if nk is None else nk
    Q = rng.normal(0, 1, (B, n, H, d)).astype(np.float16)
    K = rng.normal(0, 1, (B, nk, H, d)).astype(np.float16)
    V = rng.normal(0, 1, (B, nk, H, d)).astype(np.float16)
    return Q, K, V


@pytest.mark.parametrize("bits", [8, 4])
def test_small_self_attention(bits):
    torch, b = gpu()
    Q, K, V = _qkv(1, 2, 3, 300, 40)          # 5 key blocks, ragged last block, ragged row block
    _compare(torch, b, Q, K, V, bits)


@pytest.mark.parametrize("B,H,n,nk,d", [
    (1, 1, 16, 3, 40),        # one partial key block
    (2, 2, 64, 64, 64),       # exactly one key block
    (1, 2, 130, 257, 80),     # nk != nq, ragged everything
    (1, 1, 129, 128, 128),
    (1, 2, 70, 65, 160),
])
def test_shapes(B, H, n, nk, d):
    torch, b = gpu()
    Q, K, V = _qkv(2, B, H, n, d, nk)
    _compare(torch, b, Q, K, V, 8)


def test_fixed_scale():
    torch, b = gpu()
    Q, K, V = _qkv(3, 2, 2, 200, 40)
    _compare(torch, b, Q, K, V, 6, fixed=[1.0, 0.25])


@pytest.mark.parametrize("d", [40, 64, 80, 128, 160])
@pytest.mark.parametrize("bits", [2, 3, 4, 5, 6])
def test_few_codes(bits, d):
    """Up to 5 bits the last code's weight is not an fp16 zero (2^-17 at 5 bits, below the normal fp16 numbers): logits spread far
    beyond the last code, so most scores carry that weight, and with values of one sign it shows in the output (at 4 bits 380 x 2^-15,
    12 times the tolerance; at 5 bits it does not).  6 bits is the first count whose last codes are fp16 zeros, another kernel.
    Bounds as in the other cases."""
    torch, b = gpu()
    Q, K, V = _qkv(60 + bits, 1, 2, 385, d)
    _compare(torch, b, Q * np.float16(8), K, np.abs(V), bits)


@pytest.mark.parametrize("d", [40, 64, 80, 128, 160])
@pytest.mark.parametrize("n", [127, 128, 129, 257, 385, 513, 640])
@pytest.mark.parametrize("bits,fixed", [(8, None), (4, None), (8, [0.5])])
def test_key_block_counts(n, d, bits, fixed):
    """One to five key blocks, full and ragged: every stage of the K ring is used again, and for heads of 40 and 64 every phase of the score
    buffers meets the change from the walks that use four of them to the one that uses two.  Bounds as in the
    other cases: codes within one level, outputs 1e-3 plus what a moved code explains."""
    torch, b = gpu()
    Q, K, V = _qkv(20 + n, 1, 2, n, d)
    _compare(torch, b, Q, K, V, bits, fixed)


def test_level_at_1024_tokens():
    """32 x 32 level: 1024 tokens, 8 heads of 80 features; the whole output against the oracle."""
    torch, b = gpu()
    Q, K, V = _qkv(4, 1, 8, 1024, 80)
    _compare(torch, b, Q, K, V, 8)


@pytest.mark.parametrize("B,H,n,d", [
    (4, 10, 2048, 64),        # 320 CTAs of two query tiles
    (8, 8, 1024, 80),         # 512 CTAs of one
    (4, 8, 1024, 128),        # 256
    (8, 8, 1024, 160),        # 512, the softmax warps in one team
])
def test_several_rounds_of_ctas(B, H, n, d):
    """More CTAs than the device holds at once (one per SM), so that their key and value loads compete and land late: a wait that passes
    before its load would show as a time-out or as wrong rows.  Five calls give the same bits, no wait ran out,
    and sampled rows of every prompt and head are held to the oracle with the bounds of the other cases."""
    torch, b = gpu()
    Q, K, V = _qkv(80 + d, B, H, n, d)
    dev = [to_dev(torch, x) for x in (Q, K, V)]
    O, codes = b.self_attn_logq(*dev, 8, want_codes=True)
    for _ in range(5):
        again, _ = b.self_attn_logq(*dev, 8)
        assert torch.equal(O, again)
    assert b.device_status() == 0
    rows = np.random.default_rng(d).choice(n, 12, replace=False)
    O_ref, codes_ref, s_ref, _ = oa.self_attn_logq(Q[:, rows], K, V, 8)
    at = torch.from_numpy(rows).cuda()
    c = codes[:, :, at].cpu().numpy().astype(np.int64)
    diff = check_codes(c, codes_ref)
    Og = O[:, at].float().cpu().numpy().astype(np.float64)
    bound = 1e-3 * np.max(np.abs(O_ref)) + flipped_output_bound(diff, c, codes_ref, s_ref, V)
    assert np.all(np.abs(Og - O_ref) <= bound), f"max excess {np.max(np.abs(Og - O_ref) - bound):.3e}"


def test_argument_errors():
    torch, b = gpu()
    Q, K, V = [to_dev(torch, x) for x in _qkv(5, 1, 1, 16, 40)]
    with pytest.raises(Exception):
        b.self_attn_logq(Q, K, V, 9)
    Q48 = torch.zeros((1, 16, 1, 48), dtype=torch.float16, device="cuda")
    with pytest.raises(Exception):
        b.self_attn_logq(Q48, Q48, Q48, 8)


def test_codes_against_64_bits():
    """How often a code is the neighbour of the one that 64-bit arithmetic gives on the same fp16 inputs, over 2.7e8 scores.
    The boundaries lie one unit apart in the log2 domain, so the share of such codes is about the mean error of the
    logit distance.  Its parts: the row maximum's product with the scale (half a unit in the last place of numbers up to 8,
    2^-22), the fp32 accumulation of the logits (2^-23 and below) and the exponential (2^-22 relative, times log2 e).
    Together below 2^-21."""
    torch, b = gpu()
    B, H, n, d = 2, 8, 4096, 40
    gen = torch.Generator(device="cuda").manual_seed(11)
    q, k, v = (torch.randn(B, n, H, d, generator=gen, device="cuda").half() for _ in range(3))
    _, codes = b.self_attn_logq(q, k, v, 8, want_codes=True)
    flips, largest = 0, 0
    for i in range(B):
        for h in range(H):
            t = q[i, :, h].double() @ k[i, :, h].double().T * (np.log2(np.e) / np.sqrt(d))
            ref = torch.clamp(torch.round(t.amax(1, keepdim=True) - t), 0, 255)
            diff = (codes[i, h].double() - ref).abs()
            flips, largest = flips + int((diff != 0).sum()), max(largest, int(diff.max()))
    assert largest <= 1 and flips <= codes.numel() * 2.0 ** -21, flips
    assert b.device_status() == 0
