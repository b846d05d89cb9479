"""GPU parity of the attention kernels at the edges of their launch rules: rows per block of the cross-attention, teams
and key blocks of the self-attention."""
import pytest

from paper_2501_04304_b200 import synth
from dgq_testlib import gpu
from test_gpu_attention import _compare
from test_gpu_self_attention import _compare as _compare_self, _qkv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,nq,d,bits", [
    (9, 16, 257, 40, 8),     # 432 blocks of 128 rows, 288 of 256: two row tiles per warp, last block of one row
    (5, 20, 300, 80, 4),     # the same with the widest head that has them
    (4, 20, 300, 64, 8),     # 240 blocks of 128 rows: one row tile per warp
    (10, 16, 260, 80, 8),    # 320 blocks of 256 rows: two kernels
])
def test_cross_attention_rows_per_block(B, H, nq, d, bits):
    torch, b = gpu()
    Q, K, V = synth.attention_inputs(6, B, H, nq, 77, d, ctx_dim=64)
    _compare(torch, b, Q, K, V, bits)


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("n,nk,d", [
    (20, 100, 80),           # one key block: one team has no tile in a walk
    (140, 300, 80),          # an odd number of key blocks: the teams' shares differ
    (260, 129, 40),          # two query tiles, the second key block holds one key
    (130, 400, 128),
    (130, 257, 160),         # a single P tile: one team
])
def test_self_attention_teams(n, nk, d, bits):
    torch, b = gpu()
    Q, K, V = _qkv(7, 1, 2, n, d, nk)
    _compare_self(torch, b, Q, K, V, bits)
    _compare_self(torch, b, Q, K, V, bits, fixed=[0.25])
