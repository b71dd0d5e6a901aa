"""Attention with the keys split over a cluster of CTAs, against the oracle.

The rule takes 2, 4 or 8 CTAs per (tile pair, head) when the pairs alone leave
SMs idle; the sizes below fall on every width, with key blocks that do not
divide evenly, a last block of one key and ragged query tiles.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

import oracle                                      # noqa: E402
from synth import generate as G                    # noqa: E402

F32 = np.float32


@pytest.fixture(scope="module")
def ec():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2608_02474_gb300 import echocache
    return echocache


def bf(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", torch.bfloat16)


def check(ec, Q, KV, H, d):
    D = H * d
    kvd = bf(KV)
    out = ec.echo_attention(bf(Q), kvd[:, :D], kvd[:, D:], H, d).float().cpu().numpy()
    ref = oracle.block.mha(Q.astype(np.float64), KV[:, :D].astype(np.float64),
                           KV[:, D:].astype(np.float64), H)
    # P and the result in bf16 (2^-9 each), sums in fp32: the bar of the one-CTA form
    rel = np.abs(out - ref).max(axis=1) / np.abs(ref).max(axis=1)
    assert rel.max() <= 2e-2 and np.abs(out - ref).sum() / np.abs(ref).sum() <= 5e-3
    assert ec.echo_get_device_error() == 0


@pytest.mark.parametrize("M,L,H,d", [
    (1, 1025, 1, 64),        # 8 CTAs, 9 blocks, the last of one key
    (257, 1025, 1, 128),     # two tile pairs, the second of one row
    (130, 7801, 2, 64),      # 8 CTAs, 61 blocks: 7 or 8 each
    (389, 2000, 16, 64),     # 4 CTAs
    (256, 2500, 19, 128),    # 4 or 8 CTAs, whole tiles
    (600, 1999, 16, 128),    # 2 CTAs
    (1100, 900, 12, 64),     # 2 CTAs, 8 blocks
    (300, 2049, 40, 64),     # one CTA per tile pair, the last block of one key
    (257, 2200, 76, 64),     # 152 CTAs, an odd number of blocks
])
def test_attention_split_keys(ec, M, L, H, d):
    D = H * d
    check(ec, G.random_rows(M, D, seed=M + d, scale=1.5),
          G.random_rows(L, 2 * D, seed=L + d, scale=1.5), H, d)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("H", [2, 40])       # keys split over a cluster; one CTA per tile pair
def test_attention_late_maxima(ec, d, H):
    """Keys whose logits exceed the first block's by far more than 2^64 in one half
    of a later block only: the rescale path, which both halves of a row take."""
    M, L = 300, 2100
    D = H * d
    g = np.random.default_rng(d + H)
    Q = np.full((M, D), 2.0, dtype=F32) + g.standard_normal((M, D)).astype(F32) * F32(0.05)
    K = g.standard_normal((L, D)).astype(F32) * F32(0.1)
    K[700:710] += F32(3.0)
    K[1500:1505] += F32(6.0)
    V = g.standard_normal((L, D)).astype(F32)
    Q, K, V = (G.to_bf16_values(a) for a in (Q, K, V))
    check(ec, Q, np.concatenate([K, V], axis=1), H, d)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("lo,hi", [(0, 300), (3000, 4000), (1900, 2100)])
def test_attention_split_maxima_differ(ec, d, lo, hi):
    """Keys lo..hi hold nearly all of the weight: the CTAs' maxima lie far
    apart, and all but one or two of them contribute next to nothing."""
    H, M, L = 2, 150, 4000
    D = H * d
    g = np.random.default_rng(d)
    Q = np.full((M, D), 2.0, dtype=F32) + g.standard_normal((M, D)).astype(F32) * F32(0.05)
    K = g.standard_normal((L, D)).astype(F32) * F32(0.1)
    K[lo:hi] += F32(3.0)
    V = g.standard_normal((L, D)).astype(F32)
    Q, K, V = (G.to_bf16_values(a) for a in (Q, K, V))
    check(ec, Q, np.concatenate([K, V], axis=1), H, d)


@pytest.mark.parametrize("d", [64, 128])
def test_attention_split_first_keys_minus_infinity(ec, d):
    """8 CTAs of four key blocks each; the first block of all but one scores -inf, and
    every other score lies near -200 (in powers of two), far below 2^-126 of one: a
    CTA has to take its maximum from the block after."""
    H, M, L = 2, 150, 4000
    D = H * d
    g = np.random.default_rng(d)
    Q = g.standard_normal((M, D)).astype(F32) * F32(0.3)
    K = g.standard_normal((L, D)).astype(F32) * F32(0.3)
    V = g.standard_normal((L, D)).astype(F32)
    for h in range(H):
        Q[:, h * d] = 1.0
        K[:, h * d] = -200 / np.log2(np.e) * np.sqrt(d)
        for r in range(1, 8):
            K[512 * r:512 * r + 128, h * d] = -np.inf
    Q, K, V = (G.to_bf16_values(a) for a in (Q, K, V))
    check(ec, Q, np.concatenate([K, V], axis=1), H, d)


@pytest.mark.parametrize("M,L,H,d", [(7800, 1000, 16, 64), (7800, 2100, 16, 64), (389, 2000, 16, 64),
                                     (3000, 2100, 8, 128)])
def test_attention_repeats(ec, M, L, H, d):
    """The same call gives the same bits every time.  (A wait for the last P V that
    took the one before it for done gave a few wrong rows in up to 4% of launches.)"""
    import torch
    D = H * d
    g = torch.Generator(device="cuda").manual_seed(M)
    Q = torch.randn(M, D, generator=g, device="cuda").bfloat16()
    KV = torch.randn(L, 2 * D, generator=g, device="cuda").bfloat16()
    ref = ec.echo_attention(Q, KV[:, :D], KV[:, D:], H, d).clone()
    outs = [torch.empty_like(ref) for _ in range(8)]
    bad = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(100):
        for o in outs:
            ec.echo_attention(Q, KV[:, :D], KV[:, D:], H, d, out=o)
        bad += sum((o != ref).any().to(torch.int64) for o in outs)
    assert int(bad) == 0
    assert ec.echo_get_device_error() == 0


@pytest.mark.parametrize("M,L,H,d", [
    (256, 2049, 153, 64),    # a whole wave and one item over 8 CTAs, the last block of one key
    (513, 2100, 52, 64),     # 156 items: four of the second launch, the last rows ragged
    (257, 2200, 88, 128),    # 176 items: the first launch ends inside a head
    (2560, 4000, 16, 64),    # 160 items: whole tiles
    (700, 2049, 101, 64),    # 303 items: nearly two waves, one launch
])
def test_attention_last_wave(ec, M, L, H, d):
    D = H * d
    check(ec, G.random_rows(M, D, seed=M + d, scale=1.5),
          G.random_rows(L, 2 * D, seed=L + d, scale=1.5), H, d)


@pytest.mark.parametrize("M,L,H,d,launches", [
    (513, 2100, 52, 64, 2), (257, 2200, 88, 128, 2), (7800, 7800, 16, 64, 2),
    (700, 2049, 101, 64, 1), (389, 2000, 16, 64, 1), (300, 160, 16, 64, 1),
])
def test_attention_launches_are_counted(ec, M, L, H, d, launches):
    """Every kernel of a call is counted and recorded; the records' queries add up."""
    import torch
    D = H * d
    Q = torch.zeros(M, D, dtype=torch.bfloat16, device="cuda")
    KV = torch.zeros(L, 2 * D, dtype=torch.bfloat16, device="cuda")
    ec.echo_profile_read()
    n0 = ec.echo_launch_count()
    ec.echo_profile_enable(True)
    ec.echo_attention(Q, KV[:, :D], KV[:, D:], H, d)
    ec.echo_profile_enable(False)
    rec = ec.echo_profile_read()
    assert ec.echo_launch_count() - n0 == launches == len(rec)
    assert sum(r[1] for r in rec) == M and all(r[1] > 0 and r[2:4] == (L, D) for r in rec)
