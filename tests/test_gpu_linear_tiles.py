"""The projection's epilogue forms on both tile widths (256 x 128 and 256 x 256),
at ragged row counts and column counts that end inside a tile, against the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

import oracle                                      # noqa: E402
from synth import generate as G                    # noqa: E402

F32 = np.float32
SIZES = [
    # M, Kd, N
    (1, 128, 64),            # half of a 128-column tile
    (257, 192, 192),         # two row tiles, the second of one row; 1.5 column tiles
    (127, 1024, 320),
    (300, 64, 1088),
    (5000, 128, 2112),       # 128-column tiles, several per pair, the last half wide
    (5000, 256, 2112),       # 256-column tiles, several per pair, the last a quarter wide
    (4097, 320, 1600),
]


@pytest.fixture(scope="module")
def ec():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2608_02474_gb300 import echocache
    return echocache


def bf(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", torch.bfloat16)


@pytest.mark.parametrize("M,Kd,N", SIZES)
def test_linear_epilogues(ec, M, Kd, N):
    A = G.random_rows(M, Kd, seed=M + Kd)
    W = G.random_rows(N, Kd, seed=N + 1, scale=0.05)
    b = G.random_rows(1, N, seed=N + 2, scale=0.5)[0]
    lin = oracle.block.linear(A, W, b)
    Ad, Wd, bd = bf(A), bf(W), bf(b)
    # fp32 sums of Kd products: 2^-24 sqrt(Kd) of the terms' size; bf16 results 2^-8
    f_tol = dict(rtol=1e-5, atol=2e-5)
    h_tol = dict(rtol=2 ** -8, atol=1e-4)
    close = np.testing.assert_allclose

    def host(t):
        return t.float().cpu().numpy()

    close(host(ec.echo_linear(Ad, Wd, bd)), lin, **h_tol)
    close(host(ec.echo_linear(Ad, Wd, bd, act=1)), oracle.block.gelu_tanh(lin), **h_tol)
    R = G.random_rows(M + 40, N, seed=4)
    rows = np.sort(np.random.default_rng(5).permutation(M + 40)[:M]).astype(np.int32)
    close(host(ec.echo_linear(Ad, Wd, bd, resid=bf(R), resid_rows=torch.from_numpy(rows).to("cuda"),
                              out_dtype=torch.float32)), lin + R[rows], **f_tol)
    R2 = np.random.default_rng(6).standard_normal((M, N)).astype(F32)
    R2d = torch.from_numpy(R2).to("cuda")
    close(host(ec.echo_linear(Ad, Wd, bd, resid=R2d, out_dtype=torch.float32)), lin + R2, **f_tol)
    close(host(ec.echo_linear(Ad, Wd, bd, resid=R2d)), lin + R2, **h_tol)
    # a wider output: the columns beside it stay as they are
    wide = torch.full((M, N + 64), 7.0, device="cuda", dtype=torch.bfloat16)
    ec.echo_linear(Ad, Wd, None, out=wide[:, :N])
    close(host(wide[:, :N]), lin - b, **h_tol)
    assert bool((wide[:, N:] == 7).all())
    assert ec.echo_get_device_error() == 0


def test_gelu_of_every_bf16_value(ec):
    """GELU over every bf16 value, both output forms (bf16: one exponential and one
    quotient; fp32: tanhf).  The projection passes each value through unchanged.

    bf16: x / (1 + 2^w), w = -2 u log2(e), |w| <= 126 where the result is not below the
    smallest normal number.  Four fp32 roundings make w (2^-24 each, of which the ones of
    x^2 and of its factor count at most once), so 2^w is off by at most
    126 ln 2 * 4 * 2^-24 = 2.1e-5 of itself, the exponential and the quotient by 2 ulp;
    then the rounding to bf16's 8 bits, at most 2^-8.  Results below 11 * 2^-126 may vanish."""
    bits = torch.arange(65536, dtype=torch.int32).to(torch.uint16)
    x = bits.view(torch.bfloat16)
    A = torch.zeros(65536, 64, dtype=torch.bfloat16)
    A[:, 0] = x
    W = torch.zeros(64, 64, dtype=torch.bfloat16)
    W[:, 0] = 1
    A, W = A.cuda(), W.cuda()
    got16 = ec.echo_linear(A, W, None, act=1)
    got32 = ec.echo_linear(A, W, None, act=1, out_dtype=torch.float32)
    assert bool((got16.view(torch.uint16) == got16.view(torch.uint16)[:, :1]).all())
    # what the two forms make of infinities and NaN: the same
    assert torch.equal(torch.isnan(got16), torch.isnan(got32))
    assert torch.equal(torch.isinf(got16), torch.isinf(got32))
    g = got16[:, 0].double().cpu()
    v = x.double()
    fin = torch.isfinite(v)
    assert torch.isnan(g[torch.isnan(v)]).all()
    assert g[v == float("inf")] == float("inf") and torch.isnan(g[v == float("-inf")])
    assert torch.isfinite(g[fin]).all()
    v, g = v[fin], g[fin]
    u = np.sqrt(2 / np.pi) * (v + 0.044715 * v ** 3)
    exact = v / (1 + torch.exp(-2 * u))             # (1 + tanh u) / 2 without its cancellation
    assert bool(((g - exact).abs() <= (2 ** -8 + 3e-5) * exact.abs() + 11 * 2.0 ** -126).all())
    # and as often the bf16 value next to the exact one as the tanhf form rounded to bf16
    nearest = exact.float().bfloat16().double()
    old = got32[:, 0].bfloat16().double().cpu()[fin]
    assert int((g != nearest).sum()) <= int((old != nearest).sum())
    assert ec.echo_get_device_error() == 0
