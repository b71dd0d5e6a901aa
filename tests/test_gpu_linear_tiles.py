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
    (5000, 128, 2112),       # 256-column tiles, several per pair, the last a quarter wide
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
