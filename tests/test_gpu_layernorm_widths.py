"""Layer norm at the widths where the form of the kernel changes (a lane holds 1, 4
or 8 chunks; the last width with a row per warp and the first beyond it), at row
counts around a block's, against the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

import oracle                                      # noqa: E402
from synth import generate as G                    # noqa: E402


@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("n,D", [(1, 8), (9, 256), (8, 264), (1025, 1024), (7, 1032), (1030, 1032),
                                 (1023, 2040), (1030, 2048), (17, 2056)])
def test_layernorm_widths(n, D, bf16):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2608_02474_gb300 import echocache as ec
    x = G.random_rows(n, D, seed=n + D, scale=2.0) + np.float32(0.5)
    if bf16:
        x = G.to_bf16_values(x)
    t = torch.from_numpy(x).to("cuda", torch.bfloat16 if bf16 else torch.float32)
    out = ec.echo_layernorm(t).float().cpu().numpy()
    ref = oracle.block.layer_norm(x)
    # fp32 sums (2^-24 sqrt(D) of the row), the result in bf16: 2^-9 of the value
    assert np.all(np.abs(out - ref) <= 2 ** -8 * np.abs(ref) + 1e-4)
    rows = torch.arange(n, dtype=torch.int32, device="cuda")
    if bf16:
        assert torch.equal(ec.echo_layernorm(t, rows), ec.echo_layernorm(t))
    assert ec.echo_get_device_error() == 0


@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("D", [256, 1024, 1032, 1536, 2048, 2056, 5120])
def test_layernorm_of_a_row_whatever_comes_with_it(D, bf16):
    """A row has the same bits alone, in a small batch and in a large one: from 1025 to
    2048 fp32 values the kernel changes with the row count."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2608_02474_gb300 import echocache as ec
    g = torch.Generator(device="cuda").manual_seed(D)
    x = torch.randn(3000, D, generator=g, device="cuda") * 2 + 0.5
    x = x.bfloat16() if bf16 else x
    out = ec.echo_layernorm(x)
    for n in (1, 64, 1023, 1024, 1025):
        assert torch.equal(ec.echo_layernorm(x[:n].contiguous()), out[:n])
    assert ec.echo_get_device_error() == 0
