"""Cache writes and reads at the widths where a kernel holds more chunks of a row
per thread, or falls back to reading it twice, bit for bit against the oracle."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

import oracle                                      # noqa: E402
from oracle import refcache as R                   # noqa: E402
from synth import generate as G                    # noqa: E402

F32 = np.float32


@pytest.fixture(scope="module")
def ec():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2608_02474_gb300 import echocache
    return echocache


def dev(a, dt=None):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)


@pytest.mark.parametrize("n,D", [(1, 8), (9, 1016), (8, 1024), (17, 1032), (5, 2048), (7, 2056),
                                 (3, 5120), (4, 5128), (2, 8192)])
def test_quant_widths(ec, n, D):
    v = G.to_bf16_values(G.random_rows(n + 3, D, seed=D, scale=3.0))
    v[0] = 0.0
    v[n // 2, D // 2] = np.nan if n % 2 else np.inf
    v[n + 2] *= F32(2.0 ** 100)                    # exact: still bf16 values
    rows = np.random.default_rng(1).permutation(2 * n + 6)[:n + 3].astype(np.int32)
    q = torch.full((2 * n + 6, D), 9, dtype=torch.int8, device="cuda")
    s = torch.full((2 * n + 6,), -1.0, device="cuda")
    ec.echo_cache_quant(dev(v, torch.bfloat16), dev(rows), q, s)
    assert ec.echo_get_device_error() == 5          # the row that is not finite
    bad = n // 2                                    # header: q = 0, scale = amax (NaN or inf)
    gq, gs = q.cpu().numpy(), s.cpu().numpy()
    assert not gq[rows[bad]].any()
    assert np.isnan(gs[rows[bad]]) if n % 2 else np.isinf(gs[rows[bad]])
    oq, os_ = np.full((2 * n + 6, D), 9, np.int8), np.full(2 * n + 6, -1.0, F32)
    fine = np.arange(n + 3) != bad
    oracle.cache.quant_scatter(v[fine], rows[fine], oq, os_)
    keep = np.arange(2 * n + 6) != rows[bad]
    assert np.array_equal(gq[keep], oq[keep]) and np.array_equal(gs[keep], os_[keep])
    # reconstruction of every row, and of a gathered few, on the same widths
    if D % 16 == 0:
        got = ec.echo_cache_dequant(q, s).float().cpu().numpy()
        assert np.array_equal(got[keep], oracle.cache.dequant_gather(oq, os_)[keep])


@pytest.mark.parametrize("D", [16, 1024, 1040, 2064, 3504, 5120, 5136, 8192, 8208, 8928, 8944, 16592])
@pytest.mark.parametrize("R_cap", [40, 3])           # 3: runs without a slot, plain int8
def test_ref_cache_widths(ec, D, R_cap):
    ref_cache(ec, D, R_cap, 60, 20)


@pytest.mark.parametrize("NT,seg", [(152 * 14, 14), (153 * 14, 14), (152 * 27 - 5, 27), (500, 3)])
@pytest.mark.parametrize("D", [16, 320])
def test_ref_cache_segment_counts(ec, NT, seg, D):
    """Up to 152 segments the scan takes twelve rows at a time, above six: a whole
    window, one row more than two, a last segment cut short."""
    ref_cache(ec, D, NT // 2, NT, seg)


def ref_cache(ec, D, R_cap, NT, seg):
    g = ec.DeviceCache(ec.CACHE_REF, NT, D, R_cap=R_cap, seg_len=seg, tau=0.9)
    o = R.RefCache(NT, D, R_cap, seg, 0.9)
    rs = np.random.default_rng(D)
    for it in range(3):
        n = NT if it == 0 else int(rs.integers(1, NT + 1))
        rows = np.sort(rs.choice(NT, n, replace=False)).astype(np.int32)
        v = G.correlated_rows(n, D, seed=it + D, rho=0.95)
        g.write(dev(v, torch.bfloat16), dev(rows))
        o.write(rows, v)
        assert ec.echo_get_device_error() == 0
        assert np.array_equal(g.t["q"].cpu().numpy(), o.q)
        assert np.array_equal(g.t["scale"].cpu().numpy(), o.s)
        assert np.array_equal(g.t["ref"].cpu().numpy(), o.ref)
        assert np.array_equal(g.read().float().cpu().numpy(), o.reconstruct_bf16())


FIRST_WRITE = """
import sys, torch
from paper_2608_02474_gb300 import echocache as ec
c = ec.DeviceCache(ec.CACHE_REF, 24, 3504, seg_len=12)
rows = torch.arange(24, dtype=torch.int32, device="cuda")
for _ in range(2):
    c.write(torch.randn(24, 3504, device="cuda").bfloat16(), rows)
sys.exit(int(c.t["refcount"].sum()) != 24 or ec.echo_get_device_error())
"""


def test_ref_cache_first_write_of_a_process(ec):
    """3504 is the width whose staged rows fit the 48 KB that need no raised limit only
    without the scan's static buffers.  In a process of its own: a wider write before
    it would have raised the limit."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", FIRST_WRITE], cwd=root, check=True, timeout=300)


def test_ref_cache_too_wide_row_changes_nothing(ec):
    """A row that the scan cannot stage is refused before anything is enqueued."""
    D = 16608
    c = ec.DeviceCache(ec.CACHE_REF, 8, D, seg_len=4)
    c.load(ref=np.arange(8, dtype=np.int32), refcount=np.ones(8, np.int32))
    before = {n: t.clone() for n, t in c.t.items() if n != "pool"}
    with pytest.raises(ec.EchoError) as e:
        c.write(torch.zeros(8, D, dtype=torch.bfloat16, device="cuda"),
                torch.arange(8, dtype=torch.int32, device="cuda"))
    assert e.value.status == 2                      # ECHO_ERR_SHAPE
    torch.cuda.synchronize()
    for n, t in before.items():
        assert torch.equal(c.t[n], t), n
