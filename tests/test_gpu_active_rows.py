"""Finding the active rows: up to D = 2048 each row is looked up in the index list
by its layer norm's warp, otherwise (and with K/V kept by the caller) a kernel of
its own makes the row map.  Both routes give the same bits, at list lengths around
the 32 probes of a look-up step and with the first and last rows in or out."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from synth import generate as G                    # noqa: E402

NT = 1100


def make(D, d, NT, F=64):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2608_02474_gb300 import echocache as ec
    g = torch.Generator(device="cuda").manual_seed(0)
    rn = lambda *s: (torch.randn(*s, generator=g, device="cuda") * 0.05)  # noqa: E731
    W = {"W" + p: rn(D, D) for p in ("q", "k", "v", "o", "qc", "kc", "vc", "oc")}
    W.update({"b" + p: rn(D) for p in ("q", "k", "v", "o", "qc", "kc", "vc", "oc")})
    W.update(W1=rn(F, D), b1=rn(F), W2=rn(D, F), b2=rn(D))
    blk = ec.DeviceBlock.from_host(W, rn(3, D))
    dims = ec.BlockDims(1, NT, D, D // d, d, F, 3)
    x = torch.randn(NT, D, generator=g, device="cuda").bfloat16()
    kv = torch.empty(NT, 2 * D, dtype=torch.bfloat16, device="cuda")
    q, s = (torch.from_numpy(a).cuda() for a in G.random_cache(NT, D, seed=1))
    ec.echo_block_step_kv(blk, dims, x, None, 0, kv, False, q.clone(), s.clone())
    return ec, blk, dims, x, kv, q, s


@pytest.fixture(scope="module")
def setup():
    return make(64, 64, NT)


@pytest.mark.parametrize("K", [1, 2, 31, 32, 33, 63, 64, 65, 1000, 1023, 1024, 1025, NT - 1, NT])
@pytest.mark.parametrize("ends", [True, False])
def test_routes_agree(setup, K, ends):
    routes_agree(setup, K, ends)


@pytest.mark.parametrize("D,d", [(320, 64), (1024, 128), (1088, 64), (2048, 128), (2112, 64)])
@pytest.mark.parametrize("K", [1, 33, 333, 1025, NT])
def test_routes_agree_at_width(D, d, K):
    """The other forms of the layer norm that looks the rows up (a lane holds 4 or 8
    chunks), at their first and last widths, and one width beyond them."""
    routes_agree(make(D, d, NT), K, True)


def routes_agree(setup, K, ends):
    ec, blk, dims, x, kv, q, s = setup
    rs = np.random.default_rng(K)
    rows = rs.choice(NT, K, replace=False)
    if ends and 2 <= K < NT:
        rows = np.union1d(rows[:K - 2], [0, NT - 1])
        extra = np.setdiff1d(np.arange(NT), rows)[:K - rows.size]
        rows = np.concatenate([rows, extra])
    idx = torch.from_numpy(np.sort(rows).astype(np.int32)).cuda()
    assert idx.numel() == K
    q1, s1, q2, s2 = q.clone(), s.clone(), q.clone(), s.clone()
    y1 = ec.echo_block_step(blk, dims, x, idx, K, q1, s1)
    y2 = ec.echo_block_step_kv(blk, dims, x, idx, K, kv.clone(), True, q2, s2)
    assert torch.equal(y1, y2) and torch.equal(q1, q2) and torch.equal(s1, s2)
    out = torch.ones(NT, dtype=torch.bool, device="cuda")
    out[idx.long()] = False
    assert torch.equal(q1[out], q[out]) and torch.equal(s1[out], s[out])
    assert torch.equal(y1[out], ec.echo_cache_dequant(q, s)[out])
    assert ec.echo_get_device_error() == 0


@pytest.mark.parametrize("D,d,NT,n_a,n_b,K", [
    (128, 64, 700, 1, 0, 1),            # 128-column tiles, one row each
    (320, 64, 700, 257, 130, 333),      # ragged rows and half column tiles on both sides
    (1024, 64, 5100, 4700, 299, 301),   # 256-column tiles
    (1088, 64, 5100, 5100, 5100, 1),    # every row twice; a quarter of a column tile
])
def test_projections_in_one_launch(D, d, NT, n_a, n_b, K):
    """K/V rows and Q' in one launch against each in a launch of its own: rows that are
    up to date are projected again, so K/V and every output stay as they are, bit for
    bit; other rows of a K/V buffer are not touched."""
    ec, blk, dims, x, kv, q, s = make(D, d, NT)
    rs = np.random.default_rng(D + K)
    pick = lambda n: torch.from_numpy(np.sort(rs.choice(NT, n, replace=False)).astype(np.int32)).cuda()  # noqa: E731,E501
    idx, rows_a, rows_b = pick(K), pick(n_a), pick(n_b)
    q1, s1, q2, s2 = q.clone(), s.clone(), q.clone(), s.clone()
    y1 = ec.echo_block_step_kv(blk, dims, x, idx, K, kv.clone(), True, q1, s1)       # Q' alone
    kv2 = torch.full_like(kv, 3.0)
    listed = torch.zeros(NT, dtype=torch.bool, device="cuda")
    listed[rows_a.long()] = listed[rows_b.long()] = True
    ec.echo_block_step_kv(blk, dims, x, idx, K, kv2, True, q.clone(), s.clone(), rows_a, n_a, rows_b,
                          n_b)
    assert torch.equal(kv2[listed], kv[listed]) and bool((kv2[~listed] == 3).all())
    kv3 = kv.clone()
    y3 = ec.echo_block_step_kv(blk, dims, x, idx, K, kv3, True, q2, s2, rows_a, n_a, rows_b, n_b)
    assert torch.equal(kv3, kv)
    assert torch.equal(y1, y3) and torch.equal(q1, q2) and torch.equal(s1, s2)
    assert ec.echo_get_device_error() == 0
