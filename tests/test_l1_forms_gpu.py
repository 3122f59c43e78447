"""The l1 distance kernel at the edges of its tiles and chunks, its split of a
tile over a cluster, and the pairs it computes term by term (close pairs, rows
with infinities or NaN, tiles of duplicates), against sums in FP64.

Bars. Term by term, dim FP32 additions: 7 2^-24 sqrt(dim) d. Through the
maxima, with N the rows' sums of |e|: a product over 16 values keeps 24 bits
of its partial sum, so the four of a 64-value chunk lose at most 8 2^-24 of
max(N_i, N_j) in the maxima and of N_i and N_j in the row sums; halving,
adding and subtracting the row sums round twice; doubled, that is at most
28 2^-24 (N_i + N_j). The running sum of the chunks' halves adds the first
bar again."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b
    b.build()
    syn = pkg.Synth(seconds=0.01, max_batch=1)
    yield torch, pkg, syn
    syn.close()


def _check(torch, pkg, syn, emb):
    m, dim = emb.shape
    d = pkg.l1_distances(syn, emb).cpu().numpy().astype(np.float64)
    syn.sync()
    e = emb.double().cpu().numpy()
    ref = np.abs(e[:, None, :] - e[None, :, :]).sum(2) if m * m * dim < 3e7 else \
        np.stack([np.abs(e - r).sum(1) for r in e])
    n = np.abs(e).sum(1)
    nn = n[:, None] + n[None, :]
    bar = 7 * U * np.sqrt(dim) * ref + np.where(256 * ref < 0.9 * nn, 0.0, 28 * U * nn)
    assert np.array_equal(d, d.T) and np.all(np.diag(d) == 0)
    assert np.all(np.abs(d - ref) <= bar), float(np.max(np.abs(d - ref) / np.maximum(bar, 1e-300)))


@pytest.mark.parametrize("m,dim", [(1, 1), (2, 8), (63, 127), (64, 128), (65, 129), (129, 1000),
                                   (70, 2056), (200, 4480), (3, 44160), (1100, 640)])
def test_edges_of_tiles_and_chunks(env, m, dim):
    torch, pkg, syn = env
    g = torch.Generator(device="cuda").manual_seed(m * 1000 + dim)
    ld = (dim + 7) // 8 * 8 + 8
    emb = torch.zeros(m, ld, device="cuda", dtype=torch.bfloat16)
    emb[:, :dim] = torch.randn(m, dim, device="cuda", generator=g).bfloat16()
    emb[:, dim:] = 1e30  # past a row's end: not read
    _check(torch, pkg, syn, emb[:, :dim])


@pytest.mark.parametrize("m", [60, 1000])
@pytest.mark.parametrize("spread", [0.0, 2e-3])
def test_close_pairs(env, m, spread):
    """Rows near one another: a few among others, and all of them (whole tiles
    term by term)."""
    torch, pkg, syn = env
    g = torch.Generator(device="cuda").manual_seed(5)
    dim = 4480
    base = torch.randn(1, dim, device="cuda", generator=g)
    near = (base + spread * torch.randn(m, dim, device="cuda", generator=g)).bfloat16()
    _check(torch, pkg, syn, near)
    mixed = torch.randn(m, dim, device="cuda", generator=g).bfloat16()
    mixed[5::17] = near[5::17]
    _check(torch, pkg, syn, mixed)


def test_infinities_and_nan(env):
    torch, pkg, syn = env
    g = torch.Generator(device="cuda").manual_seed(6)
    emb = torch.zeros(70, 304, device="cuda", dtype=torch.bfloat16)[:, :300]  # rows 16-byte aligned
    emb[:] = torch.randn(70, 300, device="cuda", generator=g).bfloat16()
    emb[3, 7], emb[4, 7], emb[9, 299], emb[66, 0] = float("inf"), float("-inf"), float("nan"), 3e38
    d = pkg.l1_distances(syn, emb).cpu()
    syn.sync()
    e = emb.float().cpu()
    ref = (e[:, None, :] - e[None, :, :]).abs().sum(2)
    assert torch.equal(torch.isnan(d), torch.isnan(ref)) and torch.equal(torch.isinf(d), torch.isinf(ref))
    fine = torch.isfinite(ref)
    assert torch.allclose(d[fine], ref[fine], rtol=1e-5, atol=0)
