"""Normalised renders in a row, whose launches may overlap and whose scaling goes
to a part of the CTAs, against the same calls one at a time and against the plain
render scaled by its peak: bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b
    b.build()
    return torch, pkg


# one chunk and less, several, ragged and odd lengths; integer, even-only and
# fractional samples per control interval; batches below, at and above the CTAs
@pytest.mark.parametrize("samples,rate,batches", [(100, 44100, (1, 7, 640)), (8193, 44100, (1, 5, 400)),
                                                  (51003, 44100, (1, 12, 88, 203)),
                                                  (176400, 44100, (1, 2, 5, 43, 44, 87, 128)),
                                                  (44107, 22050, (1, 16, 300)),
                                                  (64000, 16000, (3, 30, 128)), (100001, 48000, (2, 64))])
def test_normalized_launches_in_a_row(env, samples, rate, batches):
    torch, pkg = env
    syn = pkg.Synth(seconds=samples / rate, sample_rate=float(rate), max_batch=max(batches))
    calls = [(b, i) for i in range(3) for b in batches]
    want = []
    for b, i in calls:
        a, p, peak, silent = (x.clone() for x in syn.render_normalized(5, i, b, threshold=1e-3))
        plain, params = syn.render(5, i, b)
        syn.sync()
        assert torch.equal(p, params) and torch.equal(peak, plain.abs().amax(1)), b
        g = torch.where(silent.bool(), torch.ones_like(peak), 1.0 / peak)
        assert torch.equal(silent.bool(), peak < 1e-3) and torch.equal(a, plain * g[:, None]), b
        want.append((a, p, peak, silent))
    got = [syn.render_normalized(5, i, b, threshold=1e-3) for b, i in calls]  # buffers of their own
    one = torch.empty(max(batches), samples, device="cuda")
    for b, i in calls:  # one buffer: each launch waits for the one before
        last = syn.render_normalized(5, i, b, threshold=1e-3, out=one[:b])
    syn.sync()
    for w, r in zip(want, got):
        assert all(torch.equal(x, y) for x, y in zip(w, r))
    assert all(torch.equal(x, y) for x, y in zip(want[-1], last))
    syn.close()
