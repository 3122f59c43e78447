"""Renders of few voices, whose tiles several CTAs share and whose launches
overlap in a row, against the same voices rendered as part of a launch too large
for either: bit for bit (a voice depends on its seed and index alone)."""
import numpy as np
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


# one interval, one window less than full, two windows and a bit, ragged lengths;
# integer, divisible-by-2-only and fractional samples per interval
@pytest.mark.parametrize("samples,rate", [(100, 44100), (25499, 44100), (51003, 44100), (176400, 44100),
                                          (22050 * 2 + 7, 22050), (64000, 16000), (100001, 48000)])
def test_few_voices_match_the_full_launch(env, samples, rate):
    torch, pkg = env
    total = 768  # more tiles than CTAs even with one window each
    syn = pkg.Synth(seconds=samples / rate, sample_rate=float(rate), max_batch=total)
    full, params = syn.render(11, 0, total)
    for batch in (1, 2, 3, 8, 24, 96):
        a, p = syn.render(11, 5, batch)
        g = slice(5 * batch, 6 * batch)
        assert torch.equal(a, full[g]) and torch.equal(p, params[g]), batch
        u = params[g].contiguous()
        assert torch.equal(syn.render(11, 5, batch, params_in=u)[0], full[g]), batch
    syn.sync()
    syn.close()


def test_launches_in_a_row(env):
    """Launches of changing sizes with no wait between them, into buffers of
    their own and into one buffer, and replayed from a graph."""
    torch, pkg = env
    syn = pkg.Synth(seconds=1.0, max_batch=96)
    sizes = [1, 1, 3, 96, 1, 16, 64, 2, 1, 30] * 3
    want = [syn.render(7, i, b)[0].clone() for i, b in enumerate(sizes)]
    syn.sync()
    outs = [torch.empty_like(w) for w in want]

    def burst():
        for i, b in enumerate(sizes):
            syn.render(7, i, b, out=outs[i])

    burst()
    syn.sync()
    assert all(torch.equal(o, w) for o, w in zip(outs, want))
    one = torch.empty(96, 44100, device="cuda")
    for i, b in enumerate(sizes):
        syn.render(7, i, b, out=one[:b])
    syn.sync()
    assert torch.equal(one[:sizes[-1]], want[-1])
    for o in outs:
        o.zero_()
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    params = [torch.empty(b, 78, device="cuda") for b in sizes]
    with torch.cuda.graph(graph, stream=st):
        for i, b in enumerate(sizes):
            syn.render(7, i, b, out=outs[i], params_out=params[i])
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    syn.sync()
    assert all(torch.equal(o, w) for o, w in zip(outs, want))
    syn.close()
