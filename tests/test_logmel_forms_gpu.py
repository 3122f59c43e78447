"""Log-mel features where work items take 16 frames (many voices) against the
same voices in calls where they take 8: bit for bit (a frame's features depend on
its own samples alone)."""
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


# 5, 8, 9, 16 and 17 frames, and 4 s with a ragged last item
@pytest.mark.parametrize("samples,batch", [(2100, 600), (4095, 600), (4096, 600), (8191, 600), (8192, 600),
                                           (176400, 128)])
def test_frames_per_item(env, samples, batch):
    torch, pkg = env
    syn = pkg.Synth(seconds=samples / 44100, max_batch=batch)
    assert syn.num_samples == samples
    model = pkg.ProposalModel(syn, max_batch=batch, seed=0)
    g = torch.Generator(device="cuda").manual_seed(samples)
    audio = torch.randn(batch, samples, generator=g, device="cuda") * 0.2
    whole = model.features(audio)
    for first, count in ((0, 1), (1, 3), (batch - 13, 13)):
        part = model.features(audio[first:first + count].contiguous())
        assert torch.equal(part, whole[first:first + count]), (first, count)
    syn.sync()
    model.close()
    syn.close()
