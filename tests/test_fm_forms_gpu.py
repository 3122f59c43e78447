"""The FM voice's cuts of a voice into CTAs, which follow the batch and the length: a voice is the same bit for bit in every
batch it is rendered with, at both ends of the cuts' lengths and at a control rate dense enough for the fixed cut."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("samples,rate,control", [(1, 44100, 441.0), (4099, 44100, 441.0), (20481, 44100, 441.0),
                                                  (64000, 16000, 441.0), (88201, 48000, 441.0),
                                                  (30011, 16000, 4000.0)])
def test_cuts_agree(samples, rate, control):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b
    b.build()
    syn = pkg.Synth(seconds=samples / rate, sample_rate=float(rate), control_rate=control, max_batch=128)
    audio, drawn = syn.fm_render(11, 0, 128)
    syn.sync()
    assert torch.isfinite(audio).all() and audio.abs().max() <= 1 + 1e-5
    for voices in (1, 3, 16, 40):
        part, p = syn.fm_render(11, 0, voices)
        syn.sync()
        assert torch.equal(p, drawn[:voices]) and torch.equal(part, audio[:voices])
    syn.close()
