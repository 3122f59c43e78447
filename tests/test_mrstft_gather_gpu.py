"""The gather of the MR-STFT gradient: four samples a thread against one (which a gradient buffer off the 16-byte grid
takes), bit for bit, at lengths around the segments' starts (4096 positions) and the reflected ends; the loss with and
without the gradient."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("samples,batch", [(2052, 3), (3076, 2), (4096, 5), (7168, 2), (8188, 1), (44100, 3),
                                           (135168, 2), (200000, 1)])
def test_gather_forms(samples, batch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b
    b.build()
    syn = pkg.Synth(seconds=samples / 44100, max_batch=8)
    g = torch.Generator(device="cuda").manual_seed(samples)
    x, y = (torch.randn(batch, samples, generator=g, device="cuda") for _ in range(2))
    mr = pkg.MRSTFT(syn, batch)
    loss, grad = mr(x, y)
    loss = loss.clone()
    odd = torch.full((batch * samples + 2,), float("nan"), device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    assert pkg.lib().synth_mrstft(syn.handle, x.data_ptr(), y.data_ptr(), batch, 1, mr.loss.data_ptr(),
                                  odd[1:].data_ptr(), mr.ws.data_ptr(), mr.ws.numel(), st) == 0
    syn.sync()
    assert torch.equal(odd[1:-1].view(batch, samples), grad) and torch.isfinite(grad).all()
    assert torch.isnan(odd[0]) and torch.isnan(odd[-1])
    assert torch.equal(mr.loss, loss)
    assert torch.equal(mr(x, y, grad=False)[0], loss)
    syn.close()
