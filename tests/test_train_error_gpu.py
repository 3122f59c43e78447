"""A training step that is refused after its work has forked onto the model's own
stream: the fork is joined to the caller's stream before the error returns, so a
capture around the call ends, and the call leaves the model usable."""
import pytest

pytestmark = pytest.mark.gpu


def test_refused_step_joins_the_models_stream():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b
    b.build()
    syn = pkg.Synth(seconds=0.25, max_batch=16)
    model = pkg.ProposalModel(syn, max_batch=16, seed=4)
    dim = model.tensor(0, 0).shape[1]
    g = torch.Generator(device="cuda").manual_seed(1)
    raw = torch.randn(16 * dim + 8, device="cuda", generator=g).bfloat16()
    target = torch.rand(16, 78, device="cuda", generator=g)
    loss = torch.empty(1, device="cuda")
    weights = [model.tensor(0, layer).clone() for layer in range(4)]
    torch.cuda.synchronize()

    def step(offset):
        return pkg.lib().synth_model_train_features(
            model.handle, raw.data_ptr() + 2 * offset, target.data_ptr(), 16, 1e-3, loss.data_ptr(),
            torch.cuda.current_stream().cuda_stream)

    # the product refuses rows that start off a 16-byte boundary; the features' transpose
    # is on the model's stream by then
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        assert step(1) != 0
    graph.replay()
    torch.cuda.synchronize()
    assert step(1) != 0
    torch.cuda.synchronize()
    assert all(torch.equal(model.tensor(0, layer), w) for layer, w in enumerate(weights))
    assert step(0) == 0
    syn.sync()
    assert torch.isfinite(loss).all() and not torch.equal(model.tensor(0, 0), weights[0])
    model.close()
    syn.close()
