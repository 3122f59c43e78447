"""The adjoint at the edges of its chunks and lanes -- control points in chunks
of 512, intervals in groups of 16, eight lanes of 16 samples an interval -- with
ragged voice lengths and the smallest and largest samples per interval it takes,
against the oracle's FP64 dual-number gradient. The bar is that of the other
adjoint tests, 2e-3 of the voice's largest component: FP32 audio-rate values
rebuilt per sample."""
import numpy as np
import pytest

import seeded_inputs as si

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(oracle_mod):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b
    b.build()
    return torch, pkg, oracle_mod


def _grad(torch, syn, u, w, seed, batch_index):
    g = syn.backward(seed, batch_index, torch.tensor(u, dtype=torch.float32, device="cuda"),
                     torch.tensor(w, dtype=torch.float32, device="cuda"))
    syn.sync()
    return g.cpu().numpy().astype(np.float64)


# 1 interval; 511 and 512 intervals (one chunk and one more point); three chunks, ragged;
# R = 4 (one lane, one quad), 16, 36 (three lanes), 128 (all lanes full)
@pytest.mark.parametrize("sr,cr,samples", [(44100, 441, 57), (44100, 441, 51100), (44100, 441, 51101),
                                           (44100, 441, 104803), (44100, 11025, 6002), (8000, 500, 9003),
                                           (15876, 441, 18001), (48000, 375, 70001)])
def test_chunks_and_lanes_match_oracle(env, sr, cr, samples):
    torch, pkg, oracle = env
    B, seed = 2, 13
    syn = pkg.Synth(seconds=samples / sr, sample_rate=float(sr), control_rate=float(cr), max_batch=B)
    assert syn.num_samples == samples
    u = np.stack([oracle.draw_params(seed, g) for g in range(B)])
    u = np.clip(u, 0.02, 0.98).astype(np.float32).astype(np.float64)
    w = si.upstream_grad(seed, (B, samples))
    got = _grad(torch, syn, u, w, seed, 0)
    cfg = oracle.default_config(seconds=samples / sr)
    cfg.sample_rate, cfg.control_rate = float(sr), float(cr)
    for v in range(B):
        ref = oracle.render_vjp(cfg, u[v], seed, v, w[v])
        assert np.max(np.abs(got[v] - ref)) <= 2e-3 * np.max(np.abs(ref)) + 1e-6, v
    syn.close()


def test_unaligned_upstream_gradient_and_edge_parameters(env):
    """An upstream gradient that starts 4 bytes into its buffer (scalar loads)
    gives the bits of an aligned one; the parameter cube's corners give finite
    gradients."""
    torch, pkg, _ = env
    B = 7
    syn = pkg.Synth(seconds=0.5, max_batch=B)
    u = torch.tensor(np.concatenate([si.edge_params(5), si.uniform_params(3, 2)]), dtype=torch.float32,
                     device="cuda")
    w = torch.randn(B, syn.num_samples, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    shifted = torch.empty(w.numel() + 1, device="cuda")[1:].view_as(w).copy_(w)
    a, b = syn.backward(5, 2, u, w), syn.backward(5, 2, u, shifted)
    syn.sync()
    assert torch.equal(a, b) and bool(torch.isfinite(a).all())
    syn.close()
