"""Renders at ratios R = SR / CR at the edges of the form that takes intervals
of any length: the shortest intervals (R just above 4 and R = 5, 6, 7: every quad
but one or two of an interval straddles a boundary, and most voices meet the
Nyquist cap), one quad more or less than a run, a denominator past 23 bits, and
tiles that end within an interval. Against the FP64 oracle, with the bar of the
other rates (audio max-abs error 2e-4; it follows from the phase error, which
does not depend on R), plain and normalised, few voices and many."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as p
    from paper_2104_12922_gb300 import build as b
    b.build()
    return p


@pytest.mark.parametrize("sr,cr,n", [
    (1768.0, 441.0, 1769), (2205.0, 441.0, 2207), (2646.0, 441.0, 2646), (3087.0, 441.0, 1785),
    (7497.0, 441.0, 7497),         # R = 17
    (7938.0, 441.0, 4591),         # R = 18, a tile and a sample
    (40000003.0, 8388619.0, 2100),
])
def test_interval_lengths(pkg, oracle_mod, sr, cr, n):
    import torch
    syn = pkg.Synth(seconds=n / sr, max_batch=400, sample_rate=sr, control_rate=cr)
    assert syn.num_samples == n
    many, params = syn.render(3, 0, 400)
    few, _ = syn.render(3, 3, 5)
    assert torch.equal(few, many[15:20])
    a, _, peak, _ = syn.render_normalized(3, 0, 400, threshold=1e-3)
    assert torch.equal(peak, many.abs().amax(1))
    g = torch.where(peak >= 1e-3, 1.0 / peak, torch.ones_like(peak))
    assert torch.equal(a, many * g[:, None])
    syn.sync()
    cfg = oracle_mod.default_config(seconds=n / sr, sample_rate=sr, control_rate=cr)
    ref_a, ref_p = oracle_mod.render_batch(cfg, 3, 0, 12)
    assert np.array_equal(params[:12].cpu().numpy(), ref_p)
    got = many[:12].cpu().numpy()
    assert np.all(np.isfinite(got))
    err = float(np.max(np.abs(got - ref_a)))
    assert err <= 2e-4, f"max-abs error {err:.3e} at SR {sr}, CR {cr}"
    syn.close()
