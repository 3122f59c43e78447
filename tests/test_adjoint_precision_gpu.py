"""The adjoint's error against the oracle's FP64 dual-number gradient, at its
2-norm over a batch, on voices whose pitch adjoints cancel.

Bar: 1.2 times 4.42e-6, the error of the same 32 voices with the control rate
in float-float, phase sums and pitch adjoints in FP64 and each rounded once
(the adjoint of one kernel per module). What remains is the audio rate's
FP32 phases. Mixer outputs summed in floats, or pitch adjoints rounded before
they are added, give 7.7e-6."""
import numpy as np
import pytest

import seeded_inputs as si

pytestmark = pytest.mark.gpu


def test_cancelling_pitch_adjoints(oracle_mod):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b
    b.build()
    seed, B, samples = 13, 32, 4410
    u = np.stack([oracle_mod.draw_params(seed, g) for g in range(B)])
    u = np.clip(u, 0.02, 0.98).astype(np.float32).astype(np.float64)
    w = si.upstream_grad(seed, (B, samples)).astype(np.float32).astype(np.float64)
    cfg = oracle_mod.default_config(seconds=0.1)
    ref = np.stack([oracle_mod.render_vjp(cfg, u[v], seed, v, w[v]) for v in range(B)])
    syn = pkg.Synth(seconds=0.1, max_batch=B)
    got = syn.backward(seed, 0, torch.tensor(u, dtype=torch.float32, device="cuda"),
                       torch.tensor(w, dtype=torch.float32, device="cuda"))
    syn.sync()
    err = np.linalg.norm(got.cpu().numpy().astype(np.float64) - ref) / np.linalg.norm(ref)
    assert err <= 1.2 * 4.42e-6, err
    syn.close()
