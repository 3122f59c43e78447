"""The l1 distances' error against 64 bits, for pairs from unrelated to nearly
equal and rows from 8 values on, beside that of |a - b| added up in order in
FP32, which the distances must not exceed whatever form computes them.

Bar, for the root mean square of the relative error over 128 pairs: 1.25 times
the ordered sum's, plus 2^-25 for the rounding of the result. The mean of 256
squares (128 here, 128 there) is uncertain by 9%, so that equal errors pass."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PAIRS = 128


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


# spread: N / d is about 2.5 times this; around the line at dim / 128 it changes from the
# maxima to the terms
@pytest.mark.parametrize("kind", ["normal", "heavy"])
@pytest.mark.parametrize("dim", [8, 64, 512, 1023, 1024, 2816, 11264, 44160])
def test_no_less_precise_than_a_sum_in_order(env, kind, dim):
    torch, pkg, syn = env
    line = min(256.0, dim / 128)
    for closeness in (1, 4, 16, 64, 230, 0.85 * line, 1.2 * line):
        g = torch.Generator(device="cuda").manual_seed(dim + int(closeness))
        a = torch.randn(PAIRS, dim, device="cuda", generator=g)
        if kind == "heavy":
            a *= torch.exp(2 * torch.randn(PAIRS, dim, device="cuda", generator=g))
        noise = torch.randn(PAIRS, dim, device="cuda", generator=g)
        b = a + noise * a.abs().mean(1, keepdim=True) * (2.5 / max(closeness, 0.5))
        emb = torch.zeros(2 * PAIRS, (dim + 7) // 8 * 8, device="cuda", dtype=torch.bfloat16)[:, :dim]
        emb[0::2], emb[1::2] = a.bfloat16(), b.bfloat16()
        d = pkg.l1_distances(syn, emb).double().cpu().numpy()
        syn.sync()
        e = emb.float().cpu().numpy()
        terms = np.abs(e[0::2] - e[1::2])  # exact differences rounded to FP32, as the kernels form them
        exact = np.abs(e[0::2].astype(np.float64) - e[1::2]).sum(1)
        in_order = np.cumsum(terms, axis=1, dtype=np.float32)[:, -1].astype(np.float64)
        i = np.arange(0, 2 * PAIRS, 2)
        got = d[i, i + 1]

        def rms(x):
            return float(np.sqrt(np.mean(((x - exact) / exact) ** 2)))

        assert rms(got) <= 1.25 * rms(in_order) + 2.0 ** -25, (closeness, rms(got), rms(in_order))
