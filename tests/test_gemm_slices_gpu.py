"""Products whose K is cut into slices, with small whole numbers: every sum is
exact in FP32, so the result equals the product in 64 bits whatever the order, and
a slice lost, counted twice or cut at the wrong place shows.

Up to 4096 values of K the slices are added inside a cluster (2, 4 and 8 of them,
the last one whole, short or a single k-block of 8 values), beyond by the
reduction kernel (37 slices in one go, 138 in four)."""
import ctypes

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
    syn = pkg.Synth(seconds=0.01, max_batch=1)
    yield torch, pkg, syn
    syn.close()


def _check(torch, pkg, syn, m, n, k):
    g = torch.Generator(device="cuda").manual_seed(m + 7 * n + k)
    a, b = (torch.randint(-8, 9, (r, k), device="cuda", generator=g).to(torch.bfloat16) for r in (m, n))
    want = (0.5 * (a.double() @ b.double().T)).float()  # at most 44160 * 64 / 2 < 2^24: exact
    nb = ctypes.c_size_t()
    assert pkg.lib().synth_gemm_bf16_workspace_size(syn.handle, m, n, ctypes.byref(nb)) == 0
    ws = torch.full((nb.value // 4 + 1,), float("nan"), device="cuda")
    for ldc in (n, n + 3):
        c = torch.full((m, ldc), float("nan"), device="cuda")
        assert pkg.lib().synth_gemm_bf16_splitk(
            syn.handle, a.data_ptr(), k, b.data_ptr(), k, c.data_ptr(), ldc, m, n, k, 0.5, ws.data_ptr(),
            nb.value, torch.cuda.current_stream().cuda_stream) == 0
        syn.sync()
        assert torch.equal(c[:, :n], want) and torch.isnan(c[:, n:]).all()


# k-blocks of 64: 7 (4 + 3), 8 (the last of 8 values), 13 and 15 (4 slices, the last of 1
# and 3), 16, 29 and 32 (8 slices)
@pytest.mark.parametrize("k", [424, 456, 776, 936, 968, 1800, 1992])
@pytest.mark.parametrize("m", [1, 16, 127, 129])
@pytest.mark.parametrize("n", [62, 78, 300, 1021])
def test_slices_inside_a_cluster(env, m, n, k):
    _check(*env, m, n, k)


@pytest.mark.parametrize("m,n,k", [(9, 62, 44160), (9, 1024, 44160), (128, 300, 44160), (129, 301, 4168),
                                   (17, 78, 10504)])
def test_slices_added_by_the_reduction(env, m, n, k):
    _check(*env, m, n, k)
