"""Products of few 128 x 64 tiles and a short K, whose K-slices are added inside a cluster, at the edges of the slicing
(k-blocks of 64 per slice, ragged last slices), the tiles and the vector stores, against an FP32 product."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 16, 127, 128, 129])
@pytest.mark.parametrize("n,k", [(64, 8), (65, 192), (78, 1024), (1024, 80), (1024, 1024), (1021, 968), (300, 4096),
                                 (300, 4104), (62, 1096)])
def test_small_product(m, n, k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b_
    b_.build()
    syn = pkg.Synth(seconds=0.01, max_batch=1)
    g = torch.Generator(device="cuda").manual_seed(m + 7 * n + k)
    a = torch.randn(m, k, device="cuda", generator=g).to(torch.bfloat16)
    b = torch.randn(n, k, device="cuda", generator=g).to(torch.bfloat16)
    outs = []
    for ldc in (n, n + 3):
        c = torch.full((m, ldc), float("nan"), device="cuda")
        assert pkg.lib().synth_gemm_bf16(syn.handle, a.data_ptr(), k, b.data_ptr(), k, c.data_ptr(), ldc, m, n, k, 0.5,
                                         torch.cuda.current_stream().cuda_stream) == 0
        assert torch.isnan(c[:, n:]).all()
        outs.append(c[:, :n])
    syn.sync()
    # each side adds k exact products with at most k roundings of 2^-23 of the sum of their absolute values, and halves
    # exactly: at most k 2^-22 / 2 of it apart
    ref = 0.5 * (a.double() @ b.double().T)
    bar = (a.double().abs() @ b.double().abs().T) * (k * 2.0 ** -23) + 1e-6
    for c in outs:
        assert ((c.double() - ref).abs() <= bar).all()
    assert torch.equal(outs[0], outs[1])
    syn.close()


@pytest.mark.parametrize("m,n,k", [(5, 62, 8200), (129, 301, 4168), (9, 1024, 44160), (128, 258, 4104)])
def test_split_product(m, n, k):
    """Longer K: slices by CTA, added by the reduction kernel (rows of 8, columns of 32 or a ragged end of them)."""
    import ctypes
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b_
    b_.build()
    syn = pkg.Synth(seconds=0.01, max_batch=1)
    g = torch.Generator(device="cuda").manual_seed(m + 7 * n + k)
    a = torch.randn(m, k, device="cuda", generator=g).to(torch.bfloat16)
    b = torch.randn(n, k, device="cuda", generator=g).to(torch.bfloat16)
    nb = ctypes.c_size_t()
    assert pkg.lib().synth_gemm_bf16_workspace_size(syn.handle, m, n, ctypes.byref(nb)) == 0
    ws = torch.empty(nb.value // 4 + 1, device="cuda")
    c = torch.full((m, n + 1), float("nan"), device="cuda")
    assert pkg.lib().synth_gemm_bf16_splitk(syn.handle, a.data_ptr(), k, b.data_ptr(), k, c.data_ptr(), n + 1, m, n, k,
                                            1.0, ws.data_ptr(), nb.value,
                                            torch.cuda.current_stream().cuda_stream) == 0
    syn.sync()
    assert torch.isnan(c[:, n]).all()
    ref = a.double() @ b.double().T
    bar = (a.double().abs() @ b.double().abs().T) * (k * 2.0 ** -22) + 1e-6
    assert ((c[:, :n].double() - ref).abs() <= bar).all()
    syn.close()
