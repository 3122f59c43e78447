"""Renders behind another library's kernel that lets its successor start early
(programmatic launch): parameters that it writes late are the ones rendered, and
a buffer that it still reads is not overwritten with the drawn parameters."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def env(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b
    b.build()
    so = str(tmp_path_factory.mktemp("early") / "early_release.so")
    subprocess.run([b.NVCC, *b.ARCH, "-O2", "-shared", "-Xcompiler", "-fPIC", "-o", so,
                    os.path.join(HERE, "early_release_harness.cu")], check=True)
    launch = ctypes.CDLL(so).late_copy_launch
    launch.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]

    def late_copy(src, dst):
        assert launch(src.data_ptr(), dst.data_ptr(), dst.numel(), 200,
                      torch.cuda.current_stream().cuda_stream) == 0

    return torch, pkg, late_copy


# 44.1 kHz (R = 100) and 16 kHz (general R); tiles shared by 8 CTAs, tiles of one CTA all
# resident at once, more tiles than places
@pytest.mark.parametrize("rate", [44100, 16000])
@pytest.mark.parametrize("batch", [1, 16, 300, 700])
def test_parameters_written_late(env, rate, batch):
    torch, pkg, late_copy = env
    syn = pkg.Synth(seconds=1.0, sample_rate=float(rate), max_batch=700)
    g = torch.Generator(device="cuda").manual_seed(batch)
    want_u, old_u = (torch.rand(batch, 78, device="cuda", generator=g) for _ in range(2))
    want = syn.render(3, 1, batch, params_in=want_u)[0].clone()
    want_n = syn.render_normalized(3, 1, batch, params_in=want_u)[0].clone()
    syn.sync()
    torch.cuda.synchronize()
    u = old_u.clone()
    out = torch.empty_like(want)
    for call, ref in ((syn.render, want), (syn.render_normalized, want_n)):
        u.copy_(old_u)
        syn.render(9, 0, batch)  # a recorded launch, which the next one may overlap
        late_copy(want_u, u)
        call(3, 1, batch, params_in=u, out=out)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    syn.sync()
    syn.close()


@pytest.mark.parametrize("batch", [1, 16, 300])
def test_drawn_parameters_do_not_overtake_a_reader(env, batch):
    torch, pkg, late_copy = env
    syn = pkg.Synth(seconds=1.0, max_batch=300)
    before = torch.rand(batch, 78, device="cuda")
    drawn = syn.render(5, 2, batch)[1].clone()
    p, seen = before.clone(), torch.zeros_like(before)
    torch.cuda.synchronize()
    syn.render(9, 0, batch)
    late_copy(p, seen)
    syn.render(5, 2, batch, params_out=p)
    torch.cuda.synchronize()
    assert torch.equal(seen, before) and torch.equal(p, drawn)
    syn.sync()
    syn.close()
