"""The network's outputs and gradients at batches between those of the full-size
test, element by element within the same bars: 136 and 1152 (two and nine row
tiles, ReLU gradients and transposed copies through the one-wave products and the
split-K reduction) and 1160 (ten, where the output layer's input gradient has too
many tiles for them and is gated in the general product's epilogue)."""
import pytest

import test_fullsize_gpu as full

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_12922_gb300 as pkg
    from paper_2104_12922_gb300 import build as b
    b.build()
    return torch, pkg


@pytest.mark.parametrize("batch", [136, 1152, 1160])
def test_gradients_elementwise(env, batch):
    full.test_mlp_elementwise(env, 0.05, batch)
