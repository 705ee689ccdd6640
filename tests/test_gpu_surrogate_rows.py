"""Loss gradients of batches of other sizes than a training batch: the weight
gradients' products have one K chunk (16 rows), a ragged last one (48, 80,
1008) or more chunks than the pipeline has stages (1008, 1024), and the output
layer's kernel a last block of fewer rows.  The bound per entry is that of the
256-row test: BF16 roundings times the chain rule in absolute values."""
import numpy as np
import pytest

from oracle import mlp
from paper_2408_00559_gb300 import _lib as B
from paper_2408_00559_gb300 import build as BLD
from test_gpu_surrogate import BF16_U, GRAD_K, from_vector, to_vector

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    BLD.build()
    B.lib()


@pytest.mark.parametrize("rows", [16, 48, 80, 1008, 1024])
def test_gradients_of_any_batch_size(rows):
    s = B.Surrogate(members=1, seed=1)
    v = to_vector(mlp.init_params(width=256, n_in=8, seed=15))
    s.params(0, v)
    rng = np.random.default_rng(rows)
    x = rng.uniform(-1, 1, size=(rows, 8))
    t = rng.standard_normal(rows)
    g_gpu, loss_gpu = s.grad(0, x, t)
    s.close()
    p32 = from_vector(v)
    p32["b4"] = float(p32["b4"][0])
    L, g = mlp.loss_and_grads(p32, x, t)
    assert abs(loss_gpu - L) <= 1e-2 * L
    scale = mlp.grad_abs_scale(p32, x, t)
    gg = from_vector(g_gpu)
    for name in ("W1", "b1", "W2", "b2", "W3", "b3", "w4", "b4"):
        ratio = np.abs(np.ravel(gg[name]) - np.ravel(g[name])) / (BF16_U * np.ravel(scale[name]) + 1e-300)
        assert np.all(ratio <= GRAD_K), (name, int(ratio.argmax()), float(ratio.max()))
