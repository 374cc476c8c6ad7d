"""Bias gradients of the learned model (column sums over the rows) at the edges of their split:
fewer rows than one row phase, one row past a slice, more columns than one block holds and fewer
than one warp reads. Against the FP64 oracle's gradient, 1e-4 of each layer's largest bias
gradient (the tolerance of the model's other gradients)."""
import numpy as np
import pytest

from oracle import learned as olearned
from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,n_b,n_f,width", [(1, 2, 5, 8), (3, 5, 7, 24), (257, 12, 9, 136), (1025, 6, 33, 20)])
def test_bias_gradients_match_oracle(rows, n_b, n_f, width):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    rng = np.random.default_rng(rows)
    X = rng.normal(size=(rows, n_b + n_f)).astype(np.float32)
    T = rng.normal(size=(rows, n_b)).astype(np.float32)
    theta = sy.mlp_init(n_f, width, n_b * n_b, 3)
    net = tddft.Mlp(n_b, n_f, width)
    net.set(theta)
    _, g = net.loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda())
    _, ref = olearned.loss_grad(theta.astype(np.float64), n_b, width, X.astype(np.float64), T.astype(np.float64))
    o = n_f * width
    for start, count in ((o, width), (o + width + width * width, width), (ref.size - n_b * n_b, n_b * n_b)):
        r = ref[start:start + count]
        assert np.max(np.abs(g[start:start + count] - r)) <= 1e-4 * np.max(np.abs(r))
