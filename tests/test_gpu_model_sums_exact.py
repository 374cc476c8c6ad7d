"""Bias gradients (column sums over the rows) hold what a float64 sum holds: columns whose partial sums are
exact in float64 come out exact, also where they cancel over 50 bits or pass float32's largest number on
the way, and a NaN or infinity stays in its column.

With all weights zero the model's map is zero and the last bias gradient is the column sum of
-scale T_r,i X_r,j, scale = 2 / (rows n_b), a power of two here like T's and X's entries."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_column_sums_are_those_of_float64():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    rows, n_b, n_f, width = 64, 4, 3, 8
    T = np.zeros((rows, n_b), dtype=np.float32)
    X = np.zeros((rows, n_b + n_f), dtype=np.float32)
    X[:, :n_b] = 256.0
    T[0:20:4, 0] = [2.0 ** 50, 2.0 ** 25, 1.0, -2.0 ** 50, -2.0 ** 25]     # rows of one thread
    T[0:12:4, 1] = [2.0 ** 126, 2.0 ** 126, -2.0 ** 126]                   # summands of 2^127
    T[5, 2] = np.inf
    T[6, 3] = np.nan
    net = tddft.Mlp(n_b, n_f, width)
    net.set(np.zeros(net.size, dtype=np.float32))
    _, g = net.loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda())
    b3 = g[-n_b * n_b:].reshape(n_b, n_b)
    scale = -2.0 / (rows * n_b) * 256.0
    assert np.array_equal(b3[0], np.full(n_b, np.float32(scale)))
    assert np.array_equal(b3[1], np.full(n_b, np.float32(scale * 2.0 ** 126)))
    assert np.array_equal(b3[2], np.full(n_b, -np.inf, dtype=np.float32))
    assert np.all(np.isnan(b3[3]))
