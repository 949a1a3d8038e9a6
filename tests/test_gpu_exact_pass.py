"""The exact pass where its form changes with the layout's size: the small
pass (up to 4,096 points; chunks of 64 and 128 points) and the symmetric
one with and without cut tile pairs.  Gradient and Z against the FP64 oracle
at the tolerances of the parity tests; FP32 partials of at most 512 forces and
64 kernel values round within 3.1e-5 and 4.6e-6 of their absolute sums."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2310_11186_gb300 as pkg  # noqa: E402


def _ring(n):
    """A cycle of n >= 3 nodes with equal P, and a spread layout (with two nodes the gradient is 0)."""
    i = np.arange(n)
    col = np.sort(np.stack([(i - 1) % n, (i + 1) % n], 1), 1).reshape(-1).astype(np.int32)
    rp = np.arange(0, 2 * n + 1, 2, dtype=np.int64)
    P = np.full(col.size, 1.0 / col.size, np.float32)
    Y = (10.0 * np.random.default_rng(n).standard_normal((n, 2))).astype(np.float32)
    return rp, col, P, Y


@pytest.mark.parametrize("n", [3, 63, 64, 65, 255, 256, 257, 3072, 3073, 4095, 4096, 4097, 7169, 10007, 20011, 45056, 45057])
def test_gradient_and_Z_against_the_oracle(n):
    rp, col, P, Y = _ring(n)
    oG, oZ = oracle.gradient(n, rp, col, P.astype(np.float64), Y.astype(np.float64), 1.0)
    with pkg.Layout() as lay:
        lay.set_P(rp, col, P)
        lay.init_Y(Y)
        G, Z = lay.gradient(1.0)
        kl = lay.kl()  # a pass whose forces nobody takes
        G2, Z2 = lay.gradient(1.0)
        kl2 = lay.kl()
    assert abs(Z - oZ) <= 1e-5 * oZ
    assert np.linalg.norm(G - oG) <= 1e-4 * np.linalg.norm(oG)
    assert np.array_equal(G, G2) and Z == Z2 and kl == kl2  # every pass starts from cleared sums


@pytest.mark.parametrize("n", [1000, 9000])
def test_a_nan_in_the_layout_reaches_Z(n):
    rp, col, P, Y = _ring(n)
    Y[n // 2, 0] = np.nan
    with pkg.Layout() as lay:
        lay.set_P(rp, col, P)
        lay.init_Y(Y)
        G, Z = lay.gradient(1.0)
        assert np.isnan(Z) and np.isnan(G).all()
        with pytest.raises(pkg.TsgneError):
            lay.kl()
        lay.init_Y(np.zeros((n, 2), np.float32) + np.arange(n, dtype=np.float32)[:, None])
        assert np.isfinite(lay.gradient(1.0)[1])  # a new layout starts clean
