"""The tree's sort at the sizes where its CTAs and launches change: a tile of
2,048 keys and its ends; the last tile counts with 16 warps a CTA and with 8 (152
SMs: 311,296 points); the ranges where a pass starts beside the one before (up to
101 tiles, from 456).  Equal keys in runs longer than a tile check that passes are
stable.  The sums are compared with the oracle's restatement of the tree code,
which sorts by (key, index): tolerances as for FP32 sums of a few thousand
terms, 1e-4 (relative L2 of the gradient) and 1e-5 (Z).  Launched one by one and
in a captured pair of iterations the bits are the same."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2310_11186_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("n", [31, 2047, 2048, 2049, 206848, 206849, 311296, 311297, 931841])
def test_sorted_tree(n):
    rng = np.random.default_rng(n)
    Y = (rng.standard_normal((n, 2)) * 5.0 + 1.0).astype(np.float32)
    Y[n // 2:n // 2 + n // 4] = Y[0]
    rp, col, P = np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32)
    want, wZ = oracle.gradient_tree(n, rp, col, P, Y, 1.0, theta=1.0)
    with pkg.Layout(repulsion=1, theta=1.0) as lay:
        lay.set_P(rp, col, P)
        lay.init_Y(Y)
        got, Z = lay.gradient(1.0)
        lay.run(4)
        ran = lay.get_Y()
        lay.init_Y(Y)
        for _ in range(4):
            lay.step()
        stepped = lay.get_Y()
    assert abs(Z - wZ) <= 1e-5 * wZ, (Z, wZ)
    assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want) + 1e-12
    assert np.array_equal(ran, stepped)
