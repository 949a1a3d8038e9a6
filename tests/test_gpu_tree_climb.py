"""The tree built in tiles of 1,024 nodes and 48 tiles a step: the sums over it
against the oracle's restatement of the tree code, which builds the tree from
its definition, top down.  Sizes stand at the ends of a tile, of one step and of
two; the nested layout makes more subtrees cross the tiles' ends than a tile of
the second (50,876 points) or last (48,128) step holds.  Both sides make the
same FP32 decisions and sum in other orders, so the tolerances are those of FP32
sums of a few thousand terms: 1e-4 (relative L2 of the gradient) and 1e-5 (Z)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2310_11186_gb300 as pkg  # noqa: E402


def _nested(n, rng):
    """Clusters of 1,024 points around centres of a grid; a point differs from
    its centre from one random bit of one 24-bit coordinate downwards, so that
    every depth of the tree branches near a centre."""
    k, side = np.maximum(np.arange(n) - 512, 0) // 1024, 8  # a tile ends amid a cluster
    centre = rng.integers(1 << 19, size=(n // 1024 + 1, 2))
    c = np.stack([k % side, k // side], 1) * (1 << 19) * 4 + centre[k]
    b = rng.integers(19, size=n)
    axis = np.arange(n) & 1
    c[np.arange(n), axis] ^= (1 << b) | rng.integers(1 << b)
    return (c * 2.0 ** -20).astype(np.float32)


@pytest.mark.parametrize("n,kind,theta", [
    (1023, "spread", 0.5), (1024, "spread", 0.5), (1025, "spread", 0.5), (2049, "one spot", 0.5),
    (49152, "spread", 0.7), (49153, "spread", 0.7), (48128, "nested", 0.7), (50876, "nested", 0.7),
    (2359297, "spread", 1.0),
])
def test_tiled_tree(n, kind, theta):
    rng = np.random.default_rng(n)
    if kind == "nested":
        Y = _nested(n, rng)
    else:
        Y = (rng.standard_normal((n, 2)) * (5.0 if kind == "spread" else 0.0) + 1.0).astype(np.float32)
    rp, col, P = np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32)
    want, wZ = oracle.gradient_tree(n, rp, col, P, Y, 1.0, theta=theta)
    with pkg.Layout(repulsion=1, theta=theta) as lay:
        lay.set_P(rp, col, P)
        lay.init_Y(Y)
        for _ in range(2):  # the second pass finds the first one's slots and marks
            got, Z = lay.gradient(1.0)
            assert abs(Z - wZ) <= 1e-5 * wZ, (Z, wZ)
            assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want) + 1e-12
