"""The tree of a layout that takes two launches of the tile-joining step (above
2,359,296 points) when some tiles of the first launch hold too many subtrees:
the definition's groups, point by point, against the oracle, which builds tree
and groups from their definition.

A group split where the definition has one shows only in its own points, so
every force is compared.  Both sides take the same FP32 decisions; a force is an
FP32 sum of at most about 2,000 terms whose absolute sum is a few times the
forces' root mean square, so 1e-3 of that covers the worst rounding (2,000 x
2^-24 x 4 = 5e-4).  A wrong group opens and accepts other nodes at theta = 1."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2310_11186_gb300 as pkg  # noqa: E402

NESTED = (2, 3, 12, 13, 30, 31, 44, 45)  # cells of 64, in the order of the curve


def _layout(n, rng):
    """Equally many points in 64 cells of a square: uniform, or clusters of
    1,024 around centres from which a point differs from one random bit of one
    coordinate downwards (every depth of the tree branches there)."""
    out = []
    for k in range(64):
        corner = [sum(((k >> (2 * b + a)) & 1) << b for b in range(3)) for a in range(2)]
        c = n // 64 + (n % 64 if k == 63 else 0)
        if k in NESTED:
            q = np.arange(c) // 1024
            centre = rng.integers(1 << 17, size=(c // 1024 + 1, 2))
            p = np.stack([q % 8, q // 8], 1) * (1 << 18) + centre[q]
            b = rng.integers(17, size=c)
            p[np.arange(c), np.arange(c) & 1] ^= (1 << b) | rng.integers(1 << b)
        else:
            p = rng.integers(1 << 21, size=(c, 2))
        out.append(p + np.array(corner) * (1 << 21))
    return (np.concatenate(out) * 2.0 ** -13).astype(np.float32)  # neighbours of the uniform cells about 1 apart


def test_groups_beside_a_tile_that_gave_up():
    n = 2400000
    Y = _layout(n, np.random.default_rng(n))
    rp, col, P = np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32)
    want, wZ = oracle.gradient_tree(n, rp, col, P, Y, 1.0, theta=1.0)
    with pkg.Layout(repulsion=1, theta=1.0) as lay:
        lay.set_P(rp, col, P)
        lay.init_Y(Y)
        got, Z = lay.gradient(1.0)
    assert abs(Z - wZ) <= 1e-5 * wZ
    err = np.linalg.norm(got - want, axis=1)
    rms = np.sqrt((want ** 2).sum(1).mean())
    print(f"largest error {err.max() / rms:.2e} of the root mean square, {(err > 1e-3 * rms).sum()} points above")
    assert err.max() <= 1e-3 * rms
