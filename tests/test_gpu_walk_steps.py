"""Random walks over rows of every search length (1 to 9 entries, quarters
above 8, a hub of 1,500) and walk counts at the ends of the register sort's
widths, and distances of features that are zeros, subnormal and normal side by
side.  Both sides draw the same numbers and take the same FP64 decisions: the
structure is the same, P within 1e-6 relative for walks (the normaliser's order
of summation, one rounding to FP32) and 1e-5 for the perplexity search (its
stopping tolerance)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2310_11186_gb300 as pkg  # noqa: E402
import tsgne_synth as synth  # noqa: E402


def _graph():
    n, degrees = 2000, list(range(1, 19)) + [31, 32, 33, 40, 64, 65, 1500]
    u = np.concatenate([[i] * k for i, k in enumerate(degrees)])
    v = np.concatenate([n - 1 - (7 * i + np.arange(k)) % 1900 for i, k in enumerate(degrees)])
    return (n, *synth.csr_from_edges(n, u.astype(np.int64), v.astype(np.int64)))


def _features(n, d, seed, special):
    rng = np.random.default_rng(seed)
    X = (0.4 * rng.standard_normal((n, d))).astype(np.float32)
    if special:
        kind = rng.integers(6, size=(n, d))
        for k, val in enumerate([0.0, -0.0, 1e-40, -3e-39, 1.17549435e-38]):
            X[kind == k] = val
    return X


@pytest.mark.parametrize("special", [False, True])
@pytest.mark.parametrize("R", [1, 31, 32, 33, 64, 65, 128, 129, 256, 257])
def test_walks(R, special):
    n, rp, col = _graph()
    X = _features(n, 6, R, special)
    orp, ocol, oP = oracle.random_walk_P(n, rp, col, X.astype(np.float64), R, 3, R)
    with pkg.Layout(p_walks=R, p_walk_length=3, seed=R) as lay:
        lay.build_P(rp, col, X)
        grp, gcol, P = lay.get_P()
    assert np.array_equal(grp, orp) and np.array_equal(gcol, ocol)
    assert np.all(np.abs(P - oP) <= 1e-6 * oP + 1e-12)


@pytest.mark.parametrize("d", [1, 2, 3, 4, 8, 10])
def test_distances_of_special_floats(d):
    n, rp, col = _graph()
    X = _features(n, d, d, True)
    orp, ocol, oP = oracle.build_P(n, rp, col, X, 5.0)
    with pkg.Layout(perplexity=5.0) as lay:
        lay.build_P(rp, col, X)
        grp, gcol, P = lay.get_P()
    assert np.array_equal(grp, orp) and np.array_equal(gcol, ocol)
    assert np.all(np.abs(P - oP) <= 1e-5 * oP + 1e-9 * oP.max())
