"""A CSR that already is the symmetric structure is recognised and copied; any
other form of the same graph (one direction, shuffled rows, repeats, loops)
takes the counting path.  Both must give the oracle's structure bit for bit,
and the copy must not be taken for inputs that differ from it in one place."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2310_11186_gb300 as pkg  # noqa: E402
import tsgne_synth as synth  # noqa: E402


def _structure(n, rp, col):
    with pkg.Layout() as lay:
        lay.build_P(rp, col, np.zeros((n, 4), np.float32) + np.arange(n, dtype=np.float32)[:, None])
        grp, gcol, _ = lay.get_P()
    return grp, gcol


def _csr(n, u, v):
    o = np.argsort(u, kind="stable")
    return np.concatenate([[0], np.cumsum(np.bincount(u, minlength=n))]).astype(np.int64), v[o].astype(np.int32)


@pytest.mark.parametrize("n,m", [(2, 1), (50, 3), (3000, 1), (5000, 60), (300, 511), (300, 512), (300, 513),
                                 (700, 5000), (4000, 30000)])
def test_every_form_of_a_graph(n, m):
    rng = np.random.default_rng(n + m)
    key = np.unique(rng.integers(0, n, (4 * m, 2)) @ np.array([n, 1]))
    u, v = key // n, key % n
    u, v = np.append(u[u < v][:m], 0), np.append(v[u < v][:m], 1)
    hub = np.arange(1, n)  # node 0 meets everybody in the denser graphs
    if m > 4000:
        u, v = np.concatenate([u, np.zeros(n - 1, np.int64)]), np.concatenate([v, hub])
    rp, col = synth.csr_from_edges(n, *np.unique(np.stack([u, v]), axis=1))
    orp, ocol = oracle.structure(n, rp, col)[:2]
    assert np.array_equal(rp, orp) and np.array_equal(col, ocol)  # the input is its own structure
    forms = [(rp, col), _csr(n, u, v), _csr(n, v, u)]
    both_u, both_v = np.concatenate([u, v, u, np.arange(3) % n]), np.concatenate([v, u, v, np.arange(3) % n])
    p = rng.permutation(both_u.size)
    forms.append(_csr(n, both_u[p], both_v[p]))
    for f in forms:
        grp, gcol = _structure(n, *f)
        assert np.array_equal(grp, orp) and np.array_equal(gcol, ocol)


def test_one_entry_away_from_the_structure():
    g = synth.random_graph(600, 9.0, seed=3)
    rp, col = oracle.structure(g.n, g.row_ptr, g.col)[:2]
    row = np.repeat(np.arange(g.n), np.diff(rp))
    e = int(np.argmax(np.diff(rp)[row] >= 3))  # first entry of a row of at least three
    one_way = np.delete(np.stack([row, col]), e, axis=1)
    swapped = col.copy()
    swapped[[e, e + 1]] = swapped[[e + 1, e]]
    looped = col.copy()
    looped[e] = row[e]
    for r, c in (_csr(g.n, one_way[0], one_way[1]), (rp, swapped), (rp, looped)):
        orp, ocol = oracle.structure(g.n, r, c)[:2]
        grp, gcol = _structure(g.n, r, c)
        assert np.array_equal(grp, orp) and np.array_equal(gcol, ocol)
