"""Shortest paths at the sizes where a level's work is divided: searches that end
at, before and after the levels after which the host looks (paths of k nodes,
limits l0), rows of 31 to 33 entries and a hub, nodes left over from a warp,
every number of mask words, targets that reach nothing.  Whole numbers: equal."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2310_11186_gb300 as pkg  # noqa: E402
import tsgne_synth as synth  # noqa: E402


def _check(n, u, v, targets, l0):
    rp, col = synth.csr_from_edges(n, np.asarray(u, np.int64), np.asarray(v, np.int64))
    targets = np.asarray(targets, np.int32)
    X = pkg.tsgne_shortest_path_embedding(rp, col, targets, l0)
    srp, scol = oracle.structure(n, rp, col)
    limit = l0 if l0 > 0 else oracle.default_l0(scol.size // 2)
    assert np.array_equal(X, oracle.shortest_path_embedding(n, srp, scol, targets, limit).astype(np.float32))


@pytest.mark.parametrize("k", [2, 4, 5, 6, 8, 9, 13, 40])
@pytest.mark.parametrize("l0", [1, 3, 4, 5, 8, 100])
def test_paths(k, l0):
    _check(k + 3, np.arange(k - 1), np.arange(1, k), [0, k - 1, k // 2, k + 1, 0], l0)


@pytest.mark.parametrize("d", [1, 32, 33, 64, 65, 128, 129, 256, 300, 1024])
def test_hubs_and_words(d):
    rng = np.random.default_rng(d)
    n = 1501
    u = np.concatenate([np.full(900, 7), np.full(31, 20), np.full(32, 21), np.full(33, 22), rng.integers(1400, size=1500)])
    v = np.concatenate([np.arange(100, 1000), np.arange(400, 431), np.arange(500, 532), np.arange(600, 633),
                        rng.integers(1400, size=1500)])
    keep = u != v
    _check(n, u[keep], v[keep], rng.integers(n, size=d), 0)
