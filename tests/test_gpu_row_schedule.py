"""The row schedule of the attraction (hub rows, chain order, copies of col
and P) is built on the device.  A layout advances on it, a batch of one on the
row-by-row definition of the same sums, so after a few iterations the two
must agree bit for bit at every degree where the schedule changes form."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2310_11186_gb300 as pkg  # noqa: E402
import tsgne_synth as synth  # noqa: E402


def _graph(degrees, n):
    """Nodes 0, 1, ... with the given degrees towards the last nodes."""
    u, v = [], []
    for i, d in enumerate(degrees):
        u += [i] * d
        v += list(range(n - d, n))
    return synth.csr_from_edges(n, np.array(u, np.int64), np.array(v, np.int64))


EDGES = [0, 1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 96, 127, 128, 129]


@pytest.mark.parametrize("degrees,n", [
    ([], 2), ([1], 255), ([3] * 200, 256), ([5] * 200, 257), (EDGES, 513),
    ([33] * 64, 1000), ([33] * 65, 1000), ([128] * 130, 1500),
    (EDGES + [1023, 1024, 1025, 2047, 2048, 2049], 4099), (EDGES, 20011), (EDGES, 50021),
])
def test_layout_equals_batch_of_one(degrees, n):
    rp, col = _graph(degrees, n)
    X = np.random.default_rng(n).standard_normal((n, 8)).astype(np.float32)
    Y0 = np.random.default_rng(n + 1).standard_normal((n, 2)).astype(np.float32)
    with pkg.Layout() as lay:
        lay.build_P(rp, col, X)
        lay.init_Y(Y0)
        tile = lay.repulsion_shape()["block"] // 32
        lay.run(3)
        Y = lay.get_Y()
    with pkg.Batch(tile_warps=tile) as b:
        k = b.add(rp, col, X, Y0)
        b.run(3)
        assert np.array_equal(b.get_Y(k)[0], Y)
