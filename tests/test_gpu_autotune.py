"""The autotuners time the shapes that a layout or a batch can run and name the
one that runs: up to 45,056 points there is one symmetric shape."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2310_11186_gb300 as pkg  # noqa: E402
import tsgne_synth as synth  # noqa: E402


@pytest.mark.parametrize("n,apply", [(3000, 2), (20000, 2), (45056, 2), (45057, 5)])
@pytest.mark.parametrize("precision", [0, 1])
def test_shapes_of_a_layout(n, apply, precision):
    rp = np.zeros(n + 1, np.int64)
    with pkg.Layout(precision=precision) as lay:
        lay.set_P(rp, np.zeros(0, np.int32), np.zeros(0, np.float32))
        lay.init_Y(synth.y_init(n, seed=1))
        default = lay.repulsion_shape()
        chosen, ms = lay.autotune(2)
        timed = [s for s, t in zip(pkg.Layout.REPULSION_SHAPES, ms.values()) if t > 0]
        assert len(timed) == apply - precision and chosen in timed  # BF16: no ordered pass
        assert all(t == -1.0 for s, t in zip(pkg.Layout.REPULSION_SHAPES, ms.values()) if s not in timed)
        if apply == 2 and chosen[2]:
            assert chosen == (1, 8, 1) and lay.repulsion_shape() == default


def test_shapes_of_a_batch():
    def member(b, n, **kw):
        g = synth.random_graph(n, 6.0, seed=n)
        return b.add(g.row_ptr, g.col, np.zeros((n, 2), np.float32), synth.y_init(n, seed=2), **kw)

    with pkg.Batch() as b:
        b.set_shape(2, 16)
        member(b, 3000)
        member(b, 20000)
        member(b, 46000, repulsion=1)
        for _ in range(2):
            chosen, ms = b.autotune_shapes(trial_iters=2)
            assert chosen == b.shape() == (2, 16) and len(set(ms.values())) == 1 and min(ms.values()) > 0
        w, ms3 = b.autotune(trial_iters=2)
        assert w == 2 and len(set(ms3.values())) == 1 and min(ms3.values()) > 0 and b.cached_tile() == 2
        member(b, 46000)
        chosen, ms = b.autotune_shapes(trial_iters=2)
        assert chosen == b.shape() and len(set(ms.values())) > 1 and min(ms.values()) > 0
