"""Device memory from the library's pool: results do not depend on what a
reused block held, objects may outlive one another and use streams and threads
of their own, and idle memory stays within its bound and goes back."""

import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2310_11186_gb300 as pkg  # noqa: E402
import tsgne_synth as synth  # noqa: E402

IDLE = 256 << 20


def _layout_of(g, X, Y0, stream=None, **cfg):
    lay = pkg.Layout(stream=stream, **cfg)
    lay.build_P(g.row_ptr, g.col, X)
    lay.init_Y(Y0)
    lay.run(4)
    return lay


def _case(n, seed):
    g = synth.random_graph(n, 8.0, seed=seed)
    rng = np.random.default_rng(seed)
    return g, rng.standard_normal((n, 12)).astype(np.float32), rng.standard_normal((n, 2)).astype(np.float32)


@pytest.mark.parametrize("cfg", [{}, {"repulsion": 1}, {"precision": 1}, {"p_walks": 8}])
def test_reused_memory_changes_nothing(cfg):
    small, large = _case(900, 1), _case(30011, 2)
    first = _layout_of(*small, **cfg)
    want = first.get_Y()
    other = _layout_of(*large, **cfg)  # alive while the first one's memory goes
    want_l = other.get_Y()
    first.close()
    again = _layout_of(*small, **cfg)
    other.run(2)
    other.close()
    assert np.array_equal(again.get_Y(), want)
    again.close()
    own = _layout_of(*large, stream=torch.cuda.Stream(), **cfg)
    assert np.array_equal(own.get_Y(), want_l)
    own.close()


def test_threads_with_streams_of_their_own():
    cases = [_case(2000 + 500 * k, 10 + k) for k in range(4)]
    want = []
    for c in cases:
        with _layout_of(*c) as lay:
            want.append(lay.get_Y())
    got, errors = [None] * 4, []

    def work(k):
        try:
            for _ in range(5):
                with _layout_of(*cases[k], stream=torch.cuda.Stream()) as lay:
                    got[k] = lay.get_Y()
                    assert np.array_equal(got[k], want[k])
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not errors, errors


def test_idle_memory_is_bounded_and_goes_back():
    g, X, Y0 = _case(400000, 5)
    X = np.zeros((g.n, 256), np.float32)  # 410 MB of input beside the build's own buffers
    X[:, 0] = np.arange(g.n)
    with _layout_of(*_case(500, 3)):
        pass
    torch.cuda.synchronize()
    pkg.set_device_memory_limit(0)
    free0, _ = torch.cuda.mem_get_info()
    with _layout_of(g, X, Y0, repulsion=1):
        pass
    torch.cuda.synchronize()
    free1, _ = torch.cuda.mem_get_info()
    assert free0 - free1 <= IDLE + (64 << 20)  # 64 MiB: what a context may add besides (graphs, modules)
    pkg.set_device_memory_limit(0)
    free2, _ = torch.cuda.mem_get_info()
    assert free2 >= free1 and free0 - free2 <= (64 << 20)
