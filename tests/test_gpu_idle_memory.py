"""Memory that the library keeps for its next allocations, measured as the
device sees it while objects are alive and after calls that destroy none: at
most 256 MiB beside what the objects hold (device_memory_in_use), plus 64 MiB
for what a context may add (modules, graphs) and for the 2 MiB pages of the
allocator."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2310_11186_gb300 as pkg  # noqa: E402
import tsgne_synth as synth  # noqa: E402

ROOM = (256 << 20) + (64 << 20)


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("call", ["build", "failed build", "embedding", "batch"])
def test_idle_memory_between_calls(call):
    n = 220000
    g = synth.random_graph(n, 20.0, seed=5)
    X = np.zeros((n, 300), np.float32)  # 252 MiB: kept whole when it comes back
    X[:, 0] = np.arange(n)
    with pkg.Layout() as lay:  # modules are loaded
        lay.build_P(*[np.asarray(a) for a in (np.array([0, 1, 2]), np.array([1, 0]), np.zeros((2, 1), np.float32))])
    pkg.set_device_memory_limit(0)
    used0, free0 = pkg.device_memory_in_use(), _free()

    def check():
        held = pkg.device_memory_in_use() - used0
        assert free0 - _free() <= held + ROOM

    if call == "build":
        with pkg.Layout(p_walks=96) as lay:
            lay.build_P(g.row_ptr, g.col, X)
            check()
    elif call == "failed build":
        X[7, 3] = np.nan
        with pkg.Layout(perplexity=5.0) as lay:
            with pytest.raises(pkg.TsgneError):
                lay.build_P(g.row_ptr, g.col, X)
            check()
    elif call == "embedding":
        pkg.tsgne_shortest_path_embedding(g.row_ptr, g.col, np.arange(256, dtype=np.int32))
        check()
    else:
        with pkg.Batch() as b:
            ids = [b.add(g.row_ptr, g.col, X[:, :4].copy()) for _ in range(16)]
            for i in ids:
                b.remove(i)
            check()
    pkg.set_device_memory_limit(0)
