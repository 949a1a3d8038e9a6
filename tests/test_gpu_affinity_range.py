"""The perplexity search where FP32 sums of distances overflow: squared
distances up to 3e38, which take more than the default number of steps (beta
ends near 1e-38).  P against the FP64 oracle at the parity tests' tolerance
(1e-5 relative)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2310_11186_gb300 as pkg  # noqa: E402
import tsgne_synth as synth  # noqa: E402


# rows of about 30 (packed search) and 200 entries (warp per row); a perplexity near the degree
@pytest.mark.parametrize("deg,perp", [(28.0, 24.0), (28.0, 5.0), (200.0, 160.0)])
def test_squared_distances_near_the_end_of_fp32(deg, perp):
    n = 600
    g = synth.random_graph(n, deg, seed=int(deg))
    X = (1.7e19 * np.random.default_rng(1).random((n, 1))).astype(np.float32)
    _, _, oP = oracle.build_P(n, g.row_ptr, g.col, X, perp, max_iter=300)
    with pkg.Layout(perplexity=perp, bisect_max_iter=300) as lay:
        lay.build_P(g.row_ptr, g.col, X)
        P = lay.get_P()[2]
    assert np.all(np.abs(P - oP) <= 1e-5 * oP + 1e-9 * oP.max())
