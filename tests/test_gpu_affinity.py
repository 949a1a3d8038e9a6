"""Conditional affinities where their kernels change form: rows around 8, 32
and the perplexity (packed search, warp search, uniform rows), pairs with one
uniform end, embedding widths and addresses that allow 16-, 8- or 4-byte loads.
P against the FP64 oracle at the parity tests' tolerance (1e-5 relative)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2310_11186_gb300 as pkg  # noqa: E402
import tsgne_synth as synth  # noqa: E402

DEGREES = [1, 2, 3, 5, 6, 7, 8, 9, 16, 17, 24, 25, 31, 32, 33, 40, 63, 64, 65, 200, 700]


def _case(d, seed):
    n = 1000
    u = np.concatenate([[i] * k for i, k in enumerate(DEGREES)])
    v = np.concatenate([n - 1 - np.arange(k) for k in DEGREES])
    rp, col = synth.csr_from_edges(n, u.astype(np.int64), v.astype(np.int64))
    X = (2.0 * np.random.default_rng(seed).standard_normal((n, d))).astype(np.float32)
    return n, rp, col, X


def _check(P, oP):
    assert np.all(np.abs(P - oP) <= 1e-5 * oP + 1e-9 * oP.max())


@pytest.mark.parametrize("perp", [1.5, 5.0, 30.0])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 6, 50, 64])
def test_P_against_the_oracle(perp, d):
    n, rp, col, X = _case(d, 7 * d)
    orp, ocol, oP = oracle.build_P(n, rp, col, X, perp)
    with pkg.Layout(perplexity=perp) as lay:
        lay.build_P(rp, col, X)
        grp, gcol, P = lay.get_P()
    assert np.array_equal(grp, orp) and np.array_equal(gcol, ocol)
    _check(P, oP)


@pytest.mark.parametrize("offset", [0, 1, 2])
def test_unaligned_device_embedding(offset):
    n, rp, col, X = _case(4, 3)
    _, _, oP = oracle.build_P(n, rp, col, X, 5.0)
    flat = torch.empty(n * 4 + offset, device="cuda")
    flat[offset:] = torch.from_numpy(X).reshape(-1).cuda()
    Xd = flat[offset:].reshape(n, 4)
    assert Xd.data_ptr() % 16 == (4 * offset) % 16
    with pkg.Layout(perplexity=5.0) as lay:
        lay.build_P(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), Xd)
        _check(lay.get_P()[2], oP)
