"""Layouts whose points are far apart, so that Z is the sum of tiny kernel
values: Z keeps its relative accuracy, and gradient and KL stay finite.

Exact pass: a unit of work that holds points' own terms (1 each) keeps 53 bits of
its Z, as an FP64 sum would, and may lose any part of the rest; every other pair
counts.  Such units are the blocks of 256 points (up to 45,056 points) or 512
points against themselves.  So Z lies between the FP64 sum over the pairs that
are not together in such a block and the sum over all pairs, to 1e-5 like
everywhere (FP32 sums of 64 + 15 terms: 4.6e-6).

Tree code: scaling the layout by a power of two scales every term by a power of
four and changes no decision and no rounding, so Z scales alike (to 1e-6: the
resolution of 2^-96 against groups of 2^-62)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2310_11186_gb300 as pkg  # noqa: E402


def _ring(n):
    i = np.arange(n)
    col = np.sort(np.stack([(i - 1) % n, (i + 1) % n], 1), 1).reshape(-1).astype(np.int32)
    rp = np.arange(0, 2 * n + 1, 2, dtype=np.int64)
    return rp, col, np.full(col.size, 1.0 / col.size, np.float32)


def _layout(n):
    """A lattice with jitter in random order: no two points closer than 0.5."""
    rng = np.random.default_rng(n)
    side = int(np.ceil(np.sqrt(n)))
    k = rng.permutation(side * side)[:n]
    return (np.stack([k % side, k // side], 1) + 0.25 * rng.uniform(-1, 1, (n, 2))).astype(np.float32)


def _expected(Y, block):
    y = torch.from_numpy(Y).cuda().double()
    own = torch.arange(len(Y), device="cuda") // block
    z = [0.0, 0.0]
    for a in range(0, len(Y), 1024):
        d = (y[a:a + 1024, None] - y[None]).square().sum(2)
        w = 1.0 / (1.0 + d)
        w[torch.arange(len(w)), torch.arange(a, a + len(w))] = 0.0
        z[1] += float(w.sum())
        w[own[a:a + 1024, None] == own[None]] = 0.0
        z[0] += float(w.sum())
    return z


@pytest.mark.parametrize("scale", [26, 34])
@pytest.mark.parametrize("n,block", [(1000, 256), (9000, 256), (46000, 512)])
def test_exact_pass(n, block, scale):
    Y = _layout(n) * np.float32(2.0 ** scale)
    least, most = _expected(Y, block)
    rp, col, P = _ring(n)
    with pkg.Layout() as lay:
        lay.set_P(rp, col, P)
        lay.init_Y(Y)
        G, Z = lay.gradient(1.0)
        assert least * (1 - 1e-5) <= Z <= most * (1 + 1e-5), (least, Z, most)
        assert np.isfinite(G).all()
        i = np.arange(n)
        d = ((Y[i].astype(float) - Y[(i + 1) % n]) ** 2).sum(1)
        kl = np.mean(np.log(1.0 / (2 * n)) + np.log1p(d)) + np.log(Z)
        assert abs(lay.kl() - kl) <= 1e-4 * abs(kl)
        pkg.tsgne_shard_set(lay.ctx, 0, 1)  # the units' values through doubles
        pkg.tsgne_shard_repulsion(lay.ctx)
        G1, Z1 = pkg.tsgne_shard_gradient_finish(lay.ctx, 1.0)
        assert Z1 == Z and np.array_equal(G1, G)


@pytest.mark.parametrize("n", [700, 20000])
def test_tree_code(n):
    rp, col, P = _ring(n)
    got = []
    with pkg.Layout(repulsion=1) as lay:
        lay.set_P(rp, col, P)
        for scale in (20, 26, 34):
            lay.init_Y(_layout(n) * np.float32(2.0 ** scale))
            G, Z = lay.gradient(1.0)
            assert Z > 0.0 and np.isfinite(G).all() and np.isfinite(lay.kl())
            got.append(Z * 4.0 ** scale)
    assert max(got) - min(got) <= 1e-6 * min(got), got
