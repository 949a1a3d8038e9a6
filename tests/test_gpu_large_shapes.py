"""The exact pass's kernels of layouts above 45,056 points, which smaller ones
never run: every symmetric shape (1 or 2 warps, 8 or 16 i-points per lane) with
FP32 and BF16 storage, the batch's shapes (up to 4 warps) and a pass divided
over three contexts.  Gradient, Z and one optimiser step against the FP64
oracle at the parity tests' tolerances (1e-4 relative L2, Z 1e-5); the divided
pass and the batch's shapes that a single layout has too must equal the single
layout's bits."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2310_11186_gb300 as pkg  # noqa: E402
import tsgne_synth as synth  # noqa: E402

N = 46001
SHAPES = [(1, 8), (2, 8), (1, 16), (2, 16)]


def _bf16(a):
    return torch.from_numpy(np.asarray(a, np.float32)).to(torch.bfloat16).double().numpy()


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.fixture(scope="module")
def case():
    g = synth.random_graph(N, 7.0, seed=51)
    labels = (np.arange(N) % 7).astype(np.int32)
    X = synth.block_embedding(labels, 8, seed=51)
    rp, col, P = oracle.build_P(N, g.row_ptr, g.col, X, 30.0)
    P = P.astype(np.float32)
    Y = synth.spread_layout(labels, scale=20.0, seed=52)
    want = {p: oracle.gradient(N, rp, col, r(P), r(Y), 1.0) for p, r in ((0, lambda a: a.astype(float)), (1, _bf16))}
    return {"g": g, "X": X, "rp": rp, "col": col, "P": P, "Y": Y, "want": want}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_gradient(case, shape, precision):
    oG, oZ = case["want"][precision]
    with pkg.Layout(precision=precision) as lay:
        lay.set_P(case["rp"], case["col"], case["P"])
        lay.init_Y(case["Y"])
        lay.set_repulsion_shape(*shape)
        assert lay.repulsion_shape()["block"] == 32 * shape[0] and lay.repulsion_shape()["i_per_thread"] == shape[1]
        G, Z = lay.gradient(1.0)
        G2, Z2 = lay.gradient(1.0)
    assert abs(Z - oZ) <= 1e-5 * oZ
    assert _rel(G, oG) <= 1e-4
    assert np.array_equal(G, G2) and Z == Z2


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_three_contexts(case, shape, precision):
    lays = [pkg.Layout(precision=precision) for _ in range(3)]
    accs, zs = [], []
    for r, lay in enumerate(lays):
        lay.set_P(case["rp"], case["col"], case["P"])
        lay.init_Y(case["Y"])
        lay.set_repulsion_shape(*shape)
        G1, Z1 = lay.gradient(1.0)
        pkg.tsgne_shard_set(lay.ctx, r, 3)
        _, _, _, acc, zunit = pkg.tsgne_shard_repulsion(lay.ctx)
        accs.append(torch.as_tensor(acc, device="cuda"))
        zs.append(torch.as_tensor(zunit, device="cuda"))
    torch.cuda.synchronize()
    acc, z = sum(a.clone() for a in accs), sum(t.clone() for t in zs)
    for a, t in zip(accs, zs):
        a.copy_(acc)
        t.copy_(z)
    torch.cuda.synchronize()
    for lay in lays:
        G, Z = pkg.tsgne_shard_gradient_finish(lay.ctx, 1.0)
        assert Z == Z1 and np.array_equal(G, G1)
        lay.close()


@pytest.mark.parametrize("shape", [(1, 8), (2, 8), (4, 8), (1, 16), (2, 16), (4, 16)])
def test_batch(case, shape):
    Y0 = synth.y_init(N, seed=53)
    small = synth.random_graph(3001, 6.0, seed=54)
    Xs = np.zeros((small.n, 2), np.float32)
    with pkg.Batch() as b:
        b.set_shape(*shape)
        b.add(small.row_ptr, small.col, Xs)
        i = b.add(case["g"].row_ptr, case["g"].col, case["X"], Y0)
        b.run(1)
        Y = b.get_Y(i)[0]
    oY, _, _ = oracle.optimize(N, case["rp"], case["col"], case["P"].astype(float), Y0, 1)
    assert _rel(Y, oY) <= 1e-4
    if shape in SHAPES:
        with pkg.Layout() as lay:
            lay.build_P(case["g"].row_ptr, case["g"].col, case["X"])
            lay.init_Y(Y0)
            lay.set_repulsion_shape(*shape)
            lay.run(1)
            assert np.array_equal(lay.get_Y(), Y)
