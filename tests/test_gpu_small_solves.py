"""Plain float64 solves of small systems, whose whole iteration loop is one launch: the same bits, iteration counts
and statuses as the host-driven loop of separate kernels (both visit rows and add sums in the same order), at the
edges of widths, tiles and resident blocks; the kernels themselves are compared with the oracle in test_gpu_solver.py.
"""

import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ens():
    from paper_1711_10622_gb300 import build

    build.build()
    import paper_1711_10622_gb300 as ens

    return ens


def _long_rows(n, k):
    """Diagonally dominant, k nonzeros per row, spread over the columns: tiles that do not fit in shared memory."""
    rng = np.random.default_rng(n + k)
    col = (np.arange(n)[:, None] + np.sort(rng.choice(n - 1, k - 1, replace=False)) + 1) % n
    col = np.concatenate([np.arange(n)[:, None], col], 1)
    val = np.concatenate([np.full((n, 1), 2.0 * k), rng.standard_normal((n, k - 1))], 1)
    order = np.argsort(col, 1)
    rp = (np.arange(n + 1) * k).astype(np.int32)
    return gen.Operator("long", (n, 1, 1), ("x",) * 3, rp, np.take_along_axis(col, order, 1).astype(np.int32).ravel(),
                        np.take_along_axis(val, order, 1).ravel(), False)


OPS = {
    "dirichlet1": lambda: gen.dirichlet_box(1),
    "dirichlet8": lambda: gen.dirichlet_box(8),
    "dirichlet32": lambda: gen.dirichlet_box(32),
    "channel24x16x12": lambda: gen.channel(24, 16, 12),
    "cubes48x32x24": lambda: gen.cubes(48, 32, 24, size=4),
    "dirichlet32x32x36": lambda: gen.dirichlet_box(32, ny=32, nz=36),  # m = 4: 288 blocks
    "dirichlet32x32x41": lambda: gen.dirichlet_box(32, ny=32, nz=41),  # ... 328: separate kernels
    "dirichlet24x24x21": lambda: gen.dirichlet_box(24, ny=24, nz=21),  # m = 8: 189 blocks
    "dirichlet24x24x22": lambda: gen.dirichlet_box(24, ny=24, nz=22),  # ... 198: separate kernels
    "long3000x40": lambda: _long_rows(3000, 40),
    "long20000x9": lambda: _long_rows(20000, 9),
}


def _both(ens, op, B, X0=None, **kw):
    out = []
    with ens.Matrix.from_operator(op) as A:
        for g in (1, 0):
            x0 = None if X0 is None else torch.from_numpy(X0.copy()).cuda()
            out.append(ens.solve_block(A, torch.from_numpy(B).cuda(), x0, use_graph=g, **kw))
        (Y, t), = ens.solve_batch([(A, torch.from_numpy(B).cuda(), None if X0 is None else torch.from_numpy(X0.copy()).cuda(), kw["tol"])],
                                  max_iter=kw.get("max_iter", 10000))
    (X, s), (Z, u) = out
    for W, w in ((Z, u), (Y, t)):
        assert torch.equal(X.view(torch.int64), W.view(torch.int64))
        for k in ("iters", "status", "relres"):
            np.testing.assert_array_equal(s[k], w[k])
    return X, s


@pytest.mark.parametrize("name", list(OPS))
@pytest.mark.parametrize("m", [1, 2, 3, 4, 6, 8, 10])
def test_same_bits(ens, name, m):
    op = OPS[name]()
    B = gen.rhs_normal(op.n, m, 30 + m, zero_mean=op.singular)
    X, s = _both(ens, op, B, tol=1e-9)
    assert (s["status"] == 0).all() and np.all(s["relres"] <= 1.05e-9)
    X, s = _both(ens, op, B, gen.rhs_normal(op.n, m, 31), tol=0.0, max_iter=3)


def test_same_statuses(ens):
    """Zero, incompatible and not finite columns, values outside the split range, an iteration cap."""
    op = gen.channel(16, 12, 8)
    B = gen.rhs_normal(op.n, 8, 5, zero_mean=True)
    B[:, 1] = 0.0
    B[:, 2] = 1.0
    B[7, 3] = np.nan
    B[:, 4] *= 1e-30
    B[:, 5] *= 1e40
    X, s = _both(ens, op, B, tol=1e-9)
    assert s["status"].tolist() == [0, 0, 4, 3, 0, 0, 0, 0]
    X, s = _both(ens, op, B, tol=1e-13, max_iter=2)
    assert s["status"].tolist() == [1, 0, 4, 3, 1, 1, 1, 1]
    X, s = _both(ens, op, B, tol=1e-13, max_iter=0)
