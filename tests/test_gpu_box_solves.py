"""The solver's and the V-cycle's kernels by row boxes (operators of 65536 rows and more), the V-cycle's kernels for
small levels, and the projection by lines of cells, at the widths, chunk counts and remainders where they differ.

Fixed-step solves against the oracle's, column by column: 1e-10 of the column's norm. Each of the at most 3 x 2 x 6
products is right to 1e-12 of |A||X| (test_gpu_boxes.py), and a relative change of the products reaches X about
threefold (the oracle with a perturbed operator). V-cycles as in test_gpu_amg.py: 1e-11 (float64) and 1e-4 (float32)
of the column's largest value. Projection as in test_gpu_projection.py: 1e-14 of the terms' magnitude.
"""

import numpy as np
import pytest

import gen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ens():
    from paper_1711_10622_gb300 import build

    build.build()
    import paper_1711_10622_gb300 as ens

    return ens


_made = {}


def _cubes():
    if "op" not in _made:
        _made["op"] = gen.cubes(97, 43, 37, size=6)
        assert _made["op"].n >= 65536
    return _made["op"]


@pytest.mark.parametrize("use_graph", [1, 0])
@pytest.mark.parametrize("m,precond,steps", [(4, "none", 1), (4, "chebyshev", 1), (8, "chebyshev", 2), (8, "none", 1), (16, "chebyshev", 3),
                                             (24, "chebyshev", 4), (8, "chebyshev", 5), (6, "chebyshev", 4), (3, "chebyshev", 3)])
def test_fixed_steps(ens, m, precond, steps, use_graph):
    op = _cubes()
    B = gen.rhs_normal(op.n, m, 60 + m, zero_mean=True)
    X0 = gen.rhs_normal(op.n, m, 61 + m)
    kw = dict(precond=precond, cheb_steps=steps)
    with ens.Matrix.from_operator(op) as A:
        for x0 in (None, X0):
            X, st = ens.solve_block(A, torch.from_numpy(B).cuda(), None if x0 is None else torch.from_numpy(x0.copy()).cuda(), tol=0.0, max_iter=3,
                                    use_graph=use_graph, **kw)
            Xo, it, _, _ = oracle.solve_block(op, B, 0.0, X0=x0, max_iter=3, parallel=True, **kw)
            assert st["iters"].tolist() == it.tolist() == [3] * m
            X = X.cpu().numpy()
            assert np.all(np.linalg.norm(X - Xo, axis=0) <= 1e-10 * np.linalg.norm(Xo, axis=0))


@pytest.mark.parametrize("precond", ["chebyshev", "amg"])
@pytest.mark.parametrize("m", [4, 8, 16])
def test_mixed_to_tolerance(ens, m, precond):
    op = _cubes()
    B = gen.rhs_normal(op.n, m, 70 + m, zero_mean=True)
    with ens.Matrix.from_operator(op) as A:
        if precond == "amg":
            A.amg_setup()
        X, st = ens.solve_block(A, torch.from_numpy(B).cuda(), tol=1e-10, precond=precond, precision="mixed")
    assert (st["status"] == 0).all(), st
    R = B - oracle.gspmv(op, X.cpu().numpy())
    assert np.all(np.linalg.norm(R, axis=0) <= 1.05e-10 * np.linalg.norm(B, axis=0))


def test_coupled_keeps_its_rounding(ens):
    """The coupled solver's recurrence amplifies rounding: this block of right-hand sides converges with row-by-row
    products (about 100 iterations) and did not in 400 with those of row boxes."""
    op = gen.channel(96, 64, 48)
    B = gen.rhs_normal(op.n, 8, 1, zero_mean=True)
    with ens.Matrix.from_operator(op) as A:
        X, st = ens.solve_block_coupled(A, torch.from_numpy(B).cuda(), tol=1e-8, precond="chebyshev", max_iter=400)
    assert (st["status"] == 0).all()
    R = B - oracle.gspmv(op, X.cpu().numpy())
    assert np.all(np.linalg.norm(R, axis=0) <= 1.05e-8 * np.linalg.norm(B, axis=0))


def test_columns_are_independent(ens):
    """A column's bits do not depend on the other columns, whether these converge, start at zero or are not finite."""
    op = _cubes()
    B = gen.rhs_normal(op.n, 8, 80, zero_mean=True)
    C = B.copy()
    C[:, 1] *= 1e3
    C[:, 2] = 0.0
    C[5, 3] = np.nan
    with ens.Matrix.from_operator(op) as A:
        X, s = ens.solve_block(A, torch.from_numpy(B).cuda(), tol=1e-6, precond="chebyshev")
        Y, t = ens.solve_block(A, torch.from_numpy(C).cuda(), tol=1e-6, precond="chebyshev")
    assert t["status"][2] == 0 and t["status"][3] == 3 and not Y[:, 2].any()
    for l in (0, 4, 5, 6, 7):
        assert torch.equal(X[:, l], Y[:, l]) and s["iters"][l] == t["iters"][l]


def _vcycle(ens, op, m, opts):
    key = (op.n, tuple(sorted(opts.items())))
    if key not in _made:
        o = dict(opts)
        _made[key] = oracle.AMG(op, smooth=o.pop("smooth_steps", 2), coarse=o.pop("coarse_steps", 16), **o)
    R = gen.rhs_normal(op.n, m, 40 + m)
    ref = _made[key].vcycle(R)
    with ens.Matrix.from_operator(op) as A:
        assert A.amg_setup(**opts) == _made[key].sizes
        Z = ens.amg_apply(A, torch.from_numpy(R).cuda()).cpu().numpy()
        Z32 = ens.amg_apply(A, torch.from_numpy(R.astype(np.float32)).cuda()).cpu().numpy()
    scale = np.abs(ref).max(axis=0)
    assert np.all(np.abs(Z - ref).max(axis=0) <= 1e-11 * scale)
    assert np.all(np.abs(Z32 - ref).max(axis=0) <= 1e-4 * scale)


@pytest.mark.parametrize("m", [1, 4, 6, 8, 16, 24])
def test_vcycle_boxes(ens, m):
    _vcycle(ens, _cubes(), m, dict(theta=0.08, max_levels=8))


@pytest.mark.parametrize("name", ["cubes97x43x37", "dirichlet48"])
def test_float32_cycle_error(ens, name):
    """The float32 cycle by row boxes (m = 8) is as close to the float64 one as row by row (the same columns with m = 6):
    both round as often, so their errors agree to a few percent where no rounding repeats from row to row."""
    op = _cubes() if name.startswith("cubes") else gen.dirichlet_box(48)
    R = torch.randn(op.n, 8, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5))
    err = []
    with ens.Matrix.from_operator(op) as A:
        A.amg_setup()
        Z = ens.amg_apply(A, R.double())[:, :6]
        for m in (6, 8):
            err.append(float((ens.amg_apply(A, R[:, :m].contiguous()).double()[:, :6] - Z).norm() / Z.norm()))
    assert err[1] <= 1.15 * err[0], err


@pytest.mark.parametrize("m", [1, 2, 5, 8, 33, 64])
@pytest.mark.parametrize("nx,opts", [
    (45, dict(coarse_size=512, coarse_steps=16)),  # dense coarsest level
    (45, dict(coarse_size=512, coarse_steps=1)),
    (45, dict(coarse_size=5000, coarse_steps=5)),  # a coarsest level of 4177 rows
    (45, dict(coarse_size=16, smooth_steps=1)),
    (45, dict(coarse_size=16, smooth_steps=3)),
    (30, dict(max_levels=2)),  # a coarsest level of 1117 rows
], ids=str)
def test_vcycle_small_levels(ens, m, nx, opts):
    if nx not in _made:
        _made[nx] = gen.cubes(nx, nx * 2 // 3, nx * 3 // 5, size=4)
    _vcycle(ens, _made[nx], m, dict(dict(theta=0.08, max_levels=8), **opts))


@pytest.mark.parametrize("name", ["dirichlet33x17x9", "channel37x9x11", "channel64x16x8", "channel3x3x3", "dirichlet1x8x5"])
@pytest.mark.parametrize("m", [1, 2, 4, 5, 6, 8, 12])
def test_projection_lines(ens, name, m):
    """Lines of cells whose length times the lanes of a row is no multiple of a warp, and y extents that are no
    multiple of the marched run."""
    op = {"dirichlet33x17x9": lambda: gen.dirichlet_box(33, nz=9, ny=17), "channel37x9x11": lambda: gen.channel(37, 9, 11),
          "channel64x16x8": lambda: gen.channel(64, 16, 8), "channel3x3x3": lambda: gen.channel(3, 3, 3),
          "dirichlet1x8x5": lambda: gen.dirichlet_box(1, nz=5, ny=8)}[name]()
    g = gen.grid_of(op)
    U, V, W = gen.predictor_velocity(g, m, 100 + m, noise=0.3)
    P = np.random.default_rng(m).standard_normal((op.n, m))
    with ens.Grid.from_grid(g) as G:
        d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (U, V, W, P)]
        D = ens.divergence(G, *d[:3], scale=-2.5).cpu().numpy()
        ens.grad_correct(G, d[3], *d[:3], 0.013)
        got = [t.cpu().numpy() for t in d[:3]]
    w = [np.diff(a) for a in g.nodes]
    area = max(w[0].max() * w[1].max(), w[0].max() * w[2].max(), w[1].max() * w[2].max())
    bound = 2.5 * 6 * area * max(np.abs(c).max() for c in (U, V, W))
    assert np.all(np.abs(D - oracle.divergence(g, U, V, W, scale=-2.5)) <= 1e-14 * bound)
    ref = oracle.grad_correct(g, P, U, V, W, 0.013)
    corr = oracle.grad_correct(g, P, *(np.zeros_like(c) for c in (U, V, W)), 0.013)
    for a, b, c, e in zip(got, ref, (U, V, W), corr):
        assert np.all(np.abs(a - b) <= 1e-14 * (np.abs(b) + np.abs(c) + np.abs(e)))
