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


@pytest.mark.parametrize("m", [4, 8])
@pytest.mark.parametrize("name", ["cubes97x43x37", "dirichlet48"])
def test_coupled_with_vcycle_by_boxes(ens, name, m):
    """The coupled solver with the V-cycle, whose fine level runs by row boxes: several blocks of right-hand sides
    converge, and the true residuals are what the statuses say."""
    op = _cubes() if name.startswith("cubes") else gen.dirichlet_box(48)
    with ens.Matrix.from_operator(op) as A:
        A.amg_setup()
        for seed in range(1, 7):
            B = gen.rhs_normal(op.n, m, seed, zero_mean=op.singular)
            X, st = ens.solve_block_coupled(A, torch.from_numpy(B).cuda(), tol=1e-8, precond="amg", max_iter=100)
            assert (st["status"] == 0).all(), (seed, st)
            R = B - oracle.gspmv(op, X.cpu().numpy())
            assert np.all(np.linalg.norm(R, axis=0) <= 1.05e-8 * np.linalg.norm(B, axis=0)), seed


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


def test_float32_small_level_error(ens):
    """The float32 cycle with four threads per row (m = 8) is about as close to the float64 one as with two (m = 16): 1.04
    times; 1.14 while each thread's first product was rounded on its own."""
    op = gen.channel(32, 32, 32)
    err = np.zeros(2)
    with ens.Matrix.from_operator(op) as A:
        A.amg_setup()
        for seed in range(24):
            R = torch.randn(op.n, 16, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))
            Z = ens.amg_apply(A, R.double())[:, :8]
            for k, m in enumerate((16, 8)):
                E = ens.amg_apply(A, R[:, :m].contiguous()).double()[:, :8] - Z
                err[k] += float((E.norm(dim=0) / Z.norm(dim=0)).square().sum())
    assert np.sqrt(err[1] / err[0]) <= 1.09, err


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


def _us(f, n=9):
    """Median time of f() in microseconds, after three untimed calls."""
    t = []
    for k in range(n + 3):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        if k > 2:
            t.append(a.elapsed_time(b) * 1e3)
    return float(np.median(t))


def test_projection_cost(ens):
    """The correction of one and two states per thread costs what the general kernel takes: m = 2 two thirds of m = 4's
    time and m = 6 that of m = 8 (by lines 0.95 and 1.37 times); and a small grid's divergence of 32 states (four per
    thread) at most 1.15 times that of 31 (one per thread; by lines of eight cells 1.4 times)."""
    op = gen.channel(128, 128, 128)
    with ens.Grid.from_grid(gen.grid_of(op)) as G:
        t = {}
        for m in (2, 4, 6, 8):
            U, V, W, P = (torch.randn(k, m, dtype=torch.float64, device="cuda") for k in (op.n, op.n // 128 * 129, op.n, op.n))
            t[m] = _us(lambda: ens.grad_correct(G, P, U, V, W, tau=1e-3))
    assert t[2] <= 0.8 * t[4] and t[6] <= 1.15 * t[8], t
    op = gen.dirichlet_box(20)
    g = gen.grid_of(op)
    with ens.Grid.from_grid(g) as G:
        for m in (31, 32):
            U, V, W = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in gen.predictor_velocity(g, m, 3, noise=0.1))
            D = torch.empty(op.n, m, dtype=torch.float64, device="cuda")
            t[m] = _us(lambda: [ens.divergence(G, U, V, W, scale=2.0, D=D) for _ in range(20)])
    assert t[32] <= 1.15 * t[31], t


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


@pytest.mark.parametrize("name,m", [("dirichlet45x61x47", 6), ("dirichlet45x61x47", 12), ("channel67x53x48", 6), ("channel67x53x48", 8),
                                    ("channel67x53x48", 10)])
def test_divergence_lines(ens, name, m):
    """Grids large enough for the divergence by lines of eight cells, with ragged lines and runs; two and four states
    per thread; boundary faces of every kind; face values outside the split range in some states."""
    op = gen.dirichlet_box(45, nz=47, ny=61) if name.startswith("dirichlet") else gen.channel(67, 53, 48)
    g = gen.grid_of(op)
    U, V, W = (np.ascontiguousarray(a) for a in gen.predictor_velocity(g, m, 100 + m, noise=0.3))
    W[:, 1] *= 1e-16
    U[::7, 2] *= 1e30
    with ens.Grid.from_grid(g) as G:
        D = ens.divergence(G, *(torch.from_numpy(a).cuda() for a in (U, V, W)), scale=-2.5).cpu().numpy()
    w = [np.diff(a) for a in g.nodes]
    area = max(w[0].max() * w[1].max(), w[0].max() * w[2].max(), w[1].max() * w[2].max())
    bound = 2.5 * 6 * area * np.maximum.reduce([np.abs(c).max(axis=0) for c in (U, V, W)])
    assert np.all(np.abs(D - oracle.divergence(g, U, V, W, scale=-2.5)) <= 1e-14 * bound)
