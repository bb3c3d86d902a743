"""Products by row boxes (operators of 65536 rows and more) against the CPU oracle, element by element:
ragged boxes (removed cells, odd grids), rows of different lengths, every chunk remainder, misaligned blocks,
values outside the split range, zeros and non-finite values.

Tolerances as in test_gpu_gspmv.py: float64 1e-12 of |A||X| per element, float32 (row length + 2) 2^-24.
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


def _stencil9(nx, ny, points=9):
    """A two-dimensional nine-point (or five-point) operator with missing entries: rows of 4 to 9 nonzeros, some empty."""
    rng = np.random.default_rng(nx)
    j, i = np.divmod(np.arange(nx * ny), nx)
    cols, keep = [], []
    for dj in (-1, 0, 1):
        for di in (-1, 0, 1):
            if points == 5 and di and dj:
                continue
            a, b = i + di, j + dj
            cols.append(b * nx + a)
            keep.append((a >= 0) & (a < nx) & (b >= 0) & (b < ny))
    cols, keep = np.stack(cols, 1), np.stack(keep, 1)
    keep &= rng.random(nx * ny)[:, None] > 0.001  # empty rows
    rp = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int32)
    col = cols[keep].astype(np.int32)
    return gen.Operator("stencil9", (nx, ny, 1), ("x",) * 3, rp, col, rng.standard_normal(col.size), False)


OPS = {
    "cubes97x43x37": lambda: gen.cubes(97, 43, 37, size=6),
    "channel64x40x32": lambda: gen.channel(64, 40, 32),
    "dirichlet41": lambda: gen.dirichlet_box(41),
    "stencil9_301x257": lambda: _stencil9(301, 257),
}
_cache = {}


def _op(name):
    if name not in _cache:
        _cache[name] = OPS[name]()
    assert _cache[name].n >= 65536
    return _cache[name]


def _check(op, X, Y, tol=1e-12):
    X = X.astype(np.float64)
    ref = oracle.gspmv(op, X)
    S = op.to_scipy().copy()
    S.data = np.abs(S.data)
    assert np.all(np.abs(Y.astype(np.float64) - ref) <= tol * np.asarray(S @ np.abs(X)))


@pytest.mark.parametrize("name", list(OPS))
@pytest.mark.parametrize("m", [3, 4, 5, 6, 8, 11, 12, 16, 20, 24, 33])
def test_product(ens, name, m):
    op = _op(name)
    X = gen.rhs_normal(op.n, m, m)
    X32 = X.astype(np.float32)
    op32 = gen.Operator(op.name, op.shape, op.bcs, op.row_ptr, op.col_idx, op.val.astype(np.float32).astype(np.float64), False)
    with ens.Matrix.from_operator(op) as A:
        _check(op, X, ens.gspmv(A, torch.from_numpy(X).cuda()).cpu().numpy())
        L = int(np.diff(op.row_ptr).max())
        _check(op32, X32, ens.gspmv(A, torch.from_numpy(X32).cuda()).cpu().numpy(), (L + 2) * 2.0**-24)


@pytest.mark.parametrize("m", [4, 8, 16])
def test_misaligned_blocks(ens, m):
    op = _op("cubes97x43x37")
    with ens.Matrix.from_operator(op) as A:
        for off in (1, 2):
            for dt, tol in ((torch.float64, 1e-12), (torch.float32, 9 * 2.0**-24)):
                X = torch.randn(op.n * m + off, dtype=dt, device="cuda")[off:].view(op.n, m)
                Y = torch.empty(op.n * m + off, dtype=dt, device="cuda")[off:].view(op.n, m)
                ens.gspmv(A, X, Y)
                ref = op if dt == torch.float64 else gen.Operator(op.name, op.shape, op.bcs, op.row_ptr, op.col_idx, op.val.astype(np.float32).astype(np.float64), False)
                _check(ref, X.cpu().numpy(), Y.cpu().numpy(), tol)


@pytest.mark.parametrize("m", [3, 8])
def test_ranges(ens, m):
    """Zeros, values below and above the split range, and sums beyond float go to native products."""
    op = _op("channel64x40x32")
    X = gen.rhs_normal(op.n, m, 7)
    X[::97, 0] = 0.0
    X[::89, 1] = 1e-30
    X[::83, 2] = 3e27
    X[::79, 1] = -1e280
    X[:, m - 1] *= 1e-19
    big = gen.Operator(op.name, op.shape, op.bcs, op.row_ptr, op.col_idx, op.val * 1e12, op.singular)
    for o in (op, big):
        with ens.Matrix.from_operator(o) as A:
            _check(o, X, ens.gspmv(A, torch.from_numpy(X).cuda()).cpu().numpy())
            Z = ens.gspmv(A, torch.zeros(op.n, m, dtype=torch.float64, device="cuda"))
            assert not Z.any()
            one = torch.ones(op.n, m, dtype=torch.float64, device="cuda")
            _check(o, one.cpu().numpy(), ens.gspmv(A, one).cpu().numpy())


@pytest.mark.parametrize("ex", [-71, -57, -41, -40, -39])
def test_smallest_products(ens, ex):
    """Matrix values at the bottom of the split range (2^-40) times values around the bottom of X's window: the
    error terms of the products must not fall below the smallest floats."""
    op = _op("dirichlet41")
    val = np.ldexp(op.val / np.abs(op.val).min(), -40)
    op = gen.Operator(op.name, op.shape, op.bcs, op.row_ptr, op.col_idx, val, False)
    X = np.ldexp(1.0 + np.random.default_rng(3).random((op.n, 8)), ex) * np.where(np.arange(op.n)[:, None] % 3 == 0, -1.0, 1.0)
    with ens.Matrix.from_operator(op) as A:
        _check(op, X, ens.gspmv(A, torch.from_numpy(X).cuda()).cpu().numpy())


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


@pytest.mark.parametrize("m,most", [(8, 4.1), (16, 4.5)])
def test_small_values_cost(ens, m, most):
    """A block whose values all lie below the split range goes to native products, two columns per access: 3.5 and 3.7
    times the time of one inside it (one column per access 4.6 and 5.7)."""
    op = gen.channel(128, 128, 128)
    X = torch.randn(op.n, m, dtype=torch.float64, device="cuda")
    T, Y = X * 1e-30, torch.empty_like(X)
    with ens.Matrix.from_operator(op) as A:
        assert _us(lambda: ens.gspmv(A, T, Y)) <= most * _us(lambda: ens.gspmv(A, X, Y))


@pytest.mark.parametrize("dims,dt,m,off", [((128, 128, 128), "float32", 16, 2), ((128, 128, 128), "float64", 32, 2), ((64, 40, 44), "float64", 64, 0)])
def test_not_slower_than_rows(ens, dims, dt, m, off):
    """Blocks whose rows are aligned to less than the boxes' widest access, and boxes whose last round is nearly empty:
    the product is the row-by-row one, which a forced traversal also runs (by boxes 1.37, 1.18 and 1.19 times)."""
    op = gen.channel(*dims)
    dt = getattr(torch, dt)
    with ens.Matrix.from_operator(op) as A, ens.Matrix.from_operator(op) as R:
        R.set_untiled(0)
        X, Y = (torch.randn(op.n * m + off, dtype=dt, device="cuda")[off:].view(op.n, m) for _ in range(2))
        t = [_us(lambda: ens.gspmv(M, X, Y), 21) for M in (A, R)]
    assert t[0] <= 1.1 * t[1], t


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_nonfinite(ens, dtype):
    """Infinities and NaN reach exactly the rows whose entries name them, as in the definition."""
    op = _op("cubes97x43x37")
    m = 8
    X = gen.rhs_normal(op.n, m, 8).astype(dtype)
    X[1000, 1], X[2000, 2], X[3000, 3] = np.nan, np.inf, -np.inf
    with ens.Matrix.from_operator(op) as A:
        Y = ens.gspmv(A, torch.from_numpy(X).cuda()).cpu().numpy().astype(np.float64)
    ref = oracle.gspmv(op, X.astype(np.float64))
    assert np.array_equal(np.isnan(Y), np.isnan(ref))
    assert np.array_equal(Y[np.isinf(ref)], ref[np.isinf(ref)])
    assert np.array_equal(np.isfinite(Y), np.isfinite(ref))


def test_repeatable(ens):
    op = _op("dirichlet41")
    X = torch.from_numpy(gen.rhs_normal(op.n, 8, 5)).cuda()
    with ens.Matrix.from_operator(op) as A:
        Y = ens.gspmv(A, X)
        assert all(torch.equal(Y, ens.gspmv(A, X)) for _ in range(3))


def test_threads_with_rows_of_different_lengths(ens):
    """Two threads multiply with matrices whose boxes need different amounts of shared memory."""
    import threading

    ops = [_stencil9(301, 257), _stencil9(301, 257, 5)]
    X = gen.rhs_normal(ops[0].n, 8, 4)
    bad = []

    def work(op):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s), ens.Matrix.from_operator(op) as A:
                x = torch.from_numpy(X).cuda()
                want = ens.gspmv(A, x)
                for _ in range(300):
                    if not torch.equal(ens.gspmv(A, x), want):
                        bad.append(op.name)
                _check(op, X, want.cpu().numpy())
        except Exception as e:  # noqa: BLE001
            bad.append(e)

    ts = [threading.Thread(target=work, args=(op,)) for op in ops]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad


@pytest.mark.parametrize("name", ["cubes97x43x37", "channel64x40x44"])
@pytest.mark.parametrize("dt,m,off", [("float64", 16, 2), ("float64", 28, 0), ("float64", 56, 2), ("float64", 64, 0), ("float32", 4, 0),
                                      ("float32", 14, 0), ("float32", 16, 2), ("float32", 24, 4), ("float32", 24, 1)])
def test_products_at_the_line_between_both_forms(ens, name, dt, m, off):
    """Widths, alignments and sizes on either side of the choice between row boxes and rows."""
    op = _op(name) if name in OPS else gen.channel(64, 40, 44)
    dt = getattr(torch, dt)
    ref = op if dt == torch.float64 else gen.Operator(op.name, op.shape, op.bcs, op.row_ptr, op.col_idx, op.val.astype(np.float32).astype(np.float64), False)
    X, Y = (torch.randn(op.n * m + off, dtype=dt, device="cuda")[off:].view(op.n, m) for _ in range(2))
    with ens.Matrix.from_operator(op) as A:
        ens.gspmv(A, X, Y)
    _check(ref, X.cpu().numpy(), Y.cpu().numpy(), 1e-12 if dt == torch.float64 else 9 * 2.0**-24)


@pytest.mark.parametrize("m,dtype", [(2, "f64"), (8, "f64"), (16, "f32"), (32, "f32")])
def test_tuned_variant_is_the_launch_in_use(ens, m, dtype):
    """ens_tuned_variant reports the share that ens_autotune returned and tells row boxes from the two traversals."""
    import ctypes

    from paper_1711_10622_gb300 import _native as N

    with ens.Matrix.from_operator(gen.channel(128, 64, 64)) as A:
        def variant():
            v = [ctypes.c_int32() for _ in range(3)]
            N.check(N.lib().ens_tuned_variant(A.handle, m, 1 if dtype == "f32" else 0, *(ctypes.byref(x) for x in v)))
            return [x.value for x in v]

        assert variant()[0] == -1 and variant()[2] == -1
        t = A.autotune(m, dtype)
        assert variant() == [t["lanes"], t["share"], 2 if t["boxes"] else int(t["untiled"])]
        if m in (2, 32):
            assert not t["boxes"]
        if m == 8:  # 0.7 times the fastest row-by-row launch
            assert t["boxes"] and t["share"] == 0
        A.set_untiled(0)
        assert variant()[2] in (0, 1)
