"""The work that a user of this library has it do, as cases that can be timed and compared.

The library solves the pressure-Poisson equation for m flow states that share one matrix, so the cases are
its products, its preconditioner, its solves and the projection step around a solve, on the operators of
the workloads: a Dirichlet box, a plane channel with wall-normal stretching and a channel with wall-mounted
cubes (gen/workloads.py), from the smallest boxes to the full-size channel and cube grids, with odd and
ragged sizes among them. Right-hand sides and blocks are drawn from the seed on the GPU.
"""

import functools

import numpy as np
import torch

import gen
import paper_1711_10622_gb300 as ens


def listed():
    return [
        # one product on the smallest workload: the launch and the call itself are what counts
        dict(name="product_box32_m4", kind="product", grid="box", nx=32, ny=32, nz=32, m=4, dtype="f64", tuned=False),
        # one flow state on the full-size channel, tuned once as a program that keeps one matrix does
        dict(name="product_channel_m1", kind="product", grid="channel", nx=256, ny=128, nz=128, m=1, dtype="f64", tuned=True),
        # the ordinary ensemble on the irregular operator, as the solver multiplies: not tuned
        dict(name="product_cubes_m8", kind="product", grid="cubes", nx=192, ny=128, nz=96, m=8, dtype="f64", tuned=False),
        # the widest ensemble of the product sweep on the full-size channel
        dict(name="product_channel_m32", kind="product", grid="channel", nx=256, ny=128, nz=128, m=32, dtype="f64", tuned=True),
        # odd sizes in every direction and an odd number of states
        dict(name="product_odd_m5", kind="product", grid="channel", nx=101, ny=67, nz=83, m=5, dtype="f64", tuned=False),
        # the inner product of the mixed-precision solves
        dict(name="product_f32_m16", kind="product", grid="channel", nx=256, ny=128, nz=128, m=16, dtype="f32", tuned=False),
        # the projection step on either side of the solve: right-hand sides, then the velocity correction
        dict(name="projection_m8", kind="projection", grid="channel", nx=128, ny=128, nz=128, m=8, dtype="f64"),
        # one multigrid V-cycle in float32, the preconditioner of the mixed-precision solves
        dict(name="vcycle_f32_m8", kind="vcycle", grid="cubes", nx=96, ny=96, nz=96, m=8, dtype="f32"),
        # a small plain solve: every kernel is short, so launches and gaps weigh most
        dict(name="solve_box32_m4", kind="solve", grid="box", nx=32, ny=32, nz=32, m=4, precond="none", precision="f64", tol=1e-12, max_iter=1000),
        # the ensemble solve in float64 with the Chebyshev preconditioner, a fixed number of iterations
        # per time step, as the paper runs its solver
        dict(name="solve_cubes_cheb_m8", kind="solve", grid="cubes", nx=192, ny=128, nz=96, m=8, precond="chebyshev", precision="f64", tol=0.0, max_iter=10),
        # what the server runs: float32 inner solves with the V-cycle, refined in float64
        dict(name="solve_mixed_amg_m8", kind="solve", grid="channel", nx=96, ny=96, nz=96, m=8, precond="amg", precision="mixed", tol=1e-11, max_iter=1000),
        # several systems of uneven size and width in one launch
        dict(name="batch_mixed_amg", kind="batch", nx=64, ny=48, nz=40, m=4, nx2=45, ny2=33, nz2=51, m2=16, nx3=96, ny3=64, nz3=48, m3=8, tol=1e-11),
    ]


def _loguniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """Products of every width, type and operator; now and then a projection, a V-cycle, a solve or a batch."""
    kind = rng.choice(["product"] * 6 + ["projection", "vcycle", "solve", "solve", "batch"])
    grid = rng.choice(["box", "channel", "channel", "cubes"])
    top = {"product": 256, "projection": 128, "vcycle": 96, "solve": 96, "batch": 64}[kind]
    nx, ny, nz = _loguniform(rng, 24, top), _loguniform(rng, 24, min(top, 128)), _loguniform(rng, 24, min(top, 128))
    if kind == "product":
        dtype = rng.choice(["f64", "f64", "f32"])
        return dict(kind=kind, grid=grid, nx=nx, ny=ny, nz=nz, m=rng.choice([1, 2, 3, 4, 6, 7, 8, 8, 12, 16, 16, 20, 24, 32]), dtype=dtype, tuned=rng.random() < 0.3)
    if kind == "projection":
        return dict(kind=kind, grid="channel", nx=nx, ny=ny, nz=nz, m=rng.choice([1, 2, 4, 5, 8]), dtype="f64")
    if kind == "vcycle":
        return dict(kind=kind, grid=grid, nx=nx, ny=ny, nz=nz, m=rng.choice([1, 2, 4, 6, 8]), dtype=rng.choice(["f32", "f32", "f64"]))
    if kind == "solve":
        precision = rng.choice(["f64", "mixed"])
        precond = rng.choice(["chebyshev", "amg"])
        m = rng.choice([1, 2, 4, 5, 8])
        if precision == "f64":
            return dict(kind=kind, grid=grid, nx=nx, ny=ny, nz=nz, m=m, precond=precond, precision=precision, tol=0.0, max_iter=10)
        return dict(kind=kind, grid="channel", nx=nx, ny=ny, nz=nz, m=m, precond=precond, precision=precision, tol=1e-11, max_iter=1000)
    s = [_loguniform(rng, 24, 64) for _ in range(9)]
    return dict(kind=kind, nx=s[0], ny=s[1], nz=s[2], m=rng.choice([1, 4, 8]), nx2=s[3], ny2=s[4], nz2=s[5], m2=rng.choice([2, 8, 16]),
                nx3=s[6], ny3=s[7], nz3=s[8], m3=rng.choice([3, 4, 8]), tol=1e-11)


# The grids do not depend on the seed: an application assembles its operator once on the host.
@functools.lru_cache(maxsize=16)
def _operator(grid, nx, ny, nz):
    if grid == "box":
        return gen.dirichlet_box(nx, nz=nz, ny=ny)
    if grid == "channel":
        return gen.channel(nx, ny, nz)
    return gen.cubes(nx, ny, nz, size=min(nx // 6, ny // 2, nz // 6))


def _op(case):
    return _operator(case["grid"], case["nx"], case["ny"], case["nz"])


def _systems(case):
    """The three systems of a batch: (operator, width)."""
    return [(_operator("channel", case["nx" + k], case["ny" + k], case["nz" + k]), case["m" + k]) for k in ("", "2", "3")]


def _normal(g, rows, m, dtype=torch.float64):
    return torch.randn(rows, m, generator=g, device="cuda", dtype=torch.float64).to(dtype)


def _rhs(g, op, m):
    """Right-hand sides: N(0, 1), without the part that a singular operator cannot reach."""
    B = _normal(g, op.n, m)
    return B - B.mean(dim=0, keepdim=True) if op.singular else B


def _velocity(g, case):
    """m staggered velocity fields of the channel: a parabolic profile and perturbations, zero on the walls."""
    nx, ny, nz, m = case["nx"], case["ny"], case["nz"], case["m"]
    y = torch.as_tensor(_op(case).meta["nodes"][1], device="cuda", dtype=torch.float64)
    prof = 1.5 * (1.0 - (0.5 * (y[1:] + y[:-1])) ** 2)
    U = 0.05 * _normal(g, nz * ny * nx, m).view(nz, ny, nx, m) + prof.view(1, ny, 1, 1)
    V = 0.05 * _normal(g, nz * (ny + 1) * nx, m).view(nz, ny + 1, nx, m)
    V[:, 0] = 0.0
    V[:, ny] = 0.0
    W = 0.05 * _normal(g, nz * ny * nx, m)
    return U.reshape(-1, m).contiguous(), V.reshape(-1, m).contiguous(), W


TAU = 1e-3


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    state = {"kind": kind, "case": case}
    if kind == "batch":
        state["systems"] = []
        for op, m in _systems(case):
            A = ens.Matrix.from_operator(op)
            A.amg_setup()
            state["systems"].append((A, _rhs(g, op, m), None, case["tol"]))
        return state
    op = _op(case)
    if kind == "projection":
        state["grid"] = ens.Grid.from_grid(gen.grid_of(op))
        state["velocity"] = _velocity(g, case)
        state["pressure"] = _normal(g, op.n, case["m"])
        state["D"] = torch.empty(op.n, case["m"], dtype=torch.float64, device="cuda")
        return state
    state["A"] = A = ens.Matrix.from_operator(op)
    if kind == "solve":
        if case["precond"] == "amg":
            A.amg_setup()
        state["B"] = _rhs(g, op, case["m"])
        return state
    if kind == "vcycle":
        A.amg_setup()
    elif case["tuned"]:
        A.autotune(case["m"], case["dtype"])
    state["X"] = _normal(g, op.n, case["m"], torch.float64 if case["dtype"] == "f64" else torch.float32)
    state["Y"] = torch.empty_like(state["X"])
    return state


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "product":
        return ens.gspmv(state["A"], state["X"], state["Y"])
    if kind == "vcycle":
        return ens.amg_apply(state["A"], state["X"], state["Y"])
    if kind == "projection":
        U, V, W = state["velocity"]
        D = ens.divergence(state["grid"], U, V, W, scale=-1.0 / TAU, D=state["D"])
        ens.grad_correct(state["grid"], state["pressure"], U, V, W, tau=TAU)
        return D, U, V, W
    # Solutions and statuses. The iteration counts and final residuals that come beside them describe
    # the path a solve took and not its result.
    if kind == "solve":
        opts = dict(precond=case["precond"], precision=case["precision"])
        if case["precision"] == "f64":
            opts["max_iter"] = case["max_iter"]
        X, stats = ens.solve_block(state["A"], state["B"], tol=case["tol"], **opts)
        return X, stats["status"]
    out = ens.solve_batch(state["systems"], precond="amg", precision="mixed", x0_zero=True)
    return [(X, stats["status"]) for X, stats in out]


def _product_work(n, nnz, m, size):
    return {"bytes": 4 * (n + 1) + (4 + size) * nnz + 2 * size * m * n, "flops": 2 * nnz * m}


def _solve_work(n, nnz, m, iterations, products):
    """A solve reads the matrix and the right-hand sides and writes the solutions; each iteration multiplies
    `products` times and updates and reduces about ten blocks."""
    return {"bytes": 4 * (n + 1) + 12 * nnz + 16 * m * n, "flops": iterations * (2 * nnz * m * products + 20 * n * m)}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_solve_work(op.n, op.nnz, m, 20, 10) for op, m in _systems(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    op, m = _op(case), case["m"]
    if kind == "product":
        return _product_work(op.n, op.nnz, m, 8 if case["dtype"] == "f64" else 4)
    if kind == "projection":
        # divergence: three components in, one block out; correction: the pressure in, three components in and out
        faces = case["nx"] * case["nz"] * (3 * case["ny"] + 1)
        return {"bytes": 8 * m * (faces + op.n) + 8 * m * (2 * faces + op.n), "flops": m * (7 * op.n + 9 * op.n)}
    if kind == "vcycle":
        # four products on the fine level (two smoothings, two residuals), one block in and one out
        w = _product_work(op.n, op.nnz, m, 8 if case["dtype"] == "f64" else 4)
        return {"bytes": w["bytes"], "flops": 4 * w["flops"]}
    if case["precision"] == "f64":
        iterations = min(case["max_iter"], 100)
    else:
        iterations = 40 if case["precond"] == "amg" else 120
    return _solve_work(op.n, op.nnz, m, iterations, {"none": 2, "chebyshev": 8, "amg": 10}[case["precond"]])


def _poisson_direct(op, B):
    """A x = b by separation of variables: on these grids A is a sum of one 1D operator in one direction and
    the cell widths in the other two, so the 1D eigenvectors (symmetrically scaled by the widths) solve it."""
    dims, lam, vec, root = op.shape, [], [], []
    for N, nodes, bc in zip(dims, op.meta["nodes"], op.bcs):
        w = np.diff(nodes)
        c = 0.5 * (nodes[1:] + nodes[:-1])
        K = np.zeros((N, N))
        for i in range(N - 1):
            a = 1.0 / (c[i + 1] - c[i])
            K[i, i] += a
            K[i + 1, i + 1] += a
            K[i, i + 1] -= a
            K[i + 1, i] -= a
        if bc == "periodic":
            a = 1.0 / (c[0] + nodes[-1] - nodes[0] - c[-1])
            K[0, 0] += a
            K[-1, -1] += a
            K[0, -1] -= a
            K[-1, 0] -= a
        elif bc == "dirichlet":
            K[0, 0] += 2.0 / w[0]
            K[-1, -1] += 2.0 / w[-1]
        s = np.sqrt(w)
        ev, Q = np.linalg.eigh(K / s[:, None] / s[None, :])
        if op.singular:
            ev[0] = 0.0
        lam.append(torch.as_tensor(ev, device="cuda"))
        vec.append(torch.as_tensor(Q, device="cuda"))
        root.append(torch.as_tensor(s, device="cuda"))
    nx, ny, nz = dims
    scale = (root[2].view(nz, 1, 1, 1) * root[1].view(1, ny, 1, 1)) * root[0].view(1, 1, nx, 1)
    T = B.view(nz, ny, nx, -1) / scale
    T = torch.einsum("zyxm,xa->zyam", T, vec[0])
    T = torch.einsum("zyxm,ya->zaxm", T, vec[1])
    T = torch.einsum("zyxm,za->ayxm", T, vec[2])
    total = lam[2].view(nz, 1, 1, 1) + lam[1].view(1, ny, 1, 1) + lam[0].view(1, 1, nx, 1)
    T = torch.where(total.abs() > 0, T / torch.where(total.abs() > 0, total, torch.ones_like(total)), torch.zeros_like(T))
    T = torch.einsum("zyxm,az->ayxm", T, vec[2])
    T = torch.einsum("zyxm,ay->zaxm", T, vec[1])
    T = torch.einsum("zyxm,ax->zyam", T, vec[0])
    X = (T / scale).reshape(op.n, -1)
    return X - X.mean(dim=0, keepdim=True) if op.singular else X


def _multiply(op, X):
    """Y = A X in float64, 64 MB of products at a time."""
    m = X.shape[1]
    Y = torch.empty_like(X)
    rp = op.row_ptr.astype(np.int64)
    step = max(1, (1 << 23) // (7 * m))
    val, col = torch.as_tensor(op.val, device="cuda"), torch.as_tensor(op.col_idx, device="cuda").long()
    lens = torch.as_tensor(np.diff(rp), device="cuda")
    for r in range(0, op.n, step):
        e = min(op.n, r + step)
        a, b = int(rp[r]), int(rp[e])
        P = val[a:b, None] * X[col[a:b]]
        Y[r:e] = torch.segment_reduce(P, "sum", lengths=lens[r:e], axis=0)
    return Y


def exact(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    if kind == "batch":
        out = []
        for op, m in _systems(case):
            out.append((_poisson_direct(op, _rhs(g, op, m)), None))
        return out
    if kind == "vcycle" or (kind == "solve" and (case["precision"] == "f64" and case["tol"] == 0.0)):
        return None  # a fixed number of steps of an iteration
    op, m = _op(case), case["m"]
    if kind == "product":
        return _multiply(op, _normal(g, op.n, m, torch.float64 if case["dtype"] == "f64" else torch.float32).double())
    if kind == "projection":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        U, V, W = (t.view(nz, -1, nx, m) for t in _velocity(g, case))
        P = _normal(g, op.n, m).view(nz, ny, nx, m)
        nodes = [torch.as_tensor(a, device="cuda") for a in op.meta["nodes"]]
        wx, wy, wz = (torch.diff(a) for a in nodes)
        cx, cy, cz = (0.5 * (a[1:] + a[:-1]) for a in nodes)
        ax, ay, az = wz.view(nz, 1, 1, 1) * wy.view(1, ny, 1, 1), wz.view(nz, 1, 1, 1) * wx.view(1, 1, nx, 1), wy.view(1, ny, 1, 1) * wx.view(1, 1, nx, 1)
        D = ax * (torch.roll(U, -1, 2) - U) + ay * (V[:, 1:] - V[:, :-1]) + az * (torch.roll(W, -1, 0) - W)

        def gaps(c, nd):
            return torch.cat([(c[0] + nd[-1] - nd[0] - c[-1]).view(1), torch.diff(c)])

        U = U - TAU * (P - torch.roll(P, 1, 2)) / gaps(cx, nodes[0]).view(1, 1, nx, 1)
        W = W - TAU * (P - torch.roll(P, 1, 0)) / gaps(cz, nodes[2]).view(nz, 1, 1, 1)
        V = V.clone()
        V[:, 1:-1] -= TAU * (P[:, 1:] - P[:, :-1]) / torch.diff(cy).view(1, ny - 1, 1, 1)
        return tuple(t.reshape(-1, m) for t in (-D / TAU, U, V, W))
    return _poisson_direct(op, _rhs(g, op, m)), None
