"""Timed cases of the solver: the calls that a program makes through the
package's public entry points, over the sizes that its configurations, tests
and benchmark use.

  product  u = M lambda on device arrays (am_rpy_matvec), or a range of its
           rows against all sources (am_rpy_matvec_rows), in free space or
           above a wall, FP64 or mixed
  solve    the constrained mobility problem of a suspension at its current
           pose (am_solve: preconditioner build, GMRES from a cold start)
  step     one Euler step of a time loop (am_solve_step), the next pose
           read back
  network  loss and gradient of the initial-guess network over a set of
           samples (am_mlp_loss_grad)

Solves and steps run to relative residual 1e-10, the binding's default.
"""
import math

import numpy as np
import torch

from paper_2107_10800_gb300 import binding, workloads

DT = 1e-3
LAYERS = (144, 256, 256, 256, 32)


def listed():
    return [
        # the smallest call: one product on the blobs of four 8-body chains
        # (the settling-filament size), launch latency included
        dict(name="product_free_f64_384", path="product", n=384, rows=0, wall=False, mixed=False),
        # one product on the blobs of the diatom colony, the benchmark's size
        dict(name="product_wall_f64_2560", path="product", n=2560, rows=0, wall=True, mixed=False),
        # the mixed product of a large wall suspension
        dict(name="product_wall_mixed_60000", path="product", n=60000, rows=0, wall=True, mixed=True),
        # one rank's rows of a suspension sharded over four GPUs, ragged sizes
        dict(name="rows_free_f64_20011", path="product", n=20011, rows=5003, wall=False, mixed=False),
        # one time step of 4 free chains of 8 twelve-blob bodies, in a time
        # loop (each solve starts from the one before)
        dict(name="step_chains_f64", path="step", kind="chains", chains=4, bodies=8, mixed=False),
        # the benchmark's colony above a wall, solved at its pose
        dict(name="solve_colony_f64", path="solve", kind="colony", rods=32, nx=40, mixed=False),
        # the same in mixed precision
        dict(name="solve_colony_mixed", path="solve", kind="colony", rods=32, nx=40, mixed=True),
        # a suspension of 100 bacteria above a wall (36,000 blobs, bodies of
        # 200 and of 10 blobs)
        dict(name="solve_bacteria_mixed", path="solve", kind="bacteria", count=100, mixed=True),
        # many independent small suspensions in one handle
        dict(name="solve_batched_mixed", path="solve", kind="batched", systems=16, lo=500, hi=4000, mixed=True),
        # bacteria in a triply periodic box (77,760 blobs), spectral Ewald product
        dict(name="solve_periodic_f64", path="solve", kind="periodic", nx=6, ny=6, nz=6, mixed=False),
        # filaments of single spheres with rotational coupling (52,800 unknowns)
        dict(name="solve_spheres_f64", path="solve", kind="spheres", chains=400, bodies=15, mixed=False),
        # training of the initial-guess network: loss and gradient of 4,096 samples
        dict(name="network_gradient_4096", path="network", samples=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["product", "product", "rows", "chains", "colony", "bacteria", "batched", "periodic", "spheres",
                       "network"])
    mixed = rng.random() < 0.5
    if what == "product":
        n = _log_int(rng, 200, 60000 if mixed else 12000)
        return dict(path="product", n=n, rows=0, wall=rng.random() < 0.5, mixed=mixed)
    if what == "rows":
        n = _log_int(rng, 1000, 60000 if mixed else 20000)
        return dict(path="product", n=n, rows=max(1, n // rng.randint(2, 8)), wall=rng.random() < 0.5, mixed=mixed)
    if what == "chains":
        return dict(path=rng.choice(["step", "solve"]), kind="chains", chains=_log_int(rng, 2, 40),
                    bodies=rng.randint(2, 15), mixed=mixed)
    if what == "colony":
        return dict(path="solve", kind="colony", rods=rng.randint(3, 32), nx=rng.randint(9, 40), mixed=mixed)
    if what == "bacteria":
        return dict(path="solve", kind="bacteria", count=_log_int(rng, 3, 100), mixed=True)
    if what == "batched":
        return dict(path="solve", kind="batched", systems=rng.randint(3, 16), lo=300, hi=rng.randint(900, 4000),
                    mixed=True)
    if what == "periodic":
        return dict(path="solve", kind="periodic", nx=rng.randint(2, 4), ny=rng.randint(3, 6), nz=rng.randint(3, 6),
                    mixed=mixed)
    if what == "spheres":
        return dict(path="solve", kind="spheres", chains=_log_int(rng, 20, 400), bodies=rng.randint(5, 15),
                    mixed=False)
    return dict(path="network", samples=_log_int(rng, 100, 4096))


def _blobs(case, seed):
    return workloads.random_blobs(seed, case["n"], a=0.1, wall=1 if case["wall"] else 0)


def _suspensions(case, seed):
    """The workload dicts of a case, one per system of its handle."""
    kind = case["kind"]
    if kind == "chains":
        box = 10.0 * (case["chains"] * case["bodies"] / 32.0) ** (1.0 / 3.0)
        return [workloads.chains_free_space(seed, n_chains=case["chains"], bodies_per_chain=case["bodies"], box=box)]
    if kind == "colony":
        return [workloads.diatom_colony(seed, n_rods=case["rods"], nx=case["nx"])]
    if kind == "bacteria":  # at the lateral density of 1,000 in a square of 250
        return [workloads.bacteria_wall(seed, n_bact=case["count"], box=250.0 * math.sqrt(case["count"] / 1000.0))]
    if kind == "batched":  # blob counts spread over [lo, hi] on a log scale, whole chains of 8 bodies
        return [workloads.chains_free_space(seed * 1009 + k, n_chains=c, box=10.0 * (c / 4.0) ** (1.0 / 3.0))
                for k, c in enumerate(_batch(case))]
    if kind == "periodic":
        return [workloads.bacteria_periodic(seed, lattice=(case["nx"], case["ny"], case["nz"]))]
    box = 10.0 * (case["chains"] * case["bodies"] / 60.0) ** (1.0 / 3.0)
    w = workloads.chains_free_space(seed, n_chains=case["chains"], bodies_per_chain=case["bodies"], box=box)
    return [dict(w, a=0.5)]


def _batch(case):
    """Chains of 8 twelve-blob bodies in each system of a batch."""
    s, ratio = case["systems"], case["hi"] / case["lo"]
    return [max(1, round(case["lo"] * ratio ** ((k + 0.5) / s) / 96)) for k in range(s)]


def _network(seed):
    """He-initialised parameters in the library's flat order W1, b1, ..., W4, b4."""
    rng = np.random.default_rng(seed)
    flat = []
    for k, m in zip(LAYERS[:-1], LAYERS[1:]):
        flat += [rng.standard_normal(m * k) * math.sqrt(2.0 / k), 0.1 * rng.standard_normal(m)]
    return np.concatenate(flat).astype(np.float32)


def _samples(case, seed):
    rng = np.random.default_rng(seed + 1)
    n = case["samples"]
    return (rng.standard_normal((n, LAYERS[0])).astype(np.float32),
            rng.standard_normal((n, LAYERS[-1])).astype(np.float32))


def prepare(case, seed):
    if case["path"] == "product":
        r, lam = _blobs(case, seed)
        prec = "mixed" if case["mixed"] else "fp64"
        n, rows = case["n"], case["rows"]
        if rows:
            work = binding.rpy_matvec_rows_workspace(n, rows, prec)
        else:
            work = binding.rpy_matvec_workspace(n, prec)
        dev = torch.device("cuda")
        return dict(case=case, prec=prec, r=torch.tensor(r, device=dev), lam=torch.tensor(lam, device=dev),
                    u=torch.empty((rows or n, 3), dtype=torch.float64, device=dev),
                    work=torch.empty(work, dtype=torch.uint8, device=dev), row0=(n - rows) // 2 if rows else 0)
    if case["path"] == "network":
        net = binding.Mlp()
        net.set_params(_network(seed))
        X, T = _samples(case, seed)
        return dict(case=case, net=net, X=X, T=T)
    ws = _suspensions(case, seed)
    kw = dict(precision="mixed" if case["mixed"] else "fp64", tol=1e-10, max_iter=2000)
    if case["kind"] == "batched":
        solver = binding.Solver.from_workloads(ws, **kw)
    elif case["kind"] == "spheres":
        solver = binding.Solver.from_workload(ws[0], single_blob=True, **kw)
    else:
        solver = binding.Solver.from_workload(ws[0], **kw)
    return dict(case=case, solver=solver, step=0)


def run(state):
    case = state["case"]
    if case["path"] == "product":
        n, rows, wall = case["n"], case["rows"], 1 if case["wall"] else 0
        work, stream = state["work"], torch.cuda.current_stream().cuda_stream
        ptr = (state["r"].data_ptr(), state["lam"].data_ptr(), state["u"].data_ptr())
        if rows:
            binding.rpy_matvec_rows_ptr(*ptr, n, state["row0"], rows, 1.0, 0.1, wall, state["prec"], work.data_ptr(),
                                        work.numel(), stream)
        else:
            binding.rpy_matvec_ptr(*ptr, n, 1.0, 0.1, wall, state["prec"], work.data_ptr(), work.numel(), stream)
        return state["u"]
    if case["path"] == "network":
        loss, grad = state["net"].loss_grad(state["X"], state["T"])
        return dict(loss=loss, grad=grad)
    solver = state["solver"]
    if case["path"] == "step":  # passive links: a step of the time loop
        U, phi, lam, _ = solver.step(state["step"] * DT, DT)
        q, theta = solver.bodies()
        state["step"] += 1
        return dict(U=U, phi=phi, lam=lam, q=q, theta=theta)
    U, phi, lam, _ = solver.solve()
    if case["kind"] == "spheres":
        return dict(U=U, phi=phi)
    # Two links between the same two bodies are redundant: their forces are
    # determined only up to null(C^T), everything else is unique
    if case["kind"] in ("colony", "bacteria", "periodic"):
        return dict(U=U, lam=lam)
    return dict(U=U, phi=phi, lam=lam)


def _pair_flops(wall):
    """Per unordered pair, both directions (the mobility is symmetric): the
    pair's coefficients once, applied to two forces."""
    return 126 if wall else 53


def work(case):
    if case["path"] == "product":
        n, rows = case["n"], case["rows"]
        if rows:  # rows x n pairs, rows x rows of them in both directions
            one = 119 if case["wall"] else 35
            flops = rows * (n - rows) * one + 0.5 * rows * rows * _pair_flops(case["wall"])
            return {"bytes": 48.0 * n + 24.0 * rows, "flops": float(flops)}
        return {"bytes": 72.0 * n, "flops": 0.5 * n * n * _pair_flops(case["wall"])}
    if case["path"] == "network":
        n = case["samples"]
        weights = sum(k * m for k, m in zip(LAYERS[:-1], LAYERS[1:]))
        return {"bytes": 4.0 * (n * (LAYERS[0] + LAYERS[-1]) + 2 * weights), "flops": 6.0 * n * weights}
    # A solve reads its bodies and writes its solution; its operations are
    # those of 20 products, fewer than any of these takes, and of the
    # body blocks' factorisations ((3n)^3 / 3 multiply-adds each).
    if case["kind"] == "colony":
        nbs, bodies, wall = [2 * case["nx"] * case["rods"]], [2 * case["nx"]] * case["rods"], True
    elif case["kind"] == "bacteria":
        nbs, bodies, wall = [360 * case["count"]], ([200] + [10] * 16) * case["count"], True
    elif case["kind"] == "periodic":
        count = case["nx"] * case["ny"] * case["nz"]
        # about 60 pairs within the cutoff and a 12-point window per blob
        near = 360.0 * count * (60 * 30 + 2 * 3 * 12 ** 3 * 2)
        return {"bytes": 360.0 * count * 96, "flops": 20 * near + 2 / 3 * count * (600.0 ** 3 + 16 * 30.0 ** 3)}
    elif case["kind"] == "batched":
        nbs, bodies, wall = [96 * c for c in _batch(case)], [12] * (8 * sum(_batch(case))), False
    elif case["kind"] == "spheres":
        m = case["chains"] * case["bodies"]
        return {"bytes": m * 200.0, "flops": 20 * 0.5 * m * m * 180}
    else:
        m = case["chains"] * case["bodies"]
        nbs, bodies, wall = [12 * m], [12] * m, False
    flops = sum(20 * 0.5 * n * n * _pair_flops(wall) for n in nbs) + sum(2 / 3 * (3.0 * b) ** 3 for b in bodies)
    return {"bytes": sum(96.0 * n for n in nbs) + 150.0 * len(bodies), "flops": flops}


# ---- what the outputs are, in 64 bits, by plain torch ----------------------


def _mobility(x, y, a, eta, wall):
    """The 3 x 3 blocks (len(x), 3, len(y), 3) of the blob mobility: the
    Rotne-Prager-Yamakawa tensor, with a wall the image part as well."""
    d = x[:, None] - y[None]
    r = d.norm(dim=-1)
    safe = r.clamp_min(1e-300)
    far = r >= 2 * a
    pre = 1.0 / (8 * math.pi * eta)
    c1 = torch.where(far, pre / safe * (1 + 2 * a * a / (3 * safe * safe)),
                     (1 - 9 * r / (32 * a)) / (6 * math.pi * eta * a))
    c2 = torch.where(far, pre / safe * (1 - 2 * a * a / (safe * safe)), 3 * r / (32 * a) / (6 * math.pi * eta * a))
    h = d / safe[..., None]
    eye = torch.eye(3, dtype=x.dtype, device=x.device)
    M = c1[..., None, None] * eye + (c2[..., None] * h)[..., :, None] * h[..., None, :]
    if wall:
        R = torch.cat([d[..., :2], (x[:, None, 2] + y[None, :, 2])[..., None]], dim=-1)
        s = 1 / R.norm(dim=-1)
        h = R * s[..., None]
        hs, ez, A = y[None, :, 2] * s, h[..., 2], a * a * s * s
        u = hs * x[:, None, 2] * s
        t1, t2 = A * ez * ez, A * A * ez * ez
        cI = -1 - 2 * u - 2 / 3 * A + 2 * t1 + 2 / 3 * A * A - 10 / 3 * t2
        cRR = -1 + 6 * u + 2 * A - 10 * t1 - 10 / 3 * A * A + 70 / 3 * t2
        cRz = 2 * hs + ez * (-2 * cRR - 2 + 20 / 3 * A * A)
        czR = 2 * hs - 20 / 3 * A * A * ez
        czz = -4 * hs * hs - 4 * t1 - 8 / 3 * A * A + 20 * t2
        W = cI[..., None, None] * eye + (cRR[..., None] * h)[..., :, None] * h[..., None, :]
        W[..., :, 2] += cRz[..., None] * h
        W[..., 2, :] += czR[..., None] * h
        W[..., 2, 2] += czz
        M += (pre * s)[..., None, None] * W
    return M.permute(0, 2, 1, 3)


def _apply(x, y, lam, a, eta, wall):
    step = max(1, 4_000_000 // len(y))
    out = [torch.einsum("iajb,jb->ia", _mobility(x[i:i + step], y, a, eta, wall), lam)
           for i in range(0, len(x), step)]
    return torch.cat(out)


def _rotation(theta):
    s, p = theta[:, 0], theta[:, 1:]
    R = 2 * (p[:, :, None] * p[:, None, :] + s[:, None, None] * _cross(p))
    return R + (2 * s * s - 1)[:, None, None] * torch.eye(3, dtype=theta.dtype, device=theta.device)


def _cross(v):
    z = torch.zeros_like(v[:, 0])
    return torch.stack([z, -v[:, 2], v[:, 1], v[:, 2], z, -v[:, 0], -v[:, 1], v[:, 0], z], dim=1).reshape(-1, 3, 3)


def _solution(w):
    """(U, phi, lambda) of one suspension from dense factorisations:
    N = (K^T M^-1 K)^-1, C N C^T phi = B - C N F (least squares where the
    links are redundant), U = N (F + C^T phi), lambda = M^-1 K U."""
    dev = torch.device("cuda")
    t = lambda v: torch.tensor(np.asarray(v), dtype=torch.float64, device=dev)  # noqa: E731
    q, R, F = t(w["q"]), _rotation(t(w["theta"])), t(w["F"]).reshape(-1)
    off = np.asarray(w["blob_offset"])
    body = torch.tensor(np.repeat(np.arange(len(q)), np.diff(off)), device=dev)
    arm = torch.einsum("iab,ib->ia", R[body], t(w["rho"]))
    r = q[body] + arm
    n, m = len(r), len(q)
    M = torch.empty((n, 3, n, 3), dtype=torch.float64, device=dev)
    step = max(1, 4_000_000 // n)
    for i in range(0, n, step):
        M[i:i + step] = _mobility(r[i:i + step], r, w["a"], w["eta"], w["wall"])
    K = torch.zeros((n, 3, m, 6), dtype=torch.float64, device=dev)
    at = torch.arange(n, device=dev)
    K[at, :, body, :3] = torch.eye(3, dtype=torch.float64, device=dev)
    K[at, :, body, 3:] = -_cross(arm)
    K = K.reshape(3 * n, 6 * m)
    L = torch.linalg.cholesky(M.reshape(3 * n, 3 * n))
    del M
    MK = torch.cholesky_solve(K, L)
    del L
    S = torch.linalg.cholesky(K.T @ MK)
    bp, bq = (torch.tensor(np.asarray(w[k]), device=dev) for k in ("body_p", "body_q"))
    if w.get("dl") is not None:
        dlp, dlq, dlpd, dlqd = (t(v) for v in w["dl"](0.0))
        turn = lambda b, v: torch.einsum("iab,ib->ia", R[b], v)  # noqa: E731
        lp, lq, B = turn(bp, dlp), turn(bq, dlq), turn(bq, dlqd) - turn(bp, dlpd)
    else:
        lp, lq = t(w["joints"]) - q[bp], t(w["joints"]) - q[bq]
        B = torch.zeros_like(lp)
    links = torch.arange(len(bp), device=dev)
    C = torch.zeros((len(bp), 3, m, 6), dtype=torch.float64, device=dev)
    C[links, :, bp, :3] += torch.eye(3, dtype=torch.float64, device=dev)
    C[links, :, bq, :3] -= torch.eye(3, dtype=torch.float64, device=dev)
    C[links, :, bp, 3:] -= _cross(lp)
    C[links, :, bq, 3:] += _cross(lq)
    C = C.reshape(3 * len(bp), 6 * m)
    NC = torch.cholesky_solve(C.T.contiguous(), S)
    NF = torch.cholesky_solve(F[:, None], S)[:, 0]
    val, vec = torch.linalg.eigh(C @ NC)
    keep = val > 1e-11 * val.max()
    c = vec.T @ (B.reshape(-1) - C @ NF)
    phi = vec @ torch.where(keep, c / torch.where(keep, val, 1.0), 0.0)
    U = NF + NC @ phi
    return U.reshape(-1, 6), phi.reshape(-1, 3), (MK @ U).reshape(-1, 3)


def exact(case, seed):
    if case["path"] == "product":
        r, lam = (torch.tensor(v, device="cuda") for v in _blobs(case, seed))
        n, rows = case["n"], case["rows"]
        x = r[(n - rows) // 2:(n - rows) // 2 + rows] if rows else r
        return _apply(x, r, lam, 0.1, 1.0, case["wall"])
    if case["path"] == "network":
        p = torch.tensor(_network(seed).astype(np.float64), device="cuda", requires_grad=True)
        X, T = (torch.tensor(v.astype(np.float64), device="cuda") for v in _samples(case, seed))
        k = 0
        for i, (a, b) in enumerate(zip(LAYERS[:-1], LAYERS[1:])):
            X = X @ p[k:k + a * b].reshape(b, a).T + p[k + a * b:k + a * b + b]
            X = X.relu() if i < 3 else X
            k += a * b + b
        loss = ((X - T) ** 2).mean()
        loss.backward()
        return dict(loss=float(loss.detach()), grad=p.grad)
    if case["kind"] in ("periodic", "spheres") or (case["kind"] == "bacteria" and case["count"] > 30):
        return None
    sols = [_solution(w) for w in _suspensions(case, seed)]
    U, phi, lam = (torch.cat(v) for v in zip(*sols))
    if case["path"] == "step":
        return dict(U=U, phi=phi, lam=lam, q=None, theta=None)
    if case["kind"] in ("colony", "bacteria"):
        return dict(U=U, lam=lam)
    return dict(U=U, phi=phi, lam=lam)
