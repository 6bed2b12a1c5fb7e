"""What a user of the library has it do, as timed cases.

Each case is one call chain through the Python binding: an evaluation of the
advection term (``Rom.nonlinear``), a run of time steps that hands the new
state back (``Trajectories.step_host``), a CP fit (``Als.fit``) or a batch of
serving requests (``Server.serve``).  Sizes are those of the benchmark, its
workloads and the tests: N = 64 ... 1024, ranks up to N, 1 ... 1024
trajectories, all storage types and layouts, odd sizes among them.

Inputs follow the repository's synthetic recipes, drawn on the GPU: skew
tensors (G_ijk - G_kji) / N, CP factors whose columns decay as 1/r, initial
states z_i / i, stiffness diag((i/N)^2), nu = 1e-2, dt = 1e-3.
"""
import math

import numpy as np
import torch

import paper_2311_03694_gb300 as grom

NU, DT = 1e-2, 1e-3
ELEM = {"f64": 8, "f32x2": 8, "f32": 4, "bf16": 2}
ON_CHIP = 128 << 20  # operators above this are read from memory again in every step
SERVED = ((128, 64, "bf16"), (256, 256, "f64"), (512, 256, "bf16"), (1024, 512, "f64"))  # (N, R, storage) of a serving mix


def _full(name, n, storage, layout, batch, steps):
    return {"name": name, "kind": "full", "n": n, "storage": storage, "layout": layout, "batch": batch, "steps": steps}


def _cp(name, n, rank, form, storage, batch, steps):
    return {"name": name, "kind": "cp", "n": n, "rank": rank, "form": form, "storage": storage, "batch": batch,
            "steps": steps}


def listed():
    """steps = 0: one evaluation of the advection term; else that many time steps."""
    return [
        # one right-hand side of a small G-ROM, as an outer integrator asks for it: latency
        _full("full_f64_n64_eval", 64, "f64", "dense", 1, 0),
        # the FP64 G-ROM of the N = 512 workload, one trajectory
        _full("full_f64_n512_step", 512, "f64", "dense", 1, 16),
        # the benchmark's headline: N = 1024 at FP64 tolerance, skew-packed, one trajectory
        _full("full_f32x2_packed_n1024_step", 1024, "f32x2", "skew_packed", 1, 8),
        # right-hand sides of three trajectories at an odd size, FP64 skew-packed
        _full("full_f64_packed_n769_eval", 769, "f64", "skew_packed", 3, 0),
        # ensemble of a mid-size G-ROM, dense BF16 tensor
        _full("full_bf16_n512_b256_step", 512, "bf16", "dense", 256, 4),
        # the largest ensemble: N = 1024, 1024 trajectories, skew-packed BF16 tensor
        _full("full_bf16_packed_n1024_b1024_step", 1024, "bf16", "skew_packed", 1024, 4),
        # long single run of the CPD-ROM
        _cp("cp_skew_bf16_n1024_b1_step", 1024, 1024, "cp_skew", "bf16", 1, 64),
        # one right-hand side of a general CP model, FP64, ragged sizes
        _cp("cp_f64_n500_r129_eval", 500, 129, "cp", "f64", 1, 0),
        # large ensemble of the CPD-ROM, BF16 factors
        _cp("cp_skew_bf16_n1024_b1024_step", 1024, 1024, "cp_skew", "bf16", 1024, 8),
        # ensemble of the CPD-ROM at FP64 tolerance, the size of a serving pool
        _cp("cp_skew_f64_n1024_b64_step", 1024, 512, "cp_skew", "f64", 64, 8),
        # fitting a CP model to a tensor, two ALS iterations
        {"name": "fit_plain_n512_r256", "kind": "fit", "n": 512, "rank": 256, "method": "plain", "iters": 2},
        # a mix of requests served over four resident CPD-ROMs
        {"name": "serve_mix_48", "kind": "serve", "requests": 48, "slots": 32, "longest": 128},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["full", "full", "full", "cp", "cp", "fit", "serve"])
    if kind == "full":
        n, storage = _log_int(rng, 48, 1024), rng.choice(["f64", "f32x2", "f32", "bf16"])
        layout = rng.choice(["dense", "skew_packed"])
        batch = _log_int(rng, 1, 1024 if storage == "bf16" else 4)
        # batches of more than 8 BF16 trajectories go to the tensor cores, the others stream the tensor
        room = (2 << 40 if batch > 8 else 2 << 30) // (n ** 3 * batch)
        steps = rng.choice([0, _log_int(rng, 1, max(1, min(32, room)))])
        while batch > 1 and n ** 3 * batch * max(steps, 1) > (2 << 40 if batch > 8 else 2 << 30):
            batch = max(batch // 2, 1)
        return {"kind": kind, "n": n, "storage": storage, "layout": layout, "batch": batch, "steps": steps}
    if kind == "cp":
        n = _log_int(rng, 64, 1024)
        rank, storage = _log_int(rng, max(16, n // 8), n), rng.choice(["f64", "bf16", "f32"])
        batch = _log_int(rng, 1, 64 if storage == "f32" else 1024)
        form = rng.choice(["cp_skew", "cp_skew", "cp"])
        room = (1 << 32) // (n * rank * batch)
        # a general CP model conserves no energy: its right-hand side only
        steps = 0 if form == "cp" else rng.choice([0, _log_int(rng, 1, max(1, min(64, room)))])
        return {"kind": kind, "n": n, "rank": rank, "form": form, "storage": storage, "batch": batch, "steps": steps}
    if kind == "fit":
        n = _log_int(rng, 96, 512)
        return {"kind": kind, "n": n, "rank": _log_int(rng, 16, min(256, n)), "method": rng.choice(["plain", "skew"]),
                "iters": rng.randint(1, 2)}
    return {"kind": kind, "requests": rng.randint(12, 48), "slots": rng.choice([16, 24, 32]),
            "longest": _log_int(rng, 32, 128)}


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, dtype=torch.float64, device="cuda")


def _skew_tensor(g, n):
    G = _normal(g, n, n, n)
    C = G - G.transpose(0, 2)
    C /= n
    return C


def _factors(g, n, rank):
    """Three n x rank factors z / (r sqrt(rank)), the middle one scaled so that
    advection rates are like those of the skew tensors."""
    d = 1.0 / (torch.arange(1, rank + 1, dtype=torch.float64, device="cuda") * math.sqrt(rank))
    A, B, C = (_normal(g, n, rank) * d for _ in range(3))
    return A, B * (0.05 * rank ** 1.5 / math.sqrt(n)), C


def _states(g, batch, n):
    return _normal(g, batch, n) / torch.arange(1, n + 1, dtype=torch.float64, device="cuda")


def _stiffness(n):
    return (torch.arange(1, n + 1, dtype=torch.float64, device="cuda") / n) ** 2


def _inputs(case, seed):
    """Tensors of a case from the seed alone, in the order in which they are drawn."""
    g = _gen(seed)
    if case["kind"] == "full":
        return _skew_tensor(g, case["n"]), _states(g, case["batch"], case["n"])
    if case["kind"] == "cp":
        return _factors(g, case["n"], case["rank"]), _states(g, case["batch"], case["n"])
    if case["kind"] == "fit":
        n, rank = case["n"], case["rank"]
        U, V, W = (_normal(g, n, 24) for _ in range(3))
        X = ((U[:, None, :] * V[None]).reshape(n * n, 24) @ W.T).reshape(n, n, n) / math.sqrt(24.0)
        X += 1e-2 * _normal(g, n, n, n)
        if case["method"] == "skew":
            X = X - X.transpose(0, 2)
            shapes = [(n, 2 * (rank // 2)), (n, rank // 2)]
        else:
            shapes = [(n, rank)] * 3
        return X.contiguous(), [(_normal(g, *s) / math.sqrt(n)).cpu().numpy() for s in shapes]
    models = [_factors(g, n, rank) for n, rank, _ in SERVED]
    # the same load for every seed (log-uniform horizons, the models in turn), other states
    which = np.arange(case["requests"]) % len(SERVED)
    lot = np.random.default_rng(case["requests"])
    horizons = np.exp(lot.uniform(math.log(16), math.log(case["longest"]), case["requests"])).astype(np.int64)
    lot = np.random.default_rng(int(seed))
    u0 = [lot.standard_normal(SERVED[m][0]) / np.arange(1, SERVED[m][0] + 1) for m in which]
    return models, which, horizons, u0


def prepare(case, seed):
    """The resident model (and trajectories, fit context or server) and the inputs of the call."""
    ops = {"nu": NU, "dt": DT}
    if case["kind"] in ("full", "cp"):
        n, batch = case["n"], case["batch"]
        op, u = _inputs(case, seed)
        if case["kind"] == "full":
            rom = grom.Rom(n, "full", case["storage"], tensor=op, stiffness=_stiffness(n), max_batch=batch,
                           layout=case["layout"], **ops)
        else:
            rom = grom.Rom(n, case["form"], case["storage"], factors=op, stiffness=_stiffness(n), max_batch=batch, **ops)
        state = {"rom": rom, "u": u, "out": torch.empty_like(u), "steps": case["steps"]}
        if case["steps"]:
            state["traj"] = grom.Trajectories(rom, u)
        return state
    if case["kind"] == "fit":
        X, factors = _inputs(case, seed)
        return {"als": grom.Als(X), "factors": factors, "iters": case["iters"], "method": case["method"]}
    models, which, horizons, u0 = _inputs(case, seed)
    server = grom.Server(1 << 34, quantum=16)
    streams = [torch.cuda.Stream() for _ in SERVED]
    torch.cuda.synchronize()  # the factors are read on the ROMs' own streams
    for (n, rank, storage), f, s in zip(SERVED, models, streams):
        server.add_rom(grom.Rom(n, "cp_skew", storage, factors=f, stiffness=_stiffness(n), max_batch=case["slots"],
                                stream=s, **ops), case["slots"])
    return {"server": server, "streams": streams, "which": which, "horizons": horizons, "u0": u0,
            "arrivals": np.zeros(len(which))}


def run(state):
    if "server" in state:
        got = state["server"].serve(state["which"], state["horizons"], state["arrivals"], state["u0"], want_final=True)
        return {"final": got["final"], "steps": got["steps"]}
    if "als" in state:
        factors, residuals = state["als"].fit(state["factors"], state["iters"], method=state["method"], ridge=1e-5)
        return {"factors": factors, "residuals": residuals}
    if state["steps"]:
        state["traj"].step_host(state["steps"], None, state["out"])
        return state["out"]
    return state["rom"].nonlinear(state["u"], state["out"])


def _operator(case):
    """(values of the advection operator that its result depends on, multiply-adds
    per evaluation of one trajectory).  A quadratic form needs the sum of C_ijk and
    C_ikj only; skewness in (i, k) leaves n (n^2 - 1) / 3 of those independent."""
    n = case["n"]
    if case["kind"] == "full":
        v = n * (n * n - 1) // 3 if case["layout"] == "skew_packed" else n * n * (n + 1) // 2
        return v, v
    return 3 * n * case["rank"], (5 if case["form"] == "cp_skew" else 3) * n * case["rank"]


def work(case):
    if case["kind"] == "fit":
        n, r, iters = case["n"], case["rank"], case["iters"]
        updates = 3 if case["method"] == "plain" else 2
        per = updates * (2.0 * n ** 3 * r + 2.0 * n * r * r + r ** 3 / 3.0)  # MTTKRP, solves, Cholesky
        return {"bytes": iters * updates * 2.0 * n ** 3, "flops": iters * per}
    if case["kind"] == "serve":
        steps = case["requests"] * (case["longest"] - 16) / math.log(case["longest"] / 16.0) / len(SERVED)
        return {"bytes": float(sum(3 * n * r * ELEM[s] for n, r, s in SERVED)),
                "flops": steps * sum(10.0 * n * r for n, r, _ in SERVED)}
    values, macs = _operator(case)
    evals = max(case["steps"], 1)
    op = values * ELEM[case["storage"]]
    # an evaluation reads u and writes c; a run of steps reads and writes the history (three u, three n)
    state = (12 if case["steps"] else 2) * 8.0 * case["n"] * case["batch"]
    return {"bytes": float(op * (evals if op > ON_CHIP else 1)) + state, "flops": 2.0 * macs * evals * case["batch"]}


def _term(op, form, u):
    """C(u)u in 64 bits for the states u (batch x n)."""
    if form == "full":
        n, batch = op.shape[0], u.shape[0]
        c = torch.empty_like(u)
        rows = max(1, (1 << 28) // (n * batch))
        for i in range(0, n, rows):
            d = (op[i:i + rows].reshape(-1, n) @ u.T).reshape(-1, n, batch)
            c[:, i:i + rows] = (d * u.T).sum(1).T
        return c
    A, B, C = op
    p, q = u @ B, u @ C
    if form == "cp":
        return (p * q) @ A.T
    return (p * q) @ A.T - (p * (u @ A)) @ C.T


def _steps(op, form, u, n, steps):
    """BDF3/EXT3 from one state: orders 1 and 2 in the first two steps."""
    beta = ((1.0, -1.0), (1.5, -2.0, 0.5), (11.0 / 6.0, -3.0, 1.5, -1.0 / 3.0))
    alpha = ((1.0,), (2.0, -1.0), (3.0, -3.0, 1.0))
    a, us, cs = _stiffness(n), [u], []
    for s in range(steps):
        k = min(s + 1, 3)
        cs = [_term(op, form, us[0])] + cs[:2]
        rhs = sum(alpha[k - 1][q] * cs[q] for q in range(k)) + sum(beta[k - 1][q + 1] / DT * us[q] for q in range(k))
        us = [-rhs / (beta[k - 1][0] / DT + NU * a)] + us[:2]
    return us[0]


def _als(X, factors, method, iters):
    """ALS through the normal equations, ridge 1e-5 of the largest diagonal entry."""
    n = X.shape[0]
    norm = torch.linalg.norm(X)

    def update(F, mode):
        P, Q = [F[m] for m in range(3) if m != mode]
        Y = X.movedim(mode, 0).reshape(n, n * n)
        M = Y @ (P[:, None, :] * Q[None]).reshape(n * n, -1)
        H = (P.T @ P) * (Q.T @ Q)
        H = H + 1e-5 * H.diagonal().max() * torch.eye(H.shape[0], dtype=H.dtype, device=H.device)
        return torch.linalg.solve(H, M.T).T.contiguous()

    def residual(F):
        K = (F[0][:, None, :] * F[1][None]).reshape(n * n, -1) @ F[2].T
        return float(torch.linalg.norm(X.reshape(n * n, n) - K) / norm)

    def skew(A, B):
        h = A.shape[1] // 2
        return [A, torch.cat([B, B], 1), torch.cat([A[:, h:], -A[:, :h]], 1)]

    F, res = list(factors), []
    for _ in range(iters):
        if method == "plain":
            for mode in range(3):
                F[mode] = update(F, mode)
            res.append(residual(F))
        else:
            A, B = F
            h = A.shape[1] // 2
            B = update(skew(A, B), 1)
            B = 0.5 * (B[:, :h] + B[:, h:])
            A = 0.5 * A + 0.5 * update(skew(A, B), 0)
            F = [A, B]
            res.append(residual(skew(A, B)))
    return F, np.array(res)


def exact(case, seed):
    if case["kind"] in ("full", "cp"):
        op, u = _inputs(case, seed)
        form = "full" if case["kind"] == "full" else case["form"]
        return _steps(op, form, u, case["n"], case["steps"]) if case["steps"] else _term(op, form, u)
    if case["kind"] == "fit":
        X, factors = _inputs(case, seed)
        F, res = _als(X, [torch.from_numpy(f).cuda() for f in factors], case["method"], case["iters"])
        return {"factors": F, "residuals": res}
    models, which, horizons, u0 = _inputs(case, seed)
    final = [_steps(models[m], "cp_skew", torch.from_numpy(u)[None].cuda(), len(u), int(h))[0].cpu().numpy()
             for m, h, u in zip(which, horizons, u0)]
    return {"final": final, "steps": None}
