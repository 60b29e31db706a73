"""The workloads whose speed this framework answers for, as callers run them.

Each case is one call (or one forward/backward pair, or one burst of server
requests) through the package's public binding: many independent gas cells of
one reaction network integrated from 0 to ``years``. Networks are the seeded
synthetic ones of ``synth`` (the sizes of the tests and of the benchmark,
and others between them); a program draws its network once and keeps the
compiled handle, so handles are kept here too. Cells (density, temperature,
extinction, metallicity of the gas) come from the seed.
"""
import functools
import math

import numpy as np
import torch

from paper_2511_10558_gb300 import carbox, synth

YR = synth.YEAR
RTOL, ATOL = 1e-4, 1e-20


def listed():
    return [
        # one zone of an atomic network: an interactive call, all latency (the reference single cell's network)
        {"name": "zone32", "kind": "solve", "S": 32, "R": 200, "C": 1, "years": 1e6, "prec": "fp64", "method": "bdf"},
        # a parameter grid with the small network
        {"name": "grid32", "kind": "solve", "S": 32, "R": 200, "C": 2048, "years": 1e6, "prec": "fp64",
         "method": "bdf"},
        # the headline workload at the benchmark's oracle-sample size: 150 species, 1 Myr, both precisions
        {"name": "grid150", "kind": "solve", "S": 150, "R": 1500, "C": 1216, "years": 1e6, "prec": "fp64",
         "method": "bdf"},
        {"name": "grid150_mixed", "kind": "solve", "S": 150, "R": 1500, "C": 1501, "years": 1e6, "prec": "mixed",
         "method": "bdf"},
        # one chemistry step of an operator-split hydrodynamics run: more cells, a short span
        {"name": "hydro150", "kind": "solve", "S": 150, "R": 1500, "C": 2500, "years": 3e2, "prec": "fp64",
         "method": "bdf"},
        # the large network, in both precisions
        {"name": "large500_mixed", "kind": "solve", "S": 500, "R": 6000, "C": 200, "years": 1e4, "prec": "mixed",
         "method": "bdf"},
        {"name": "large500", "kind": "solve", "S": 500, "R": 6000, "C": 160, "years": 1e3, "prec": "fp64",
         "method": "bdf"},
        # a network between the tuned sizes, with the other integrator
        {"name": "esdirk97", "kind": "solve", "S": 97, "R": 873, "C": 333, "years": 1e4, "prec": "fp64",
         "method": "esdirk"},
        # collapsing cells: the environment follows tracks in time
        {"name": "track128", "kind": "track", "S": 128, "R": 1200, "C": 500, "years": 1e5, "prec": "fp64",
         "method": "bdf"},
        # sensitivities: recorded solve and discrete adjoint with the environment's gradients
        {"name": "adjoint150", "kind": "adjoint", "S": 150, "R": 1500, "C": 304, "years": 1e5, "prec": "fp64",
         "method": "bdf"},
        # the same through torch.autograd, as a sampler's gradient step runs it on a few observed cells
        {"name": "autograd61", "kind": "autograd", "S": 61, "R": 480, "C": 64, "years": 1e5, "prec": "fp64",
         "method": "bdf"},
        # a service: requests of three networks in host memory, answered as they finish
        {"name": "serve", "kind": "serve", "S": 150, "R": 1500, "C": 120, "years": 1e5, "prec": "mixed",
         "method": "bdf"},
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "host", "track", "adjoint", "autograd", "serve"])
    prec = rng.choice(["fp64", "mixed"])
    method = rng.choice(["bdf", "bdf", "bdf", "esdirk"]) if kind in ("solve", "host", "track") else "bdf"
    hi = {"solve": 512, "host": 256, "track": 256, "adjoint": 150, "autograd": 100, "serve": 150}[kind]
    S = int(round(_logu(rng, 30, hi)))
    R = int(round(S * rng.uniform(5.8, 6.2 if S < 64 else 11.5)))
    # large networks and the integrator with four stages a step are asked for shorter spans
    top = 1e6
    if S > 256:
        top = 1e3 if prec == "fp64" else 1e4
    if method == "esdirk":
        top = min(top, 1e4 if S >= 64 else 1e3)
    if kind in ("adjoint", "autograd"):
        top = 1e5
    years = float("%.3g" % _logu(rng, 1e2, top))
    cap = 0.3 / _cell_seconds(S, years, prec, method) * (0.4 if kind in ("adjoint", "autograd", "serve") else 1.0)
    most = {"autograd": 64, "adjoint": 400, "serve": 200}.get(kind, 4000)
    C = max(1, int(round(_logu(rng, 1, max(2.0, min(most, cap))))))
    return {"kind": kind, "S": S, "R": R, "C": C, "years": years, "prec": prec, "method": method}


def _counts(S, years, method):
    """Typical factorisations and Newton iterations of one cell over a span."""
    lt = min(max(math.log10(years), 2.0), 7.0)
    lu = np.interp(lt, [2, 3, 4, 5, 6, 7], [22, 27, 39, 60, 88, 120])
    it = np.interp(lt, [2, 3, 4, 5, 6, 7], [150, 180, 245, 365, 530, 700])
    return (2.2 * lu, 3.0 * it) if method == "esdirk" else (lu, it)


def _cell_seconds(S, years, prec, method):
    """Rough device seconds a cell adds to a large batch (bounds what draw() asks for)."""
    lu, it = _counts(S, years, method)
    one = 2.5e-7 * (lu * 1.2 * (S / 150) ** 3 + it * (0.2 + 0.15 * (S / 150) ** 2)) / 0.15
    return one * (0.7 if prec == "mixed" and S > 64 else 1.0)


# ---------------------------------------------------------------- what a program has in hand


@functools.lru_cache(maxsize=None)
def _drawn(S, R):
    return synth.make_network(S, R)


@functools.lru_cache(maxsize=None)
def _network(S, R):
    return carbox.Network.from_synth(_drawn(S, R))


def _cells(net, C, seed):
    """phi [C, 5] and x0 [S, C]: the cells of ``synth`` with a metallicity each."""
    phi = synth.cells(C, seed=seed)
    x0 = np.repeat(synth.initial_abundances(net)[:, None], C, axis=1)
    z = 10.0 ** np.random.default_rng(seed + 1).uniform(-0.5, 0.3, C)
    for name in ("C+", "O", "N", "e-"):
        x0[net.index(name)] *= z
    return phi, x0


def _options(case):
    return carbox.options(rtol=RTOL, atol=ATOL,
                          precision=carbox.CBX_MIXED if case["prec"] == "mixed" else carbox.CBX_FP64,
                          method=carbox.CBX_METHOD_ESDIRK if case["method"] == "esdirk" else carbox.CBX_METHOD_BDF)


_OBSERVED = ("H", "H+", "H2", "He", "C", "C+", "N", "O", "e-", "H3+")


def _cotangent(net, C, seed):
    """Cotangents on the observed species, zero elsewhere."""
    w = np.zeros((net.n_species, C))
    rng = np.random.default_rng(seed + 2)
    for name in _OBSERVED:
        w[net.index(name)] = rng.uniform(-0.5, 0.5, C)
    return w


def prepare(case, seed):
    S, R, C, kind = case["S"], case["R"], case["C"], case["kind"]
    net, handle = _drawn(S, R), _network(S, R)
    st = {"kind": kind, "net": handle, "opt": _options(case), "t_end": case["years"] * YR}
    if kind == "serve":
        # a burst of requests of the small, this and (a few cells, a short span) the large network
        st["server"] = carbox.Server(mem_budget=8 << 30, n_streams=8, max_ctas=76)
        st["requests"] = []
        for k, (s, r, c, years) in enumerate([(S, R, C, case["years"]), (32, 200, 3 * C, 0.1 * case["years"]),
                                              (S, R, max(1, C // 3), 0.3 * case["years"]), (32, 200, C, case["years"]),
                                              (200, 1800, max(1, C // 10), 1e3), (S, R, 1, 1e4)]):
            phi, x0 = _cells(_drawn(s, r), c, seed + 10 * k)
            st["requests"].append((_network(s, r), phi, x0, years * YR))
        return st
    phi, x0 = _cells(net, C, seed)
    if kind == "host":
        st.update(phi=phi, x0=x0)
        return st
    dev = torch.device("cuda")
    st.update(phi=torch.tensor(phi, device=dev), x0=torch.tensor(x0, device=dev).contiguous())
    if kind == "track":
        st["track"] = torch.tensor(synth.tracks(phi, st["t_end"], 4), device=dev)
    if kind == "adjoint":
        st["tape"] = carbox.Tape(handle, C, 2000)
        st["cot"] = torch.tensor(_cotangent(net, C, seed), device=dev)
    if kind == "autograd":
        st["cot"] = torch.tensor(_cotangent(net, C, seed), device=dev)
        alpha = np.log(net.alpha) + np.random.default_rng(seed + 3).normal(0.0, 0.1, R)
        st["log_alpha"] = torch.tensor(alpha, device=dev, requires_grad=True)
        st["log_nH"] = torch.tensor(np.log(phi[:, 0]), device=dev, requires_grad=True)
        st["T"] = torch.tensor(phi[:, 1], device=dev, requires_grad=True)
        st["env"] = torch.tensor(phi[:, 2:], device=dev).contiguous()
    return st


def run(st):
    kind, net, opt, t_end = st["kind"], st["net"], st["opt"], st["t_end"]
    if kind == "solve":
        x, status, _ = carbox.solve(net, st["phi"], st["x0"], 0.0, t_end, opt)
        return {"x": x, "status": status}
    if kind == "host":
        x, status, _ = carbox.solve_host(net, st["phi"], st["x0"], 0.0, t_end, opt)
        return {"x": x, "status": status}
    if kind == "track":
        x, status, _ = carbox.solve_track(net, st["track"], st["x0"], 0.0, t_end, opt)
        return {"x": x, "status": status}
    if kind == "adjoint":
        x, status = carbox.solve_record(net, st["tape"], st["phi"], st["x0"], 0.0, t_end, opt)
        names = ("ln_alpha", "ln_nH", "T", "ln_zeta", "ln_G0", "A_V")
        g = carbox.grad_env(st["tape"], st["cot"], st["phi"].shape[0])
        return {"x": x, "status": status, **dict(zip(names, g))}
    if kind == "autograd":
        y = carbox.cell_solve(st["log_alpha"], st["log_nH"], st["T"], net, st["x0"], st["env"], t_end, opt)
        g = torch.autograd.grad(y, (st["log_alpha"], st["log_nH"], st["T"]), grad_outputs=st["cot"])
        return {"log_x": y.detach(), "ln_alpha": g[0], "ln_nH": g[1], "T": g[2]}
    srv = st["server"]
    ids = [srv.submit(n, phi, x0, 0.0, t, opt) for n, phi, x0, t in st["requests"]]
    out = {}
    for k, i in enumerate(ids):
        x, status, _ = srv.wait(i)
        out["x%d" % k], out["status%d" % k] = x, status
    return out


def work(case):
    """Inputs and outputs once; the structural operations of a typical cell's
    factorisations, solves and right-hand sides."""

    def of(S, R, C, years):
        info = _network(S, R).info()
        lu, it = _counts(S, years, case["method"])
        return C * (16.0 * S + 44.0), C * (lu * info["lu_flops"] + it * (2.0 * info["nnz_lu"] + 8.0 * R))

    S, R, C, years, kind = case["S"], case["R"], case["C"], case["years"], case["kind"]
    if kind == "serve":
        parts = [of(S, R, C, years), of(32, 200, 3 * C, 0.1 * years), of(S, R, max(1, C // 3), 0.3 * years),
                 of(32, 200, C, years), of(200, 1800, max(1, C // 10), 1e3), of(S, R, 1, 1e4)]
    else:
        parts = [of(S, R, C, years)]
    b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    if kind == "track":
        b += C * 4 * 48.0
    if kind in ("adjoint", "autograd"):
        # one factorisation and one transposed solve per accepted step (a third
        # of the Newton iterations); the cotangents in, the gradients out
        info, (_, it) = _network(S, R).info(), _counts(S, years, "bdf")
        steps = it / 2.5
        f += C * steps * (info["lu_flops"] + 2.0 * info["nnz_lu"] + 12.0 * R)
        b += C * (8.0 * S + 40.0) + 8.0 * R
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------- 64-bit values


def exact(case, seed):
    """x(t_end) of a constant-environment solve of one or two cells of a small
    network, from a linearly implicit extrapolation method at tight tolerance
    (Hairer & Wanner, Solving ODEs II, Sec. IV.9); None elsewhere, where it
    would take minutes."""
    if case["kind"] not in ("solve", "host") or case["S"] > 64 or case["C"] > 2:
        return None
    net = _drawn(case["S"], case["R"])
    phi, x0 = _cells(net, case["C"], seed)
    x = np.stack([_reference(net, phi[c], x0[:, c], case["years"] * YR) for c in range(case["C"])], axis=1)
    return {"x": x if case["kind"] == "host" else torch.tensor(x), "status": None}


def _reference(net, phi, x0, t_end, rtol=1e-8, atol=1e-18, kmax=9):
    n_H, T, A_V, G0, zeta = phi
    two = net.rtype == synth.TWO_BODY
    k = np.where(two, net.alpha * (T / 300.0) ** net.beta * np.exp(-net.gamma / T) * n_H,
                 np.where(net.rtype == synth.COSMIC_RAY, net.alpha * zeta, net.alpha * G0 * np.exp(-net.gamma * A_V)))
    S, R = net.n_species, net.n_reactions
    j = np.arange(R)
    nu = np.zeros((S, R))
    for col in net.reac.T:
        np.add.at(nu, (col[col >= 0], j[col >= 0]), -1.0)
    for col in net.prod.T:
        np.add.at(nu, (col[col >= 0], j[col >= 0]), 1.0)
    a, b = net.reac[:, 0], np.where(two, net.reac[:, 1], 0)

    def f(y):
        return nu @ (k * y[a] * np.where(two, y[b], 1.0))

    def jac(y):
        d = np.zeros((R, S))
        np.add.at(d, (j, a), k * np.where(two, y[b], 1.0))
        np.add.at(d, (j[two], b[two]), (k * y[a])[two])
        return nu @ d

    t, y, H = 0.0, x0.copy(), 1e-3 * YR
    while t < t_end:
        H = min(H, t_end - t)
        J, table, best = jac(y), [], None
        for n in range(1, kmax + 1):
            inv = np.linalg.inv(np.eye(S) - H / n * J)
            z = y.copy()
            for _ in range(n):
                z = z + inv @ (H / n * f(z))
            row = [z]
            for m in range(1, n):
                row.append(row[m - 1] + (row[m - 1] - table[-1][m - 1]) / (n / (n - m) - 1.0))
            table.append(row)
            if n >= 3:
                w = atol + rtol * np.maximum(np.abs(y), np.abs(row[-1]))
                err = float(np.sqrt(np.mean(((row[-1] - row[-2]) / w) ** 2)))
                if err <= 1.0:
                    best = row[-1]
                    break
        if best is None:
            H *= 0.3
            continue
        t, y = t + H, best
        H *= 2.0 if n <= 7 else 1.2
    return y
