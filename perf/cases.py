"""The work a user has this library do, as measurable cases.

Three kinds of work, through the package's public entry points:

* ``single``  one hierarchy in a Context: rho(0) set, the whole propagation with its output rows, then rho (or, for a
  checkpointed run, the whole state in and out);
* ``scan``    many hierarchies with different baths, temperatures and depths in one Batch (a parameter scan);
* ``serve``   a burst of requests of mixed sizes through the continuous-batching Server.

Models are drawn as in ``workloads``: seeded FMO-like Hamiltonians (site energies U(12100, 12600), couplings N(0, 40)),
three weakly coupled 8-site blocks for the 24-site aggregate, trapping 1/ps on the third site and 1/ns recombination.
``exact`` propagates the same model in complex128 with plain torch and classic RK4.

Results of mixed-precision runs are handed on as float32: that is what those runs carry (the auxiliaries are float).
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

from paper_1012_4382_gb300 import heom, serving

CM = 2.0 * math.pi * 2.99792458e-5  # cm^-1 -> rad/fs
KB = 0.6950348004  # cm^-1 / K


def listed():
    return [
        # the smallest call: the two-site model of the tests, every step an output row; FP64 is a Context's default
        _single("dimer depth 4 fp64", 2, 4, "fp64", 1000, 1),
        # the benchmark's headline: seven sites with a trap, depth 6 (1716 nodes), single precision
        _single("7 sites depth 6 mixed", 7, 6, "fp32", 1000, 10),
        # the same hierarchy in double precision
        _single("7 sites depth 6 fp64", 7, 6, "fp64", 400, 10),
        # the deeper rows of the paper's timing table (6435, 19448 and 50388 nodes)
        _single("7 sites depth 8 mixed", 7, 8, "fp32", 500, 10),
        _single("7 sites depth 10 fp64", 7, 10, "fp64", 100, 10),
        _single("7 sites depth 12 mixed", 7, 12, "fp32", 200, 10),
        # a checkpointed run with a complex Hamiltonian and the Markov terminator: state in, steps, state out
        _single("5 sites depth 7 resumed", 5, 7, "fp32", 400, 20, cplx=True, term=1, resume=True),
        # the 24-site aggregate (20475 nodes) in both precisions
        _single("24 sites depth 4 mixed", 24, 4, "fp32", 100, 10),
        _single("24 sites depth 4 fp64", 24, 4, "fp64", 20, 10),
        # the batched scan of the benchmark (256 models, depths 4 to 8), and a smaller one in double precision
        _scan("scan of 256 mixed", 7, 256, 4, 8, "fp32", 60, 10),
        _scan("scan of 24 fp64", 7, 24, 4, 7, "fp64", 40, 10),
        # a burst of short requests of 2 to 8 sites and depths 3 to 8
        {"name": "burst of 40 requests", "kind": "serve", "count": 40, "steps_lo": 100, "steps_hi": 500, "every": 100,
         "prec": "fp32"},
    ]


def _single(name, N, K, prec, steps, every, cplx=False, term=0, low_temp=0, scaled=0, resume=False):
    return {"name": name, "kind": "single", "N": N, "K": K, "prec": prec, "steps": steps, "every": every, "cplx": cplx,
            "term": term, "low_temp": low_temp, "scaled": scaled, "resume": resume}


def _scan(name, N, count, k_lo, k_hi, prec, steps, every):
    return {"name": name, "kind": "scan", "N": N, "count": count, "k_lo": k_lo, "k_hi": k_hi, "prec": prec,
            "steps": steps, "every": every}


# ------------------------------------------------------------------- drawing

_MOST_FLOPS = {"fp32": 8e11, "fp64": 4.5e10}  # of one drawn pass (the largest listed pass of each precision)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "wide", "scan", "serve"])
    prec = rng.choice(["fp32", "fp64"])
    if kind == "serve":
        lo = _log_int(rng, 40, 200)
        return {"kind": "serve", "count": _log_int(rng, 6, 40), "steps_lo": lo, "steps_hi": lo + _log_int(rng, 50, 300),
                "every": rng.choice([10, 50, 100]), "prec": "fp32"}
    if kind == "scan":
        k_lo = rng.randint(2, 5)
        c = _scan("", rng.randint(3, 8), _log_int(rng, 4, 96), k_lo, rng.randint(k_lo, 7), prec, 0, rng.choice([1, 5, 10]))
        c["steps"] = _log_int(rng, 20, 200)
    else:
        N = rng.randint(9, 24) if kind == "wide" else rng.randint(2, 8)
        most = _log_int(rng, 60, 20475) if kind == "wide" else _log_int(rng, 10, 50388)
        K = 1
        while math.comb(N + K + 1, N) <= most and K < 24:
            K += 1
        c = _single("", N, K, prec, 0, rng.choice([1, 5, 10, 25]), cplx=rng.random() < 0.25,
                    term=1 if rng.random() < 0.25 else 0, low_temp=1 if rng.random() < 0.25 else 0,
                    scaled=1 if rng.random() < 0.2 else 0, resume=rng.random() < 0.2)
        c["steps"] = _log_int(rng, 50, 1000)
    del c["name"]
    while work(c)["flops"] > _MOST_FLOPS[c["prec"]] and c["steps"] > 3:
        c["steps"] = c["steps"] * 2 // 3
    while work(c)["flops"] > _MOST_FLOPS[c["prec"]]:
        c["count"] = c["count"] * 2 // 3
    return c


# ------------------------------------------------------------------- models

def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _hamiltonian(g, N, cplx):
    eps = g.uniform(12100.0, 12600.0, size=N)
    J = g.normal(0.0, 40.0, size=(N, N))
    if N == 24:  # three 8-site blocks, weakly coupled
        blk = np.arange(N) // 8
        J = np.where(blk[:, None] == blk[None, :], J, J / 8.0)
    J = np.triu(J, 1)
    H = np.diag(eps) + J + J.T + 0j
    if cplx:
        Ji = np.triu(g.normal(0.0, 20.0, size=(N, N)), 1)
        H = H + 1j * (Ji - Ji.T)
    return H


def _model(N, K, H, lam, T, term=0, low_temp=0, scaled=0):
    trap = np.zeros(N)
    trap[min(2, N - 1)] = 1.0
    return {"N": N, "K": K, "H": H, "lam": np.broadcast_to(np.asarray(lam, dtype=np.float64), (N,)).copy(),
            "gam": np.full(N, 106.0), "T": T, "trap": trap, "recomb": np.full(N, 1e-3), "terminator": term,
            "add_reorg": 0, "low_temp": low_temp, "scaled": scaled}


def _rho0(N, site):
    r = np.zeros((N, N), dtype=np.complex128)
    r[site, site] = 1.0
    return r


def _models(case, seed):
    """The models of a case with their initial states and step counts: a list of (params, rho0, steps)."""
    g = _rng(seed)
    if case["kind"] == "single":
        N = case["N"]
        lam = g.uniform(20.0, 60.0, size=N)
        p = _model(N, case["K"], _hamiltonian(g, N, case["cplx"]), lam, float(g.uniform(250.0, 300.0)), case["term"],
                   case["low_temp"], case["scaled"])
        return [(p, _rho0(N, int(g.integers(0, N))), case["steps"])]
    out = []
    for i in range(case["count"]):
        if case["kind"] == "scan":
            N = case["N"]
            # the depths of a scan are part of its size: the same for every seed
            K = case["k_lo"] + (i * 7 + 3) % (case["k_hi"] - case["k_lo"] + 1)
            p = _model(N, K, _hamiltonian(g, N, False), float(g.uniform(2.0, 200.0)), float(g.uniform(77.0, 300.0)))
            out.append((p, _rho0(N, 0), case["steps"]))
        else:
            # sizes and lengths of the requests belong to the case, their models to the seed
            s = _rng(1234 + i)
            N, K = int(s.integers(2, 9)), int(s.integers(3, 9))
            p = _model(N, K, _hamiltonian(g, N, False), 35.0, 300.0)
            out.append((p, _rho0(N, 0), int(s.integers(case["steps_lo"], case["steps_hi"] + 1))))
    return out


def _start_state(N, nodes, seed, root):
    """A checkpoint to resume from: rho and Hermitian auxiliaries that decay with the node's index."""
    g = _rng(seed + 77)
    a = g.normal(size=(nodes, N, N)) + 1j * g.normal(size=(nodes, N, N))
    a = (a + np.conj(np.transpose(a, (0, 2, 1)))) * (1e-3 / (1.0 + np.arange(nodes)))[:, None, None]
    a[0] = root
    return a.astype(np.complex64).astype(np.complex128)


# --------------------------------------------------------------- entry points

def prepare(case, seed):
    models = _models(case, seed)
    st = {"case": case, "dt": 1.0, "models": models}
    if case["kind"] == "single":
        p, rho0, _ = models[0]
        st["ctx"] = heom.Context(p, case["prec"])
        st["rho0"] = rho0
        if case["resume"]:
            st["state"] = _start_state(p["N"], st["ctx"].nodes, seed, rho0)
    elif case["kind"] == "scan":
        st["batch"] = heom.Batch([m[0] for m in models], case["prec"])
        st["rho0"] = [m[1] for m in models]
    else:
        st["server"] = serving.Server(2 << 30, 64 << 20, 32)
    return st


def _real(a, case):
    return np.asarray(a, dtype=np.float32 if case["prec"] == "fp32" else np.float64)


def _complex(a, case):
    return np.asarray(a, dtype=np.complex64 if case["prec"] == "fp32" else np.complex128)


def run(st):
    case = st["case"]
    if case["kind"] == "single":
        c = st["ctx"]
        if case["resume"]:
            c.set_state(st["state"])
        else:
            c.set_rho0(st["rho0"])
        r = c.propagate(st["dt"], case["steps"], case["every"])
        out = {"pops": _real(r["pops"], case), "eta": _real(r["eta"], case)}
        if case["resume"]:
            state, extra = c.state()
            out["state"] = _complex(state, case)
            out["extra"] = _real(extra, case)
        else:
            out["rho"] = _complex(c.rho(), case)
            out["t_mean"] = _real(c.trapping_time()[0], case)
        return out
    if case["kind"] == "scan":
        b = st["batch"]
        b.set_rho0(st["rho0"])
        rows = b.propagate(st["dt"], case["steps"], case["every"])
        return {"pops": _real(np.stack([r["pops"] for r in rows]), case),
                "eta": _real(np.stack([r["eta"] for r in rows]), case)}
    srv = st["server"]
    ids = [srv.submit(p, rho0, st["dt"], steps, case["every"], case["prec"]) for p, rho0, steps in st["models"]]
    left = set(ids)
    while left:
        if srv.progress():
            left -= {i for i in left if srv.status(i) in (serving.DONE, serving.FAILED)}
        time.sleep(5e-5)
    res = [srv.result(i) for i in ids]
    for i in ids:
        srv.release(i)
    return {"pops": _real(np.concatenate([r["pops"].reshape(-1) for r in res]), case),
            "eta": _real(np.concatenate([r["eta"] for r in res]), case),
            "loss": _real(np.concatenate([r["loss"] for r in res]), case)}


# ------------------------------------------------------------------ the work

def _sizes(case):
    """(N, nodes, steps) of every hierarchy of the case."""
    if case["kind"] == "single":
        return [(case["N"], math.comb(case["N"] + case["K"], case["K"]), case["steps"])]
    if case["kind"] == "scan":
        n = case["k_hi"] - case["k_lo"] + 1
        ks = [case["k_lo"] + (i * 7 + 3) % n for i in range(case["count"])]
        return [(case["N"], math.comb(case["N"] + k, k), case["steps"]) for k in ks]
    out = []
    for i in range(case["count"]):
        s = _rng(1234 + i)
        N, K = int(s.integers(2, 9)), int(s.integers(3, 9))
        out.append((N, math.comb(N + K, K), int(s.integers(case["steps_lo"], case["steps_hi"] + 1))))
    return out


def work(case):
    """One pass: the packed hierarchy (N^2 reals a node) and its links read once and the hierarchy written once, plus
    the output rows; the multiply-adds of the Hermitian-packed right-hand side in every stage of every step."""
    r = 8 if case["prec"] == "fp64" else 4
    flops = nbytes = 0.0
    for N, M, steps in _sizes(case):
        per = N * (N - 1) // 2 * ((8 * N - 12 if case.get("cplx") else 4 * N - 6) + 12) + N * (2 * N + 1)
        flops += 2.0 * per * M * 4 * steps
        nbytes += 2.0 * M * N * N * r + 8.0 * M * N + (steps // case["every"] + 1) * (N + 2) * 8.0
        if case.get("resume"):
            nbytes += 2.0 * M * N * N * 16
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------- in 64 bits

def _nodes(N, K):
    """Multi-indices with |n| <= K by level, then lexicographically descending, and the rows of n + e_j and n - e_j
    (the number of nodes where there is none)."""
    rows = [np.zeros((1, N), np.int64)]
    for lev in range(1, K + 1):
        up = (rows[-1][:, None, :] + np.eye(N, dtype=np.int64)[None]).reshape(-1, N)
        key = _key(up, K)
        rows.append(up[np.unique(key, return_index=True)[1]][::-1])
    n = np.concatenate(rows)
    key = _key(n, K)
    order = np.argsort(key)
    M = len(n)

    def find(m, ok):
        k = _key(m, K)
        pos = np.minimum(np.searchsorted(key[order], k), M - 1)
        return np.where(ok & (key[order][pos] == k), order[pos], M)

    level = n.sum(1)
    up = np.stack([find(n + np.eye(N, dtype=np.int64)[j], level < K) for j in range(N)], 1)
    dn = np.stack([find(n - np.eye(N, dtype=np.int64)[j], n[:, j] > 0) for j in range(N)], 1)
    return n, up, dn


def _key(n, K):
    k = np.zeros(len(n), np.int64)
    for j in range(n.shape[1]):
        k = k * (K + 2) + np.maximum(n[:, j], 0)
    return k


def _exact_system(models, state=None):
    """The right-hand side of models with the same N, side by side, in complex128.

    d sigma/dt = A + A^+, A = -i H_eff sigma + (row part of the hierarchy couplings) - (damping)/2: every term of the
    hierarchy's right-hand side acts on the rows of a Hermitian matrix and, conjugated, on its columns."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    N = models[0]["N"]
    B, iu, idn, wu, wd, ng, off, off_damp = [], [], [], [], [], [], [0], []
    total = sum(math.comb(p["N"] + p["K"], p["K"]) for p in models)
    cache = {}
    a_i = np.arange(N)
    for p in models:
        if p["K"] not in cache:
            cache[p["K"]] = _nodes(N, p["K"])
        n, up, dn = cache[p["K"]]
        M, base = len(n), off[-1]
        kT = KB * p["T"] * CM
        lam, gam = p["lam"] * CM, p["gam"] * CM
        al, be = 2.0 * lam * kT, lam * gam
        theta = be + 1j * al
        gl = (p["trap"] + p["recomb"]) * 1e-3
        H = p["H"] - np.eye(N) * np.mean(np.real(np.diag(p["H"])))
        B.append(np.broadcast_to(-1j * H * CM - np.diag(0.5 * gl), (1, N, N)))
        lt = np.zeros(N)
        if p["low_temp"]:
            lt = 2.0 * lam * kT / gam - lam / np.tan(gam / (2.0 * kT))
        damp = -(lt[:, None] + lt[None, :])
        np.fill_diagonal(damp, 0.0)
        off_damp.append(damp[None])
        sc = np.where(np.abs(theta) > 0, np.abs(theta), 1.0)
        u_w = np.sqrt((n + 1) * sc) if p["scaled"] else np.ones(n.shape)
        d_w = np.sqrt(n / sc) if p["scaled"] else n.astype(np.float64)
        ngam = n @ gam
        # element (a, b) of the row part reads element (a, b) of n + e_a and of n - e_a
        iu.append(np.where(up == M, total, up + base))
        idn.append(np.where(dn == M, total, dn + base))
        own = np.zeros((M, N), dtype=np.complex128)
        if p["terminator"]:
            leaf = (n.sum(1) == p["K"])[:, None]
            own = np.where(leaf, (n + 1) / (ngam[:, None] + gam[None, :]), 0.0)
        wu.append(1j * u_w)
        wd.append(d_w * theta)
        ng.append((ngam, own, 1j * theta, -1j * np.conj(theta)))
        off.append(base + M)
    inst = np.concatenate([np.full(off[i + 1] - off[i], i) for i in range(len(models))])
    t = lambda x: torch.as_tensor(np.ascontiguousarray(x), device=dev)  # noqa: E731
    inst_t = t(inst)
    one = len(models) == 1
    Bt = t(np.concatenate(B))
    Bt = Bt[0] if one else Bt[inst_t]
    dampt = t(np.concatenate(off_damp))
    dampt = dampt[0] if one else dampt[inst_t]
    upt, dnt = t(np.concatenate(iu)), t(np.concatenate(idn))
    cols = torch.arange(N * N, device=dev).view(1, N, N)
    gu = (upt.view(-1, N, 1) * (N * N) + cols).reshape(-1)
    gd = (dnt.view(-1, N, 1) * (N * N) + cols).reshape(-1)
    wut, wdt = t(np.concatenate(wu)).view(-1, N, 1), t(np.concatenate(wd)).view(-1, N, 1)
    ngt = t(np.concatenate([x[0] for x in ng])).view(-1, 1, 1)
    # terminator: n + e_j beyond the last level ~ (n_j+1)/(ngam+gamma_j) theta_j sigma_n, theta_j X = i alpha V^x X +
    # beta V^o X, then i V_j^x of it: for element (a, b), j = a gives c_a i (beta_a + i alpha_a) sigma_ab
    term = any(p["terminator"] for p in models)
    tt = t(np.concatenate([x[1] * x[2][None, :] for x in ng])).view(-1, N, 1) if term else None
    if term:  # V^x leaves the diagonal alone
        tt = tt * (1.0 - torch.eye(N, device=dev, dtype=torch.float64))
    half = (-0.5 * ngt + 0.5 * dampt)

    sig = torch.zeros(total + 1, N, N, dtype=torch.complex128, device=dev)
    roots = t(np.array(off[:-1]))
    if state is not None:
        sig[:total] = t(state)

    def rhs(s):
        flat = s.reshape(-1)
        A = torch.matmul(Bt, s[:total])
        # up links act through V^x: nothing on the diagonal (the row and column parts cancel there)
        A += wut * flat[gu].view(total, N, N)
        A += wdt * flat[gd].view(total, N, N)
        A += half * s[:total]
        if tt is not None:
            A += tt * s[:total]
        return A + A.mH

    trap = t(np.stack([p["trap"] for p in models]) * 1e-3)
    rec = t(np.stack([p["recomb"] for p in models]) * 1e-3)
    return sig, rhs, roots, total, off, trap, rec


def _exact_run(models, rho0s, steps, every, state=None):
    N = models[0]["N"]
    sig, rhs, roots, total, off, trap, rec = _exact_system(models, state)
    if state is None:
        sig[roots] = torch.as_tensor(np.stack(rho0s), device=sig.device)
    h = 1.0
    acc = torch.zeros(3, len(models), dtype=torch.float64, device=sig.device)  # eta, loss, int eta
    pops, eta, loss = [], [], []

    def pop(s):
        return torch.diagonal(s[roots], dim1=1, dim2=2).real

    def row():
        pops.append(pop(sig).clone())
        eta.append(acc[0].clone())
        loss.append(acc[1].clone())

    def flux(s, e):
        q = pop(s)
        return torch.stack([(q * trap).sum(1), (q * rec).sum(1), e])

    tmp = torch.zeros_like(sig)
    row()
    for k in range(steps):
        k1, f1 = rhs(sig), flux(sig, acc[0])
        tmp[:total] = sig[:total] + 0.5 * h * k1
        f2 = flux(tmp, acc[0] + 0.5 * h * f1[0])
        k2 = rhs(tmp)
        tmp[:total] = sig[:total] + 0.5 * h * k2
        f3 = flux(tmp, acc[0] + 0.5 * h * f2[0])
        k3 = rhs(tmp)
        tmp[:total] = sig[:total] + h * k3
        f4 = flux(tmp, acc[0] + h * f3[0])
        k4 = rhs(tmp)
        k1 += 2.0 * k2
        k1 += 2.0 * k3
        k1 += k4
        sig[:total] += (h / 6.0) * k1
        acc = acc + (h / 6.0) * (f1 + 2.0 * f2 + 2.0 * f3 + f4)
        if (k + 1) % every == 0:
            row()
    t_end = steps * h
    host = lambda x: x.cpu().numpy()  # noqa: E731
    return {"pops": host(torch.stack(pops, 1)), "eta": host(torch.stack(eta, 1)), "loss": host(torch.stack(loss, 1)),
            "rho": host(sig[roots]), "state": host(sig[:total]), "acc": host(acc),
            "t_mean": host(t_end * acc[0] - acc[2])}


def exact(case, seed):
    models = _models(case, seed)
    if case["kind"] == "single":
        p, rho0, steps = models[0]
        state = None
        if case["resume"]:
            state = _start_state(p["N"], math.comb(p["N"] + p["K"], p["K"]), seed, rho0)
        r = _exact_run([p], [rho0], steps, case["every"], state)
        out = {"pops": r["pops"][0], "eta": r["eta"][0]}
        if case["resume"]:
            out["state"] = r["state"]
            out["extra"] = r["acc"][:2, 0]
        else:
            out["rho"] = r["rho"][0]
            out["t_mean"] = np.asarray(r["t_mean"][0])
        return out
    if case["kind"] == "scan":
        r = _exact_run([m[0] for m in models], [m[1] for m in models], case["steps"], case["every"])
        return {"pops": r["pops"], "eta": r["eta"]}
    res = [_exact_run([p], [rho0], steps, case["every"]) for p, rho0, steps in models]
    return {k: np.concatenate([r[k][0].reshape(-1) for r in res]) for k in ("pops", "eta", "loss")}
