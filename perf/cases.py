"""Performance cases: what a user of the library has it do, through the Python entry points.

Every case is one whole call sequence of a program that holds a handle (or a batch) and
has a new Hamiltonian in device memory (lattices: COO triplets in host memory): load F,
run a purification scheme, read the density into a device tensor the program owns.

kinds
  dense    one Hamiltonian F = Q diag(lambda) Q^T on a handle: float64 (the default
           precision) or mixed, spectral ends given or estimated, beta or trace rule,
           with or without a float64 refinement step
  gap      the same with the gap edges unknown: estimated first, then used
  batch    many Hamiltonians of uneven size purified together in one call
  serve    requests that arrive while others run (continuous batching)
  lattice  a sparse tight-binding Hamiltonian on a block-sparse handle
"""
import math
import random

import numpy as np
import torch

import paper_1101_0265_gb300 as P
from paper_1101_0265_gb300 import inputs as I

DEV = "cuda"
HAAR_MAX_N = 4096  # larger dense inputs are rotated by reflections (the QR would take seconds)


# ---- the cases -------------------------------------------------------------------------

def _dense(name, n, occ, gap, scheme, precision, tol, bounds="given", rule="beta", refine=0):
    c = {"kind": "dense", "n": n, "occ": occ, "gap": gap, "scheme": scheme, "precision": precision,
         "tol": tol, "bounds": bounds, "rule": rule, "refine": refine}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the small float64 configuration: a molecule's worth of basis functions, default options
        _dense("fp64_tc_n256", 256, 0.5, 1e-1, "TC_SF", "fp64", 1e-12),
        # an ordinary float64 run of ragged size whose spectral ends are not known
        _dense("fp64_mu_n1000_est", 1000, 0.37, 1e-2, "FIXED_MU_SF", "fp64", 1e-12, bounds="estimated"),
        # the large float64 configuration, the reference the mixed path is judged against
        _dense("fp64_tc_n4096", 4096, 0.5, 1e-1, "TC_SF", "fp64", 1e-12),
        # the smallest mixed calls (a request of the serving stream run alone): launches count
        _dense("mixed_tc_n200", 200, 0.5, 3e-2, "TC_SF", "mixed", 1e-9),
        # an ordinary mixed run, odd size, closed by a float64 step that sets the idempotency
        _dense("mixed_mu_n1101_refine", 1101, 0.4, 1e-3, "FIXED_MU_SF", "mixed", 1e-9, refine=1),
        # the headline workload: n = 4096, spectral ends estimated inside the call
        _dense("mixed_tc_n4096_est", 4096, 0.25, 1e-2, "TC_SF", "mixed", 1e-9, bounds="estimated"),
        # the largest size of the serving stream, fixed mu
        _dense("mixed_mu_n8192", 8192, 0.5, 1e-3, "FIXED_MU_SF", "mixed", 1e-9),
        # branch by the trace, gap unknown: the classic trace-correcting scheme
        _dense("mixed_trace_n2000", 2000, 0.5, 1e-2, "TC_MONO", "mixed", 1e-4, rule="trace"),
        # gap edges found first, then a run with them
        {"name": "gap_n1500", "kind": "gap", "n": 1500, "occ": 0.45, "gap": 3e-2, "scheme": "TC_SF",
         "precision": "mixed", "tol": 1e-9},
        # a batch over the configured size and gap ranges
        {"name": "batch_48", "kind": "batch", "count": 48, "n_lo": 64, "n_hi": 2048, "mix": 1},
        # ten requests, two admitted per call
        {"name": "serve_10", "kind": "serve", "count": 10, "n_lo": 128, "n_hi": 4096, "mix": 1},
        # a cubic lattice with a wide gap, where the density stays sparse
        {"name": "lattice_24", "kind": "lattice", "L": 24, "onsite": 3.0},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["fp64"] * 3 + ["mixed"] * 4 + ["gap", "batch", "serve", "lattice"])
    occ, gap = round(rng.uniform(0.25, 0.7), 3), float("%.3g" % _log(rng, 1e-3, 1e-1))
    bounds = rng.choice(["given", "estimated"])
    scheme = rng.choice(["TC_SF", "FIXED_MU_SF"])
    if kind == "fp64":
        return _dense("", int(_log(rng, 100, 2500)), occ, gap, scheme, "fp64", 1e-12, bounds=bounds)
    if kind == "mixed":
        rule = rng.choice(["beta", "beta", "beta", "trace"])
        if rule == "trace":
            scheme, gap = "TC_MONO", max(gap, 1e-2)
        return _dense("", int(_log(rng, 128, 8192)), occ, gap, scheme, "mixed", 1e-4 if rule == "trace" else 1e-9,
                      bounds=bounds, rule=rule)
    if kind == "gap":
        return {"kind": "gap", "n": int(_log(rng, 200, 3000)), "occ": occ, "gap": max(gap, 1e-2), "scheme": scheme,
                "precision": rng.choice(["mixed", "mixed", "fp64"]), "tol": 1e-9}
    if kind == "lattice":
        return {"kind": "lattice", "L": rng.choice([8, 12, 16, 20, 24]), "onsite": round(rng.uniform(0.5, 6.0), 2)}
    return {"kind": kind, "count": rng.randint(8, 48) if kind == "batch" else rng.randint(4, 12),
            "n_lo": 64 if kind == "batch" else 128, "n_hi": 2048 if kind == "batch" else 4096,
            "mix": rng.randrange(1 << 20)}


def _members(case):
    """The sizes, occupations, gaps and schemes of a batch or a request stream: part of the case."""
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["count"]):
        n = int(round(_log(r, case["n_lo"], case["n_hi"])))
        scheme = "TC_SF" if case["kind"] == "batch" or r.random() < 0.5 else "FIXED_MU_SF"
        out.append({"n": n, "occ": r.uniform(0.3, 0.7), "gap": _log(r, 1e-3, 1e-1), "scheme": scheme})
    return out


# ---- inputs ----------------------------------------------------------------------------

def _nocc(c):
    return min(max(int(round(c["occ"] * c["n"])), 2), c["n"] - 2)


def _spectrum(c, seed):
    """Ascending eigenvalues: nocc in [-1, -gap/2], the rest in [gap/2, 1], the four edges present."""
    r, n, nocc, g = np.random.default_rng(seed), c["n"], _nocc(c), c["gap"]
    lo = np.concatenate([[-1.0, -g / 2], r.uniform(-1.0, -g / 2, nocc - 2)])
    hi = np.concatenate([[g / 2, 1.0], r.uniform(g / 2, 1.0, n - nocc - 2)])
    return torch.from_numpy(np.sort(np.concatenate([lo, hi]))).to(DEV)


def _rotations(c, seed):
    """What rotates the diagonal: a Haar Q, or the vectors of three reflections when n is large."""
    n = c["n"]
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    if n > HAAR_MAX_N:
        v = torch.randn(3, n, generator=g, dtype=torch.float64, device=DEV)
        return v / torch.linalg.vector_norm(v, dim=1, keepdim=True)
    q, r = torch.linalg.qr(torch.randn(n, n, generator=g, dtype=torch.float64, device=DEV))
    return q * torch.sign(torch.diagonal(r))[None, :]


def _rotated(diag, rot):
    """Q diag Q^T, symmetric."""
    if rot.shape[0] == rot.shape[1]:
        F = (rot * diag[None, :]) @ rot.T
    else:
        F = torch.diag(diag)
        for v in rot:
            w = F @ v
            F = F - 2.0 * torch.outer(v, w) - 2.0 * torch.outer(w, v) + 4.0 * torch.dot(v, w) * torch.outer(v, v)
    return (0.5 * (F + F.T)).contiguous()


def _hamiltonian(c, seed):
    return _rotated(_spectrum(c, seed), _rotations(c, seed))


def _projector(c, seed):
    """The exact density: the projector on the nocc lowest eigenvectors."""
    occ = torch.zeros(c["n"], dtype=torch.float64, device=DEV)
    occ[:_nocc(c)] = 1.0
    return _rotated(occ, _rotations(c, seed))


def _lattice(case, seed):
    return I.lattice_hamiltonian(case["L"], instance=seed, onsite=case["onsite"])


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("dense", "gap"):
        s["F"] = _hamiltonian(case, seed)
        s["D"] = torch.empty_like(s["F"])
        opt = {} if kind == "gap" else {"branch_rule": case["rule"], "refine_fp64": case["refine"]}
        s["handle"] = P.Purifier(precision=case["precision"], **opt)
    elif kind in ("batch", "serve"):
        s["members"] = _members(case)
        s["F"] = [_hamiltonian(m, seed + 1000 * i) for i, m in enumerate(s["members"])]
        s["D"] = [torch.empty_like(F) for F in s["F"]]
        s["handle"] = P.Batch()
    else:
        s["lattice"] = _lattice(case, seed)
        s["D"] = torch.empty((s["lattice"].n,) * 2, dtype=torch.float64, device=DEV)
        s["handle"] = P.Purifier(precision="mixed", block_sparse=True, trunc_tau=1e-6)
    return s


# ---- one pass --------------------------------------------------------------------------

def _run_dense(s):
    c, p = s["case"], s["handle"]
    g = c["gap"]
    edges = {} if c["kind"] == "gap" or c.get("rule") == "trace" else {"homo": -g / 2, "lumo": g / 2}
    if c.get("bounds") == "given":
        edges.update(lmin=-1.0, lmax=1.0)
    mu = None if c["kind"] == "gap" else 0.0
    p.set_hamiltonian(s["F"], nocc=_nocc(c), mu=mu, **edges)
    if c["kind"] == "gap":
        p.estimate_gap()
    p.run(c["scheme"], c["tol"])
    p.density(s["D"])
    st = p.stats()
    return {"D": s["D"], "trace": st["trace"], "iterations": st["iterations"],
            "multiplications": st["multiplications"], "lmin": st["lmin"], "lmax": st["lmax"]}


def _add(s, i):
    m = s["members"][i]
    return s["handle"].add(s["F"][i], _nocc(m), -1.0, 1.0, -m["gap"] / 2, m["gap"] / 2, scheme=m["scheme"], tol=1e-9,
                           mu=0.0)


def _run_batch(s):
    b = s["handle"]
    ids = [_add(s, i) for i in range(len(s["F"]))]
    b.run()
    for i, D in zip(ids, s["D"]):
        b.density(i, D)
    traces = [b.stats(i)["trace"] for i in ids]
    for i in ids:
        b.release(i)
    return {"D": s["D"], "trace": np.array(traces)}


def _run_serve(s):
    b = s["handle"]
    waiting, live, traces = list(range(len(s["F"]))), {}, [0.0] * len(s["F"])
    while waiting or live:
        for i in waiting[:2]:
            live[_add(s, i)] = i
        waiting = waiting[2:]
        b.advance(4)
        for k, i in list(live.items()):
            if b.done(k):
                b.density(k, s["D"][i])
                traces[i] = b.stats(k)["trace"]
                b.release(k)
                del live[k]
    return {"D": s["D"], "trace": np.array(traces)}


def _run_lattice(s):
    l, p = s["lattice"], s["handle"]
    p.set_hamiltonian_coo(l.n, l.rows, l.cols, l.vals, nocc=l.nocc, mu=0.0, homo=-l.gap_bound, lumo=l.gap_bound)
    p.run("TC_SF", 1e-9, 300)
    p.density(s["D"])
    st = p.stats()
    return {"D": s["D"], "trace": st["trace"], "iterations": st["iterations"], "lmin": st["lmin"], "lmax": st["lmax"]}


def run(state):
    kind = state["case"]["kind"]
    return {"dense": _run_dense, "gap": _run_dense, "batch": _run_batch, "serve": _run_serve,
            "lattice": _run_lattice}[kind](state)


# ---- what one pass cannot do without ---------------------------------------------------

def _purification_work(c, tol, refine=0):
    """F read and D written once; n^2 (n + 1) flop for each symmetric product of the schedule."""
    n, g = c["n"], c["gap"]
    its = P.schedule(c["scheme"], -1.0, 1.0, 0.0, -g / 2, g / 2, tol)["iterations"]
    products = (2 if c["scheme"].startswith("FIXED_MU") else 1) * its + 2 * refine
    return 16.0 * n * n, float(products) * n * n * (n + 1)


def work(case):
    kind = case["kind"]
    if kind == "lattice":
        # the triplets (a site has itself and six neighbours) in, the density out; the products'
        # flops depend on which blocks survive truncation and are not counted
        n = case["L"] ** 3
        return {"bytes": 24.0 * 7 * n + 8.0 * n * n, "flops": 0.0}
    if kind in ("batch", "serve"):
        each = [_purification_work(m, 1e-9) for m in _members(case)]
    else:
        each = [_purification_work(case, case["tol"], case.get("refine", 0))]
    return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}


# ---- the same in 64 bits, without the library ------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind in ("dense", "gap"):
        return {"D": _projector(case, seed), "trace": float(_nocc(case))}
    if kind in ("batch", "serve"):
        ms = _members(case)
        return {"D": [_projector(m, seed + 1000 * i) for i, m in enumerate(ms)],
                "trace": np.array([float(_nocc(m)) for m in ms])}
    if case["L"] > 12:  # the eigendecomposition takes too long
        return None
    l = _lattice(case, seed)
    F = torch.from_numpy(l.dense()).to(DEV)
    w, V = torch.linalg.eigh(F)
    V = V[:, :l.nocc]
    return {"D": V @ V.T, "trace": float(l.nocc)}
