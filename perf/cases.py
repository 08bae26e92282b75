"""The work a user of the library has it do, case by case: inputs, one pass and
its exact result.

Every case is one call sequence through the public binding
(paper_2604_16118_gb300.native / .problem).  Hamiltonians are the repository's
synthetic workloads: "chain" (spinless orbitals with a random one-body matrix and
eight Cholesky vectors), "hubbard" (open 1D chain, t = 1, U = 4, half filling)
and "molecule" (two spins, random Cholesky integrals).  Iterates have the
block dims of a fresh random iterate and standard-normal entries, scaled per
block so that norms stay near one.
"""
import itertools
import math

import numpy as np
import torch

from paper_2604_16118_gb300 import native as nat
from paper_2604_16118_gb300 import problem

_CTX = {}


def _context():
    """The one solver context of a program (device 0, torch's default stream)."""
    if "ctx" not in _CTX:
        _CTX["ctx"] = nat.Context(0)
    return _CTX["ctx"]


def _graph_context():
    """A second context on a stream of its own, which recorded plans need."""
    if "graph" not in _CTX:
        _CTX["stream"] = torch.cuda.Stream()
        _CTX["graph"] = nat.Context(0, _CTX["stream"].cuda_stream)
    return _CTX["graph"]


# ---- the cases ---------------------------------------------------------------

def listed():
    return [
        # <x, H x> of a small chain: the Rayleigh quotient a user reads after every step; launch latency
        {"name": "rayleigh_chain12_r32", "kind": "rayleigh", "system": "chain", "sites": 12, "rank": 32},
        # H x recompressed, one small operator application (wide MPO, small sectors)
        {"name": "apply_chain12_r32", "kind": "apply", "system": "chain", "sites": 12, "rank": 32, "tol": 1e-4,
         "cap": 0},
        # H x at the headline size: Hubbard chain of 32 orbitals (64 sites), iterate at its cap 256
        {"name": "apply_hubbard32_r256", "kind": "apply", "system": "hubbard", "sites": 32, "rank": 256, "tol": 1e-4,
         "cap": 256},
        # the preconditioner's sum S x (seven or more scaled copies) brought back to low rank
        {"name": "precondition_chain14_r48", "kind": "precondition", "system": "chain", "sites": 14, "rank": 48,
         "tol": 1e-4},
        # recompression of an iterate with wide charge sectors (up to 252): the large factorisations
        {"name": "truncate_chain20_r1024", "kind": "truncate", "system": "chain", "sites": 20, "rank": 1024,
         "tol": 1e-3},
        # recompression of an odd-sized, ragged iterate (odd sites and filling)
        {"name": "truncate_chain17_r203", "kind": "truncate", "system": "chain", "sites": 17, "rank": 203,
         "tol": 1e-2},
        # one solver step (Alg. 2) of the small chain from a random iterate
        {"name": "step_chain12_r32", "kind": "step", "system": "chain", "sites": 12, "rank": 32},
        # one solver step of a Hubbard chain at half filling: some twenty truncations of mid-sized sectors
        {"name": "step_hubbard10_r48", "kind": "step", "system": "hubbard", "sites": 10, "rank": 48},
        # 48 independent molecule-like problems as one recorded graph: iterates written, replayed, read back
        {"name": "plan_molecules48", "kind": "plan", "problems": 48, "first": 3, "last": 5},
        # FP64 product on the tensor cores (eight integer slices)
        {"name": "gemm_ozaki_2048", "kind": "ozaki", "m": 2048, "n": 2048, "k": 2048},
        # split-precision product of the mixed-precision contraction, ragged
        {"name": "gemm_split_3000x1100x700", "kind": "split", "m": 3000, "n": 1100, "k": 700},
        # loss and gradients of the learned controller's network on a training batch
        {"name": "mlp_grad_8192", "kind": "mlp", "batch": 8192},
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rayleigh", "apply", "apply", "precondition", "truncate", "truncate", "step", "plan", "ozaki",
                       "split", "mlp"])
    if kind == "ozaki":
        return {"kind": kind, "m": _spread(rng, 64, 2048), "n": _spread(rng, 64, 2048), "k": _spread(rng, 64, 2048)}
    if kind == "split":
        return {"kind": kind, "m": _spread(rng, 64, 3000), "n": _spread(rng, 64, 3000), "k": _spread(rng, 32, 2000)}
    if kind == "mlp":
        return {"kind": kind, "batch": _spread(rng, 16, 8192)}
    if kind == "plan":
        return {"kind": kind, "problems": rng.randint(8, 60), "first": 3, "last": rng.randint(4, 5)}
    if kind in ("rayleigh", "apply"):
        system = rng.choice(["chain", "hubbard"])
        c = {"kind": kind, "system": system,
             "sites": rng.randint(8, 14) if system == "chain" else _spread(rng, 4, 32),
             "rank": _spread(rng, 8, 64) if system == "chain" else _spread(rng, 16, 256)}
        if kind == "apply":
            c["tol"] = rng.choice([1e-3, 1e-4])
            c["cap"] = rng.choice([0, c["rank"]]) if system == "chain" else c["rank"]
        return c
    if kind == "precondition":
        return {"kind": kind, "system": "chain", "sites": rng.randint(8, 16), "rank": _spread(rng, 8, 64),
                "tol": rng.choice([1e-3, 1e-4])}
    if kind == "truncate":
        sites = rng.randint(10, 19)
        return {"kind": kind, "system": "chain", "sites": sites, "rank": _spread(rng, 16, 512),
                "tol": rng.choice([1e-2, 1e-3])}
    system = rng.choice(["chain", "hubbard"])
    return {"kind": "step", "system": system, "sites": rng.randint(8, 12) if system == "chain" else rng.randint(3, 9),
            "rank": _spread(rng, 8, 32) if system == "chain" else _spread(rng, 8, 48)}


# ---- systems and iterates ------------------------------------------------------

def _species(spin, n_orb):
    return [0, 1] * n_orb if spin else [0] * n_orb


def _step_charge(q, species, s):
    return (q[0] + s, q[1]) if species == 0 else (q[0], q[1] + s)


def _bonds(species, target, r):
    """Sector dims of a fresh random iterate of rank at most r (bsmps_mps_random_size)."""
    K = len(species)
    tot = [species.count(0), species.count(1)]
    out, left = [], [0, 0]
    for b in range(K + 1):
        if b:
            left[species[b - 1]] += 1
        n = {}
        for q0 in range(max(0, target[0] - tot[0] + left[0]), min(target[0], left[0]) + 1):
            for q1 in range(max(0, target[1] - tot[1] + left[1]), min(target[1], left[1]) + 1):
                lc = math.comb(left[0], q0) * math.comb(left[1], q1)
                rc = math.comb(tot[0] - left[0], target[0] - q0) * math.comb(tot[1] - left[1], target[1] - q1)
                n[(q0, q1)] = (lc, rc)
        dims = {q: min(v) for q, v in n.items()}
        if sum(dims.values()) > r:
            w = sum(lc * rc for lc, rc in n.values())
            dims = {q: min(lc, rc, r * lc * rc // w) for q, (lc, rc) in n.items()}
        out.append({q: d for q, d in dims.items() if d > 0})
    return out


def _blocks(species, bonds):
    """(site, left sector, sigma, rows, cols) of every block, in the library's flat order."""
    for t, sp in enumerate(species):
        for q in sorted(bonds[t]):
            for s in (0, 1):
                q2 = _step_charge(q, sp, s)
                if q2 in bonds[t + 1]:
                    yield t, q, s, bonds[t][q], bonds[t + 1][q2]


def _iterate(species, bonds, rng):
    return np.concatenate([(rng.standard_normal(m * n) / math.sqrt(2.0 * n)) for _, _, _, m, n in
                           _blocks(species, bonds)])


def _sym(rng, n, scale):
    g = rng.standard_normal((n, n))
    return scale * (np.triu(g) + np.triu(g, 1).T)


def _system(case, seed):
    """Integrals, Cholesky vectors and particle numbers of the case's Hamiltonian."""
    n = case["sites"]
    if case["system"] == "hubbard":
        h = np.zeros((n, n))
        p = np.arange(n - 1)
        h[p, p + 1] = h[p + 1, p] = -1.0
        eri = np.zeros((n, n, n, n))
        p = np.arange(n)
        eri[p, p, p, p] = 4.0
        n_up, n_dn = (n + 1) // 2, n // 2
        gamma = problem.hubbard_shift(h, n_up, n_dn, margin=1.0)
        return {"spin": 1, "n_orb": n, "h": h, "eri": eri, "target": (n_up, n_dn), "gamma": gamma, "chol": None}
    rng = np.random.default_rng(1000 + seed)
    p = np.arange(n)
    h = _sym(rng, n, 1.0) * np.exp(-np.abs(p[:, None] - p[None, :]) / 3.0)
    h[p, p] += 0.5 * p
    chol = [_sym(rng, n, 0.1) for _ in range(8)]
    eri = sum(np.einsum("pq,rs->pqrs", c, c) for c in chol)
    gamma = problem.cholesky_shift(h, eri, n // 2, 0, 0, margin=1.0)
    return {"spin": 0, "n_orb": n, "h": h, "eri": eri, "target": (n // 2, 0), "gamma": gamma, "chol": chol}


def _theta(S):
    n = sum(S["target"])
    th = problem.theta_diagonal(S["h"], S["eri"], S["spin"], n, S["gamma"])
    lo, hi = problem.spectrum_bounds(th, S["spin"], *S["target"])
    return th, lo, hi


def _input(case, seed):
    S = _system(case, seed)
    S["species"] = _species(S["spin"], S["n_orb"])
    S["bonds"] = _bonds(S["species"], S["target"], case["rank"])
    S["values"] = _iterate(S["species"], S["bonds"], np.random.default_rng(seed))
    S["valid"] = [sorted(d) for d in _bonds(S["species"], S["target"], 1 << 40)]
    S["room"] = _room(case, S)
    return S


def _import(ctx, S):
    return nat.mps_import(ctx, S["n_orb"], S["spin"], S["target"][0], S["target"][1], S["bonds"], S["values"])


def _mpo(ctx, S):
    return nat.mpo_from_integrals(ctx, S["h"], S["eri"], S["spin"], sum(S["target"]), S["gamma"])


def _room(case, S):
    """The largest result: the iterate's own size for a truncation, the exact ranks of a chain, four times the
    iterate for a capped result of a long chain."""
    if case["kind"] == "truncate":
        return len(S["values"])
    if S["spin"]:
        return 4 * len(S["values"])
    full = _bonds(S["species"], S["target"], 1 << 40)
    return sum(m * n for _, _, _, m, n in _blocks(S["species"], full))


def _whole(S, bonds, values):
    """An iterate as arrays whose shapes the case alone decides: the dims of all sectors (0 where a sector is
    gone) and the blocks in flat order, zeros after the last."""
    dims = np.array([d.get(q, 0) for d, v in zip(bonds, S["valid"]) for q in v], dtype=np.int64)
    cores = np.zeros(S["room"])
    cores[:len(values)] = values
    return {"bonds": dims, "cores": cores}


# ---- prepare, run ----------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("ozaki", "split"):
        # factors with rows and columns of different scales, as the carries of a sweep have
        rng = np.random.default_rng(seed)
        a = rng.standard_normal((case["m"], case["k"])) * np.exp(rng.uniform(-2, 2, (case["m"], 1)))
        b = rng.standard_normal((case["k"], case["n"])) * np.exp(rng.uniform(-2, 2, (1, case["n"])))
        return {"case": case, "A": torch.from_numpy(a).cuda(), "B": torch.from_numpy(b).cuda(),
                "C": torch.empty((case["m"], case["n"]), dtype=torch.float64, device="cuda")}
    if kind == "mlp":
        widths, params, x, t = _mlp_input(case, seed)
        return {"case": case, "net": nat.MLP(_context(), widths, params), "x": x, "t": t}
    if kind == "plan":
        ctx = _graph_context()
        Ws, xs, values = [], [], []
        for i in range(case["problems"]):
            S = _molecule(case, seed, i)
            Ws.append(nat.mpo_from_integrals(ctx, S["h"], S["eri"], 1, sum(S["target"]), S["gamma"]))
            xs.append(_import(ctx, S))
            values.append(S["values"])
        return {"case": case, "xs": xs, "values": values,
                "plan": nat.ZipupPlan(ctx, Ws, xs, [-1.0] * len(xs))}
    S = _input(case, seed)
    ctx = _context()
    st = {"case": case, "S": S}
    if kind in ("rayleigh", "apply", "step"):
        st["W"] = _mpo(ctx, S)
    if kind == "step":
        # the constants of Alg. 2: those of the small random chain, alpha_0 from the interval
        th, lo, hi = _theta(S)
        alpha0, c = problem.alpha0_and_c(0.1, lo, 0.234, 1.881)
        st["p"] = nat.make_precond(th, lo, hi, 0.1, alpha0)
        st["params"] = nat.solver_params(c, 2.0, tau=1e-10, r_max=case["rank"])
        return st
    st["x"] = _import(ctx, S)
    norm = math.sqrt(nat.dot(ctx, st["x"], st["x"]))
    if kind == "apply":
        st["tol"] = case["tol"] * abs(nat.dot(ctx, st["x"], st["x"], st["W"], -0.5)) / norm
    if kind == "precondition":
        th, lo, hi = _theta(S)
        alpha0, _ = problem.alpha0_and_c(0.1, lo, 0.234, 1.881)
        st["p"] = nat.make_precond(th, lo, hi, 0.1, alpha0)
        st["tol"] = case["tol"] * norm * alpha0
    if kind == "truncate":
        st["tol"] = case["tol"] * norm
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ozaki":
        return nat.gemm_ozaki(_context(), state["A"], state["B"], state["C"], 8)
    if kind == "split":
        return nat.gemm_tf32x3(_context(), state["A"], state["B"], state["C"])
    if kind == "mlp":
        loss, grad = state["net"].loss_grad(state["x"], state["t"])
        return {"loss": np.float32(loss), "grad": grad}
    if kind == "plan":
        for x, v in zip(state["xs"], state["values"]):
            x.write(v)
        state["plan"].launch()
        return [y.export() for y in state["plan"].outputs]
    ctx = _context()
    if kind == "rayleigh":
        return {"energy": nat.dot(ctx, state["x"], state["x"], state["W"], -0.5),
                "norm2": nat.dot(ctx, state["x"], state["x"])}
    S = state["S"]
    if kind == "apply":
        y, _ = nat.apply_H(ctx, state["W"], state["x"], shift=-0.5, tol=state["tol"], r_max=case["cap"])
        return _whole(S, y.bonds(), y.export())
    if kind in ("precondition", "truncate"):
        x = nat.precondition(ctx, state["p"], state["x"])[0] if kind == "precondition" else state["x"]
        y, dropped, _ = nat.truncate(ctx, x, state["tol"])
        return dict(_whole(S, y.bonds(), y.export()), discarded=dropped)
    y, info = nat.eigensolve_step(ctx, state["W"], state["p"], state["params"], nat.solver_state(), _import(ctx, S))
    return dict(_whole(S, y.bonds(), y.export()), **{k: info[k] for k in ("lambda", "rho", "lambda_star")})


def _molecule(case, seed, i):
    """Problem i of a batch: molecule-like integrals, orbitals cycling over the case's range, exact ranks."""
    n = case["first"] + i % (case["last"] - case["first"] + 1)
    rng = np.random.default_rng(100000 + 1000 * seed + i)
    p = np.arange(n)
    off = _sym(rng, n, 0.05) * np.exp(-np.abs(p[:, None] - p[None, :]) / 6.0)
    np.fill_diagonal(off, 0.0)
    h = off + np.diag(np.linspace(-2.0, 2.0, n))
    eri = sum(np.einsum("pq,rs->pqrs", c, c) for c in (_sym(rng, n, 0.1) for _ in range(2 * n)))
    target = ((n + 1) // 2, n // 2)
    S = {"spin": 1, "n_orb": n, "h": h, "eri": eri, "target": target, "species": _species(1, n),
         "gamma": problem.cholesky_shift(h, eri, target[0], target[1], 1, margin=1.0)}
    S["bonds"] = _bonds(S["species"], target, 512)
    S["values"] = _iterate(S["species"], S["bonds"], rng)
    return S


def _mlp_input(case, seed):
    widths = [128, 256, 256, 256, 2]
    rng = np.random.default_rng(seed)
    parts = []
    for i in range(len(widths) - 1):
        parts.append(rng.standard_normal(widths[i] * widths[i + 1]) * math.sqrt(2.0 / widths[i]))
        parts.append(0.01 * rng.standard_normal(widths[i + 1]))
    params = np.concatenate(parts).astype(np.float32)
    x = rng.standard_normal((case["batch"], 128)).astype(np.float32)
    t = np.tanh(x @ (rng.standard_normal((128, 2)).astype(np.float32) / 12.0))
    return widths, params, x, t


# ---- what a pass cannot do without --------------------------------------------------

def _sweep_flops(species, bonds):
    """QR of every stacked sector left to right and of every sector's row right to left (thin, 4 m n k each)."""
    fl = 0.0
    for t, sp in enumerate(species):
        rows = {}
        for q, d in bonds[t].items():
            cols = 0
            for s in (0, 1):
                q2 = _step_charge(q, sp, s)
                if q2 in bonds[t + 1]:
                    rows[q2] = rows.get(q2, 0) + d
                    cols += bonds[t + 1][q2]
            fl += 4.0 * d * cols * min(d, cols)
        for q2, m in rows.items():
            n = bonds[t + 1][q2]
            fl += 4.0 * m * n * min(m, n)
    return fl


def work(case):
    """Bytes of the inputs and the results; flops of the products, or of one QR in each direction of a sweep."""
    kind = case["kind"]
    if kind in ("ozaki", "split"):
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8.0 * (m * k + k * n + m * n), "flops": 2.0 * m * n * k}
    if kind == "mlp":
        widths = [128, 256, 256, 256, 2]
        mac = sum(a * b for a, b in zip(widths, widths[1:]))
        return {"bytes": 4.0 * (case["batch"] * 130 + 2 * mac), "flops": 2.0 * case["batch"] * (3 * mac - 128 * 256)}
    if kind == "plan":
        by = fl = 0.0
        for i in range(case["problems"]):
            n = case["first"] + i % (case["last"] - case["first"] + 1)
            sp = _species(1, n)
            b = _bonds(sp, ((n + 1) // 2, n // 2), 512)
            by += 8.0 * 2 * sum(m * c for _, _, _, m, c in _blocks(sp, b))
            fl += _sweep_flops(sp, b)
        return {"bytes": by, "flops": fl}
    spin = case["system"] == "hubbard"
    sp = _species(spin, case["sites"])
    n = case["sites"]
    b = _bonds(sp, ((n + 1) // 2, n // 2) if spin else (n // 2, 0), case["rank"])
    size = sum(m * c for _, _, _, m, c in _blocks(sp, b))
    fl = _sweep_flops(sp, b)
    if kind == "rayleigh":
        return {"bytes": 8.0 * size, "flops": 8.0 * sum(m * c * max(m, c) for _, _, _, m, c in _blocks(sp, b))}
    return {"bytes": 16.0 * size, "flops": fl}


# ---- exact results in plain numpy ------------------------------------------------------

def _unflatten(species, bonds, values):
    cores, pos = [{} for _ in species], 0
    for t, q, s, m, n in _blocks(species, bonds):
        cores[t][(q, s)] = values[pos:pos + m * n].reshape(m, n)
        pos += m * n
    return cores


def _cut(sv, tol2, cap):
    """How many of the pooled (value, sector, index) stay; squares dropped by the tolerance and by the cap."""
    sv = sorted(sv, key=lambda v: (-v[0], v[1], v[2]))
    keep, acc = len(sv), 0.0
    while keep and acc + sv[keep - 1][0] ** 2 <= tol2:
        acc += sv[keep - 1][0] ** 2
        keep -= 1
    while 0 < keep < len(sv) and sv[keep][0] >= sv[keep - 1][0] * (1 - 1e-10):
        keep += 1
    dropped = sum(v[0] ** 2 for v in sv[keep:])
    if cap and keep > cap:
        keep = cap
    count = {}
    for _, q, _ in sv[:keep]:
        count[q] = count.get(q, 0) + 1
    return count, dropped


def _truncate(species, bonds, cores, eps, cap):
    """Left QR sweep, right SVD sweep with the pooled cut at every bond."""
    K = len(species)
    cores = [dict(c) for c in cores]
    bonds = [dict(b) for b in bonds]
    for t in range(K - 1):
        stacks = {}
        for (q, s) in sorted(cores[t]):
            stacks.setdefault(_step_charge(q, species[t], s), []).append((q, s))
        new, R = {}, {}
        for q2, keys in stacks.items():
            A = np.vstack([cores[t][k] for k in keys])
            Q, R[q2] = np.linalg.qr(A)
            pos = 0
            for k in keys:
                m = cores[t][k].shape[0]
                new[k] = Q[pos:pos + m]
                pos += m
        cores[t] = new
        cores[t + 1] = {(q, s): R[q] @ B for (q, s), B in cores[t + 1].items() if q in R}
        bonds[t + 1] = {q: r.shape[0] for q, r in R.items()}
    dropped = 0.0
    for t in range(K - 1, 0, -1):
        svd, sv = {}, []
        for q in bonds[t]:
            keys = [(q, s) for s in (0, 1) if (q, s) in cores[t]]
            if not keys:
                continue
            U, S, V = np.linalg.svd(np.hstack([cores[t][k] for k in keys]), full_matrices=False)
            big = np.argmax(np.abs(V), axis=1)
            sign = np.where(V[np.arange(len(S)), big] < 0, -1.0, 1.0)
            svd[q] = (keys, U * S * sign, V * sign[:, None])
            sv += [(v, q, j) for j, v in enumerate(S)]
        count, d = _cut(sv, eps * eps / (K - 1), cap)
        dropped += d
        old, cores[t], US = cores[t], {}, {}
        for q, (keys, us, V) in svd.items():
            k = count.get(q, 0)
            if not k:
                continue
            pos = 0
            for key in keys:
                n = old[key].shape[1]
                cores[t][key] = V[:k, pos:pos + n]
                pos += n
            US[q] = us[:, :k]
        prev = {}
        for (q, s), B in cores[t - 1].items():
            q2 = _step_charge(q, species[t - 1], s)
            if q2 in US:
                prev[(q, s)] = B @ US[q2]
        cores[t - 1] = prev
        bonds[t] = {q: u.shape[1] for q, u in US.items()}
    flat = np.concatenate([cores[t][(q, s)].ravel() for t, q, s, _, _ in _blocks(species, bonds)])
    return bonds, flat, math.sqrt(dropped)


def _hubbard_apply(n_orb, bonds, cores, scalar):
    """(H + scalar) x of the open Hubbard chain with its own operator chain: channels I (nothing placed),
    F (done), N (density waiting for the other spin), (c, s) (a hop of species s waiting for its other end)."""
    K = 2 * n_orb
    unit, z, n = {(0, 0): 1.0, (1, 1): 1.0}, {(0, 0): 1.0, (1, 1): -1.0}, {(1, 1): 1.0}
    up, down = {(1, 0): 1.0}, {(0, 1): 1.0}   # (out, in) -> weight
    hops = [(c, s) for c in (1, -1) for s in (0, 1)]
    delta = {"I": (0, 0), "F": (0, 0), "N": (0, 0)}
    delta.update({(c, s): ((c, 0) if s == 0 else (0, c)) for c, s in hops})
    names = ["I", "F", "N"] + hops
    steps = []
    for t in range(K):
        s, ops = t % 2, [("I", "I", unit), ("F", "F", unit)]
        if t == 0:
            ops.append(("I", "F", {k: scalar for k in unit}))
        ops.append(("I", "N", n) if s == 0 else ("N", "F", {(1, 1): 4.0}))
        for c in (1, -1):
            if t + 2 < K:
                ops.append(("I", (c, s), up if c == 1 else down))
            if t >= 2:
                ops.append(((c, s), "F", {k: -v for k, v in (down if c == 1 else up).items()}))
            ops.append(((c, 1 - s), (c, 1 - s), z))
        steps.append(ops)
    reach = [{"I"}]
    for ops in steps:
        reach.append({b for a, b, _ in ops if a in reach[-1]})
    live = [set() for _ in range(K + 1)]
    live[K] = {"F"}
    for t in range(K - 1, -1, -1):
        live[t] = {a for a, b, _ in steps[t] if b in live[t + 1]} & reach[t]
    off, dims = [], []
    for b in range(K + 1):
        o, d = {}, {}
        for a in names:
            if a in live[b]:
                for q in sorted(bonds[b]):
                    m = (q[0] + delta[a][0], q[1] + delta[a][1])
                    o[(a, q)] = d.get(m, 0)
                    d[m] = d.get(m, 0) + bonds[b][q]
        off.append(o)
        dims.append(d)
    out = [{} for _ in range(K)]
    for t in range(K):
        for a, b, w in steps[t]:
            if a not in live[t] or b not in live[t + 1]:
                continue
            for (q, si), B in cores[t].items():
                q2 = _step_charge(q, t % 2, si)
                for so in (0, 1):
                    if (so, si) not in w:
                        continue
                    m = (q[0] + delta[a][0], q[1] + delta[a][1])
                    m2 = (q2[0] + delta[b][0], q2[1] + delta[b][1])
                    T = out[t].setdefault((m, so), np.zeros((dims[t][m], dims[t + 1][m2])))
                    r, c = off[t][(a, q)], off[t + 1][(b, q2)]
                    T[r:r + B.shape[0], c:c + B.shape[1]] += w[(so, si)] * B
    # sectors that cannot be completed to the target particle numbers go
    target = next(iter(bonds[K]))
    dims[K] = {target: dims[K][target]}
    for t in range(K - 1, -1, -1):
        out[t] = {(m, s): T for (m, s), T in out[t].items() if _step_charge(m, t % 2, s) in dims[t + 1]}
        dims[t] = {m: dims[t][m] for m, _ in out[t]}
    seen = {next(iter(bonds[0]))}
    for t in range(K):
        out[t] = {(m, s): T for (m, s), T in out[t].items() if m in seen}
        dims[t] = {m: d for m, d in dims[t].items() if m in seen}
        seen = {_step_charge(m, t % 2, s) for m, s in out[t]}
    return dims, out


def _dense(species, bonds, cores):
    """All occupation strings of the sector (bit t = site t, ascending) and their amplitudes, spinless."""
    part = {(0, 0): (np.zeros(1, dtype=np.int64), np.ones((1, 1)))}
    for t in range(len(species)):
        nxt = {}
        for (q, s), B in sorted(cores[t].items()):
            if q in part:
                nxt.setdefault(_step_charge(q, 0, s), []).append((part[q][0] | (s << t), part[q][1] @ B))
        part = {q: (np.concatenate([a for a, _ in v]), np.vstack([b for _, b in v])) for q, v in nxt.items()}
    (have, vec), = part.values()
    n = bin(int(have[0])).count("1")
    occ = np.array(sorted(sum(1 << t for t in c) for c in itertools.combinations(range(len(species)), n)))
    full = np.zeros(len(occ))
    full[np.searchsorted(occ, have)] = vec[:, 0]
    return occ, full


def _chain_apply(S, occ, vec, scalar):
    """(H + scalar) v for H = sum (h_pq - 1/2 sum_r (pr|rq)) E_pq + 1/2 sum_g (sum_pq L^g_pq E_pq)^2."""
    K = S["n_orb"]
    def excite(M, v):
        """sum_pq M_pq a_p^* a_q v"""
        out = np.zeros_like(v)
        for q in range(K):
            has = np.flatnonzero((occ >> q) & 1)
            rest = occ[has] & ~(1 << q)
            for p in range(K):
                ok = ((rest >> p) & 1) == 0
                lo, hi = min(p, q), max(p, q)
                between = (rest[ok] >> (lo + 1)) & ((1 << max(0, hi - lo - 1)) - 1)
                par = np.array([bin(int(b)).count("1") & 1 for b in between])
                to = np.searchsorted(occ, rest[ok] | (1 << p))
                np.add.at(out, to, M[p, q] * (1.0 - 2.0 * par) * v[has[ok]])
        return out

    h = S["h"] - 0.5 * sum(c @ c for c in S["chol"])
    y = excite(h, vec) + scalar * vec
    for c in S["chol"]:
        y = y + 0.5 * excite(c, excite(c, vec))
    return y


def _from_dense(K, occ, vec):
    """The MPS whose bonds hold every left occupation string (exact, left-orthogonal)."""
    bonds, cores = [{(0, 0): 1}], []
    where = {0: 0}                       # left string -> row in its sector
    for t in range(K - 1):
        mask = (1 << (t + 1)) - 1
        strings = sorted({int(o) & mask for o in occ}, key=lambda o: (bin(o).count("1"), o))
        nxt, dims = {}, {}
        for o in strings:
            q = (bin(o).count("1"), 0)
            nxt[o] = dims.get(q, 0)
            dims[q] = nxt[o] + 1
        core = {}
        for o in strings:
            s, left = (o >> t) & 1, o & (mask >> 1)
            q, q2 = (bin(left).count("1"), 0), (bin(o).count("1"), 0)
            B = core.setdefault((q, s), np.zeros((bonds[t][q], dims[q2])))
            B[where[left], nxt[o]] = 1.0
        cores.append(core)
        bonds.append(dims)
        where = nxt
    core, mask = {}, (1 << (K - 1)) - 1
    for o, v in zip(occ, vec):
        left = int(o) & mask
        q = (bin(left).count("1"), 0)
        core.setdefault((q, (int(o) >> (K - 1)) & 1), np.zeros((bonds[K - 1][q], 1)))[where[left], 0] = v
    cores.append(core)
    bonds.append({(bin(int(occ[0])).count("1"), 0): 1})
    return bonds, cores


def _inner(cores_a, cores_b, species):
    E = {(0, 0): np.ones((1, 1))}
    for t, sp in enumerate(species):
        F = {}
        for (q, s), B in cores_b[t].items():
            if q in E and (q, s) in cores_a[t]:
                q2 = _step_charge(q, sp, s)
                F[q2] = F.get(q2, 0.0) + cores_a[t][(q, s)].T @ E[q] @ B
        E = F
    return float(sum(v.sum() for v in E.values()))


def _precondition(S, cores, alpha0, lo, hi, th):
    """S x as the list of its terms' cores: S = sum_m (x)_i diag(a, a exp(-beta_m d_i)) (Sec. 4.3)."""
    K, c0 = len(S["species"]), 0.1
    h = math.pi ** 2 / math.log(8.0 * math.sqrt(2.0) / c0 + 1.0)
    lg = abs(math.log(math.sqrt(math.pi) * c0 / 4.0))
    terms = []
    for m in range(-math.ceil((2.0 * lg + math.log(hi / lo)) / h), math.ceil(math.log(lg) / h) + 1):
        a = (h * alpha0 / math.sqrt(math.pi) * math.exp(m * h / 2.0)) ** (1.0 / K)
        f = np.exp(-math.exp(m * h) / lo * th)
        terms.append([{k: B * a * (f[t] if k[1] else 1.0) for k, B in c.items()} for t, c in enumerate(cores)])
    return terms


def _concat(species, terms):
    K = len(species)
    cores = []
    for t in range(K):
        core = {}
        for k in terms[0][t]:
            B = [x[t][k] for x in terms]
            if t == 0:
                core[k] = np.hstack(B)
            elif t == K - 1:
                core[k] = np.vstack(B)
            else:
                m, n = B[0].shape
                core[k] = np.zeros((m * len(B), n * len(B)))
                for i, b in enumerate(B):
                    core[k][i * m:(i + 1) * m, i * n:(i + 1) * n] = b
        cores.append(core)
    bonds = [{(0, 0): 1}]
    for t in range(K):
        bonds.append({_step_charge(q, species[t], s): B.shape[1] for (q, s), B in cores[t].items()})
    return bonds, cores


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "plan"):
        return None   # a whole solver step; cores in a gauge that the operator's channels fix
    if kind in ("ozaki", "split"):
        rng = np.random.default_rng(seed)
        a = rng.standard_normal((case["m"], case["k"])) * np.exp(rng.uniform(-2, 2, (case["m"], 1)))
        b = rng.standard_normal((case["k"], case["n"])) * np.exp(rng.uniform(-2, 2, (1, case["n"])))
        return a @ b
    if kind == "mlp":
        return _mlp_exact(case, seed)
    S = _input(case, seed)
    sp = S["species"]
    cores = _unflatten(sp, S["bonds"], S["values"])
    norm = math.sqrt(_inner(cores, cores, sp))
    scalar = S["gamma"] - 0.5
    if kind in ("rayleigh", "apply"):
        if S["spin"]:
            bonds, out = _hubbard_apply(S["n_orb"], S["bonds"], cores, scalar)
            energy = _inner(cores, out, sp)
        else:
            occ, vec = _dense(sp, S["bonds"], cores)
            y = _chain_apply(S, occ, vec, scalar)
            energy = float(vec @ y)
            bonds, out = _from_dense(S["n_orb"], occ, y)
        if kind == "rayleigh":
            return {"energy": energy, "norm2": norm * norm}
        b, flat, _ = _truncate(sp, bonds, out, case["tol"] * abs(energy) / norm, case["cap"])
        return _whole(S, b, flat)
    if kind == "precondition":
        th, lo, hi = _theta(S)
        alpha0, _ = problem.alpha0_and_c(0.1, lo, 0.234, 1.881)
        bonds, out = _concat(sp, _precondition(S, cores, alpha0, lo, hi, th))
        b, flat, d = _truncate(sp, bonds, out, case["tol"] * norm * alpha0, 0)
    else:
        b, flat, d = _truncate(sp, S["bonds"], cores, case["tol"] * norm, 0)
    return dict(_whole(S, b, flat), discarded=d)


def _mlp_exact(case, seed):
    """Loss and gradients in 64 bits with the weights at their BF16 values."""
    widths, params, x, t = _mlp_input(case, seed)
    w = torch.from_numpy(params).to(torch.bfloat16).double().numpy()
    layers, pos = [], 0
    for i, o in zip(widths, widths[1:]):
        layers.append((w[pos:pos + i * o].reshape(o, i), w[pos + i * o:pos + i * o + o]))
        pos += i * o + o
    h = [x.astype(np.float64)]
    for n, (W, b) in enumerate(layers):
        y = h[-1] @ W.T + b
        h.append(np.maximum(y, 0.0) if n + 1 < len(layers) else y)
    d = h[-1] - t
    loss = float(np.mean(d * d))
    d = 2.0 * d / d.size
    grads = []
    for n in range(len(layers) - 1, -1, -1):
        grads = [(d.T @ h[n]).ravel(), d.sum(axis=0)] + grads
        d = (d @ layers[n][0]) * (h[n] > 0)
    return {"loss": loss, "grad": np.concatenate(grads)}
