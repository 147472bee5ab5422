"""Workloads of the FTKomega path, each through the package's public entry points.

What a program does with this package: multiply the Hamiltonian into vectors
(``Context.hv``), iterate a typical state (``Context.tpq_step``, or
``ftk_tpq_step_noalloc`` on its own buffers), solve for Green's functions on a
grid of shifts (``Context.shifted_cocg``), do all of it for one spectrum, or
work in the momentum sectors of the cluster (``Sector``). The clusters are the
named honeycomb tori, the couplings K = -1 and |J| <= 0.3, and the vectors
random complex Gaussian states (the paper's typical states), as in the tests,
the benchmark and the server's job stream. Solves run to the residuals of
parity runs: at a loose one the truncation of the Krylov space, not the
arithmetic, would decide the digits of a result.
"""
import functools
import math

import numpy as np
import torch

import paper_1802_02854_gb300 as ftk
from ftk_inputs import characters, log_temperatures, named, omega_grid, relabel, translations

K = -1.0
SZ = 2   # the z component in apply_op


def _ell(J):
    """The iteration constant l of a job: 1/2, or more where l - H/N needs it
    (three bonds on two sites, the largest eigenvalue of a bond)."""
    return max(0.5, 1.5 * max((J + K) / 4, (J - K) / 4, -(3 * J + K) / 4))


def listed():
    return [
        # one product on the 12-site cluster: the smallest call, launches and latency
        {"name": "hv_fp64_n12", "kind": "hv", "prec": "fp64", "n": 12, "rhs": 1, "J": 0.1, "order": False},
        # a block of four right-hand sides on the server's usual cluster
        {"name": "hv_fp64_n18_b4", "kind": "hv", "prec": "fp64", "n": 18, "rhs": 4, "J": 0.1, "order": False},
        # the benchmark's cluster in the default precision, sites in the suggested order
        {"name": "hv_fp64_n24", "kind": "hv", "prec": "fp64", "n": 24, "rhs": 1, "J": 0.05, "order": True},
        # single precision: a small block, and the largest ordinary product
        {"name": "hv_fp32_n20_b2", "kind": "hv", "prec": "fp32", "n": 20, "rhs": 2, "J": -0.2, "order": False},
        {"name": "hv_fp32_n26", "kind": "hv", "prec": "fp32", "n": 26, "rhs": 1, "J": 0.1, "order": True},
        # a typical state iterated as a server job does it, and its last vector
        {"name": "tpq_n16", "kind": "tpq", "n": 16, "steps": 61, "every": 20, "J": 0.1},
        # one iteration on the caller's own buffers, at full size
        {"name": "step_n24", "kind": "step", "n": 24, "J": 0.05, "order": True},
        # the small cluster's whole spectrum: states, probes, Green's functions, temperatures
        {"name": "spectrum_n12", "kind": "spectrum", "n": 12, "prec": "fp64", "steps": 61, "every": 20, "J": 0.1,
         "shifts": 256, "eta": 0.1, "tol": 1e-11, "temps": 32},
        # Green's functions of one job in double precision
        {"name": "solve_fp64_n18", "kind": "solve", "prec": "fp64", "n": 18, "rhs": 2, "J": 0.2, "shifts": 256,
         "eta": 0.1, "tol": 1e-11, "order": False},
        # a block of four in the double-float mode, the server's and the benchmark's solver
        {"name": "solve_df_n18_b4", "kind": "solve", "prec": "df", "n": 18, "rhs": 4, "J": 0.1, "shifts": 512,
         "eta": 0.1, "tol": 1e-11, "order": False},
        # the benchmark's solver on its cluster, at a broad line so that it ends in a second
        {"name": "solve_df_n24", "kind": "solve", "prec": "df", "n": 24, "rhs": 1, "J": 0.05, "shifts": 1024,
         "eta": 0.3, "tol": 1e-9, "order": True},
        # a momentum sector: states, probe to the shifted sector, Green's function
        {"name": "sector_n20", "kind": "sector", "n": 20, "steps": 21, "every": 20, "J": 0.1, "momentum": 1,
         "probe": 2, "shifts": 256, "eta": 0.1, "tol": 1e-10},
    ]


def draw(rng):
    J = round(rng.uniform(-0.3, 0.3), 4)
    kind = rng.choice(["hv", "hv", "hv", "tpq", "step", "spectrum", "solve", "solve", "sector"])
    if kind == "hv":
        prec = rng.choice(["fp64", "fp32"])
        n = rng.choice([10, 12, 14, 16, 18, 20, 24] + ([26] if prec == "fp32" else []))
        rhs = rng.choice([1, 1, 2, 4, 8]) if n <= 20 else 1
        return {"kind": kind, "prec": prec, "n": n, "rhs": rhs, "J": J, "order": rng.random() < 0.5}
    if kind == "tpq":
        return {"kind": kind, "n": rng.choice([8, 10, 12, 14, 16, 18]), "steps": rng.randint(20, 81),
                "every": rng.choice([10, 20]), "J": J}
    if kind == "step":
        return {"kind": kind, "n": rng.choice([12, 14, 16, 18, 20, 24]), "J": J, "order": rng.random() < 0.5}
    if kind == "spectrum":
        return {"kind": kind, "n": rng.choice([8, 10, 12, 14]), "prec": rng.choice(["fp64", "df"]),
                "steps": rng.randint(41, 81), "every": 20, "J": J, "shifts": rng.randint(64, 512),
                "eta": round(rng.uniform(0.1, 0.3), 3), "tol": 1e-11, "temps": rng.randint(16, 64)}
    if kind == "solve":
        return {"kind": kind, "prec": rng.choice(["fp64", "df"]), "n": rng.choice([12, 14, 16, 18, 20]),
                "rhs": rng.choice([1, 2, 3, 4]), "J": J, "shifts": rng.randint(64, 1024),
                "eta": round(rng.uniform(0.1, 0.3), 3), "tol": rng.choice([1e-10, 1e-11]), "order": rng.random() < 0.5}
    return {"kind": kind, "n": rng.choice([8, 12, 16, 18, 20]), "steps": rng.randint(21, 41), "every": 20, "J": J,
            "momentum": rng.randint(0, 3), "probe": rng.randint(0, 3), "shifts": rng.randint(64, 512),
            "eta": round(rng.uniform(0.1, 0.3), 3), "tol": 1e-10}


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=None)
def _cluster(n, prec=None):
    """The named cluster; with a precision, its sites in the suggested order."""
    cl = named(n)
    if prec is None:
        return cl
    perm, _ = ftk.ftk_suggest_order(n, cl.bonds, ftk.PRECISIONS[prec], 1)
    return relabel(cl, perm)


def _cluster_of(case):
    if not case.get("order"):
        return _cluster(case["n"])
    return _cluster(case["n"], case.get("prec", "fp64"))


def _gaussian(n, rows, seed, dtype=torch.complex128):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return torch.randn(rows, 1 << n, dtype=dtype, device="cuda", generator=g)


def _state(n, seed):
    v = _gaussian(n, 1, seed)[0]
    return v / torch.linalg.vector_norm(v)


def _spin_z(cl, q, v):
    """N^{-1/2} sum_l exp(i q.R_l) S^z_l v."""
    ph = np.exp(1j * (cl.pos @ np.asarray(q))) / math.sqrt(cl.n_sites)
    f = torch.zeros(1, dtype=torch.complex128, device=v.device)
    for p in ph:   # site l is bit l: the upper half of every doubling has it up
        f = torch.cat([f - 0.5 * complex(p), f + 0.5 * complex(p)])
    return f * v


def _probes(case, cl, seed):
    """Probe vectors S^z_q psi of typical states, one momentum after the other."""
    lam = []
    for j in range(case["rhs"]):
        psi = _state(case["n"], seed * 64 + j)
        lam.append(_spin_z(cl, cl.momenta[(1 + j) % len(cl.momenta)], psi))
    return lam


def _sector_state(case, cl, seed):
    """A typical state and its characters in the starting sector."""
    perms, vecs = translations(cl)
    q = cl.momenta[case["momentum"] % len(cl.momenta)]
    return _state(case["n"], seed), perms, vecs, q, cl.momenta[case["probe"] % len(cl.momenta)]


# ------------------------------------------------------------------ passes
def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    cl = _cluster_of(case)
    st = {"case": case, "cl": cl}
    if kind == "hv":
        dt = torch.complex128 if case["prec"] == "fp64" else torch.complex64
        v = _gaussian(n, case["rhs"], seed, dt)
        st["v"] = v if case["rhs"] > 1 else v[0]
        st["ctx"] = ftk.Context(cl, K, case["J"], case["prec"], max_rhs=case["rhs"])
    elif kind == "step":
        st["v"] = _state(n, seed)
        st["out"] = torch.empty_like(st["v"])
    elif kind == "tpq":
        st["v"] = _state(n, seed)
        st["ctx"] = ftk.Context(cl, K, case["J"], "fp64", n_saved=case["steps"] // case["every"] + 1)
    elif kind == "spectrum":
        shells = (case["steps"] - 1) // case["every"] + 1
        st["v"] = _state(n, seed)
        st["ctx"] = ftk.Context(cl, K, case["J"], case["prec"], max_rhs=4, n_saved=shells)
        st["shells"] = min(shells, 4)
        st["omega"] = omega_grid(-2.0, 2.0, case["shifts"])
        st["temps"] = log_temperatures(0.5, 2.0, case["temps"])
    elif kind == "solve":
        st["ctx"] = ftk.Context(cl, K, case["J"], case["prec"], max_rhs=4 if case["rhs"] == 3 else case["rhs"])
        probes = _probes(case, cl, seed)
        torch.cuda.synchronize()   # the context copies them on its own stream
        for j, lam in enumerate(probes):
            st["ctx"].set_probe(j, lam.data_ptr(), 0.0)
        st["omega"] = omega_grid(-3.0, 3.0, case["shifts"])
    else:
        psi, perms, vecs, q, p = _sector_state(case, cl, seed)
        st["ctx"] = ftk.Context(cl, K, case["J"], "fp64")
        st["src"] = ftk.Sector(st["ctx"], perms, characters(vecs, q), n_slots=5)
        st["dst"] = ftk.Sector(st["ctx"], perms, characters(vecs, q + p), n_slots=4)
        st["probe"] = p
        st["src"].project(psi.cpu().numpy(), 0)
        st["v"] = st["src"].get(0)
        st["shifts"] = omega_grid(-3.0, 3.0, case["shifts"]) + 1j * case["eta"]
    return st


def run(st):
    case, cl = st["case"], st["cl"]
    kind = case["kind"]
    if kind == "hv":
        return st["ctx"].hv(st["v"])
    if kind == "step":
        stats = ftk.ftk_tpq_step_noalloc(case["n"], cl.bonds, K, case["J"], _ell(case["J"]), st["v"].data_ptr(),
                                         st["out"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return {"out": st["out"], "stats": np.array(stats)}
    ctx = st["ctx"]
    if kind == "tpq":
        ctx.set_state(st["v"].data_ptr(), _ell(case["J"]))
        u, logq, h2 = ctx.tpq_step(case["steps"], case["every"])
        return {"u": u, "logq": logq, "h2": h2, "state": ctx.get_vector(0)}
    if kind == "spectrum":
        ctx.set_state(st["v"].data_ptr(), _ell(case["J"]))
        u, _, _ = ctx.tpq_step(case["steps"], case["every"])
        for s in range(st["shells"]):
            ctx.apply_op(s, SZ, cl.momenta[1], s)
        G, _, _ = ctx.shifted_cocg(list(range(st["shells"])), st["omega"], case["eta"], tol=case["tol"])
        S, _ = ctx.spectrum(G, st["temps"])
        return {"u": u, "G": G, "S": S}
    if kind == "solve":
        G, _, _ = ctx.shifted_cocg(list(range(case["rhs"])), st["omega"], case["eta"], tol=case["tol"])
        return G
    src, dst = st["src"], st["dst"]
    src.set(0, st["v"])
    u, logq, _ = src.tpq(0, 1, _ell(case["J"]), case["steps"], case["every"], 2)
    src.apply_sz((2 + (case["steps"] - 1) // case["every"]), dst, 0, st["probe"])
    G, _ = dst.green(0, st["shifts"], tol=case["tol"])
    return {"u": u, "logq": logq, "G": G}


# -------------------------------------------------------------------- work
def _product(n, size, rhs=1):
    """Bytes and operations of one product: each amplitude read once and
    written once, a multiply-add per bond (3/2 a site) and the diagonal."""
    dim = rhs * 2 ** n
    return 2 * dim * size, dim * 4 * (1.5 * n + 1)


# iterations of a solve, by what the residual's decrease per step depends on:
# the line width against the width of the spectrum
def _iterations(case):
    return max(20, int(2.0 * math.log(1.0 / case["tol"]) / case["eta"]))


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "hv":
        b, f = _product(n, 16 if case["prec"] == "fp64" else 8, case["rhs"])
        return {"bytes": b, "flops": f}
    b, f = _product(n, 16)
    if kind == "step":
        return {"bytes": b, "flops": f + 12 * 2 ** n}
    if kind == "tpq":
        return {"bytes": case["steps"] * b, "flops": case["steps"] * (f + 12 * 2 ** n)}
    # per iteration of a solve: the product, and the recurrence over three
    # vectors, the probe and the result
    step_b, step_f = b + 5 * 16 * 2 ** n, f + 44 * 2 ** n
    if kind == "spectrum":
        it = 4 * _iterations(case)
        return {"bytes": case["steps"] * b + it * step_b, "flops": case["steps"] * f + it * step_f}
    if kind == "solve":
        it = case["rhs"] * _iterations(case)
        return {"bytes": it * step_b, "flops": it * step_f}
    it, part = _iterations(case), 2.0 / n   # a sector holds about 2/N of the states
    return {"bytes": part * (case["steps"] * b + it * 3 * b), "flops": part * (case["steps"] * f + it * (f + 16 * 2 ** n))}


# ------------------------------------------------------------- plain 64 bits
def _hamiltonian(cl, J):
    """The product with H in complex128 by views: bond (i, j) pairs the two
    bits as axes of their own."""
    n, terms = cl.n_sites, []
    for i, j, g in cl.bonds.tolist():
        lo, hi = min(i, j), max(i, j)
        par, anti = ((K / 4, K / 4 + J / 2), (-K / 4, K / 4 + J / 2), (0.0, J / 2))[g]
        d = J / 4 + (K / 4 if g == 2 else 0.0)
        c = torch.tensor([[par, anti], [anti, par]], dtype=torch.float64, device="cuda").reshape(1, 2, 1, 2, 1)
        dg = torch.tensor([[d, -d], [-d, d]], dtype=torch.float64, device="cuda").reshape(1, 2, 1, 2, 1)
        terms.append(((1 << (n - 1 - hi), 2, 1 << (hi - lo - 1), 2, 1 << lo), c, dg))

    def apply(v):
        out = torch.zeros_like(v)
        for shape, c, dg in terms:
            a, o = v.view(shape), out.view(shape)
            o += c * a.flip(1, 3)
            o += dg * a
        return out

    return apply


def _resolvent(H, lam, z, tol=1e-13, most=4000):
    """<lam|(z - H)^{-1}|lam> by the Lanczos continued fraction, until the
    residual of every shift is below tol."""
    z = torch.as_tensor(np.asarray(z), dtype=torch.complex128, device="cuda")
    norm = torch.linalg.vector_norm(lam)
    q, p, b = lam / norm, torch.zeros_like(lam), 0.0
    G = torch.zeros_like(z)
    d, y = None, torch.ones_like(z)
    for j in range(most):
        w = H(q)
        a = torch.vdot(q, w).real
        w = w - a * q - b * p
        if j == 0:
            d = z - a
        else:
            y = y * b / d
            d = z - a - b * b / d
        G = G + y * y / d
        b = torch.linalg.vector_norm(w)
        if j % 8 == 7 and float((b * (y / d).abs()).max()) < tol:
            break
        p, q = q, w / b
    return (G * norm ** 2).cpu().numpy()


def _iterate(H, n, psi, steps, ell):
    """Typical-state iteration: u_k, log Q_k, <H^2>_k and psi_0 .. psi_steps."""
    u, logq, h2, out, lq = [], [], [], [], 0.0
    for _ in range(steps):
        w = H(psi)
        u.append(float(torch.vdot(psi, w).real) / n)
        h2.append(float(torch.vdot(w, w).real))
        logq.append(lq)
        out.append(psi)
        psi = ell * psi - w / n
        q = torch.linalg.vector_norm(psi)
        lq += math.log(float(q))
        psi = psi / q
    out.append(psi)
    return np.array(u), np.array(logq), np.array(h2), out


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    cl = _cluster_of(case)
    H = _hamiltonian(cl, case["J"])
    if kind == "hv":
        v = _gaussian(n, case["rhs"], seed, torch.complex128 if case["prec"] == "fp64" else torch.complex64)
        out = torch.stack([H(r.to(torch.complex128)) for r in v])
        return out if case["rhs"] > 1 else out[0]
    if kind == "solve":
        z = omega_grid(-3.0, 3.0, case["shifts"]) + 1j * case["eta"]
        return np.stack([_resolvent(H, lam, z) for lam in _probes(case, cl, seed)])
    if kind == "sector":
        # in the full basis: the sector's part of the state, its iteration and
        # the probe's Green's function are those of the sector
        psi, perms, vecs, q, p = _sector_state(case, cl, seed)
        x = torch.arange(1 << n, device="cuda")
        part = torch.zeros_like(psi)
        for pm, ch in zip(perms, characters(vecs, q)):
            y = torch.zeros_like(x)
            for l, m in enumerate(pm.tolist()):
                y |= ((x >> l) & 1) << m
            moved = torch.empty_like(psi)
            moved[y] = psi
            part += complex(np.conj(ch)) * moved
        part /= torch.linalg.vector_norm(part)
        u, logq, _, states = _iterate(H, n, part, case["steps"], _ell(case["J"]))
        lam = _spin_z(cl, p, states[(case["steps"] - 1) // case["every"] * case["every"]])
        z = omega_grid(-3.0, 3.0, case["shifts"]) + 1j * case["eta"]
        return {"u": u, "logq": logq, "G": _resolvent(H, lam, z)}
    psi = _state(n, seed)
    if kind == "step":
        w = H(psi)
        out = _ell(case["J"]) * psi - w / n
        stats = [float(torch.vdot(psi, w).real) / n, float(torch.vdot(w, w).real), float(torch.linalg.vector_norm(out))]
        return {"out": out, "stats": np.array(stats)}
    u, logq, h2, states = _iterate(H, n, psi, case["steps"], _ell(case["J"]))
    if kind == "tpq":
        return {"u": u, "logq": logq, "h2": h2, "state": states[-1].cpu().numpy()}
    om = omega_grid(-2.0, 2.0, case["shifts"])
    G = []
    for s in range(min((case["steps"] - 1) // case["every"] + 1, 4)):
        k = s * case["every"]
        lam = _spin_z(cl, cl.momenta[1], states[k])
        G.append(_resolvent(H, lam, om + n * u[k] + 1j * case["eta"]))
    return {"u": u, "G": np.stack(G), "S": None}
