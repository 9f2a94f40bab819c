"""The framework's performance cases: what its users run, through its public entry points.

Every case is a dict of plain values; "kind" selects the call:

    sweep     restart of an ensemble from given fields, one Metropolis sweep, the equal-time
              correlation functions of every chain and its fields (one step of a bin)
    logdet    log|det(1 + B(beta,0))| and its derivatives on fixed field configurations
    energy    the energy estimator and its derivatives on fixed field configurations
    tau       lattice-resolved time-displaced correlation functions of every chain
    su2       as "sweep", in the SU(2) charge decoupling (complex)

Chains differ in lattice, U and number of slices where a field lists several values: chain c takes
lattice c * n / chains and the entries c mod n of the other lists.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1704_00131_gb300 import dqmc
from paper_1704_00131_gb300 import workloads as wl


def listed():
    return [
        # the smallest call: one chain of the 4x4 example, where launches and barriers count
        {"name": "sweep_4x4_one_chain_fp64", "kind": "sweep", "precision": "fp64", "lattices": "square 4x4", "chains": 1,
         "U": "4", "slices": "20", "dtau": 0.1, "n_wrap": 10, "delay_k": 16, "tp": 0.0, "mu": 0.0, "field": "ising"},
        # an ordinary single run at full precision: one chain of the 6x6-cell honeycomb lattice
        {"name": "sweep_honeycomb_one_chain_fp64", "kind": "sweep", "precision": "fp64", "lattices": "honeycomb 6x6",
         "chains": 1, "U": "4", "slices": "40", "dtau": 0.1, "n_wrap": 10, "delay_k": 16, "tp": 0.0, "mu": 0.0,
         "field": "ising"},
        # a parameter scan at full precision: 64 chains of the 8x8 lattice
        {"name": "sweep_8x8_64_chains_fp64", "kind": "sweep", "precision": "fp64", "lattices": "square 8x8", "chains": 64,
         "U": "2 4", "slices": "40", "dtau": 0.1, "n_wrap": 10, "delay_k": 16, "tp": 0.0, "mu": 0.0, "field": "ising"},
        # float pairs without tensor cores on many chains of the 8x8 lattice
        {"name": "sweep_8x8_128_chains_mixed", "kind": "sweep", "precision": "mixed", "lattices": "square 8x8",
         "chains": 128, "U": "2 4", "slices": "40", "dtau": 0.1, "n_wrap": 10, "delay_k": 16, "tp": 0.0, "mu": 0.0,
         "field": "ising"},
        # odd sizes, a doped lattice and the four-valued fields, stabilised more often
        {"name": "sweep_9x7_40_chains_hs4_mixed", "kind": "sweep", "precision": "mixed", "lattices": "square 9x7",
         "chains": 40, "U": "4", "slices": "30", "dtau": 0.1, "n_wrap": 5, "delay_k": 8, "tp": -0.2, "mu": -0.5,
         "field": "hs4"},
        # the production batch: 256 chains of uneven lattices and temperatures on the tensor cores
        {"name": "sweep_8x8_12x12_256_chains_mixed_tc", "kind": "sweep", "precision": "mixed_tc",
         "lattices": "square 8x8, square 12x12", "chains": 256, "U": "2 4 4", "slices": "40 80", "dtau": 0.1,
         "n_wrap": 10, "delay_k": 16, "tp": 0.0, "mu": 0.0, "field": "ising"},
        # the largest lattice: 32 chains of 16x16 with next-nearest hopping and doping
        {"name": "sweep_16x16_32_chains_mixed_tc", "kind": "sweep", "precision": "mixed_tc", "lattices": "square 16x16",
         "chains": 32, "U": "4", "slices": "20", "dtau": 0.05, "n_wrap": 10, "delay_k": 32, "tp": -0.2, "mu": -0.5,
         "field": "ising"},
        # differentiation, the log-weight: 64 configurations of the 8x8 lattice
        {"name": "logdet_backward_8x8_64", "kind": "logdet", "lattices": "square 8x8", "chains": 64, "U": "4",
         "slices": "40", "dtau": 0.1, "n_wrap": 10, "tp": 0.0, "mu": 0.0, "field": "ising"},
        # differentiation, the energy estimator on the same ensemble
        {"name": "energy_backward_8x8_64", "kind": "energy", "lattices": "square 8x8", "chains": 64, "U": "4",
         "slices": "40", "dtau": 0.1, "n_wrap": 10, "tp": 0.0, "mu": 0.0, "field": "ising"},
        # the time-displaced measurement at the end of a sweep, all imaginary times and displacements
        {"name": "tau_corr_8x8_32_chains", "kind": "tau", "precision": "mixed", "lattices": "square 8x8", "chains": 32,
         "U": "4", "slices": "40", "dtau": 0.1, "n_wrap": 10, "tp": 0.0, "mu": 0.0, "field": "ising"},
        # the SU(2) decoupling, the precision example's lattice on every SM
        {"name": "su2_4x4_304_chains", "kind": "su2", "lattices": "square 4x4", "chains": 304, "U": "4", "slices": "40",
         "dtau": 0.1, "n_wrap": 10, "tp": 0.0, "mu": 0.0, "field": "hs4"},
    ]


def draw(rng):
    """One more case of the listed kinds: lattices of 4 to 256 sites (odd and even, not square ones among them), 1 to
    256 chains, n_wrap 5 or 10, 2 to 8 stabilisation intervals."""
    kind = rng.choice(["sweep"] * 6 + ["logdet", "energy", "tau", "su2"])
    precision = rng.choice(["fp64", "mixed", "mixed_tc", "mixed_tc"])
    top = {"su2": 36, "logdet": 100, "energy": 81, "tau": 81}.get(kind, {"fp64": 121, "mixed": 196}.get(precision, 256))
    n_wrap = rng.choice([5, 10])
    while True:
        n = math.exp(rng.uniform(math.log(4.0), math.log(top)))
        lx = max(2, round(math.sqrt(n) * rng.uniform(0.7, 1.4)))
        ly = max(2, round(n / lx))
        if not 4 <= lx * ly <= top:
            continue
        name = "square"
        if kind in ("sweep", "logdet") and rng.random() < 0.25 and 2 * lx * ly <= top:
            name = "honeycomb"
        sites = lx * ly * (2 if name == "honeycomb" else 1)
        blocks = rng.randint(2, 8)
        chains = int(round(math.exp(rng.uniform(0.0, math.log(256.0)))))
        slices = blocks * n_wrap
        waves = max(1.0, chains * (1 if kind == "su2" else 2) / 152.0)
        if slices * sites ** 2 * waves <= 40 * 256 ** 2 / (4 if precision == "fp64" or kind != "sweep" else 1):
            break
    doped = rng.random() < 0.3 and name == "square"
    # four-valued fields are the only ones of the SU(2) decoupling; the others mostly take two-valued ones
    case = {"kind": kind, "lattices": f"{name} {lx}x{ly}", "chains": chains, "U": rng.choice(["2", "4", "2 4"]),
            "slices": str(slices), "dtau": rng.choice([0.05, 0.1]), "n_wrap": n_wrap, "tp": -0.2 if doped else 0.0,
            "mu": -0.5 if doped and kind != "su2" else 0.0,
            "field": "hs4" if kind == "su2" or rng.random() < 0.2 else "ising"}
    if kind in ("logdet", "energy"):
        case["U"] = case["U"].split()[-1]
    if kind == "sweep":
        case["precision"] = precision
        case["delay_k"] = rng.choice([8, 16, 16, 24, 32])
    if kind == "tau":
        case["precision"] = rng.choice(["fp64", "mixed", "mixed_tc"])
    return case


# ---- the models and inputs of a case ------------------------------------------------------------
FIELD = {"ising": wl.FIELD_ISING, "hs4": wl.FIELD_HS4}


def _lattice(text, tp, mu):
    name, size = text.split()
    a, b = (int(v) for v in size.split("x"))
    if name == "honeycomb":
        return wl.honeycomb_lattice(a, b, mu=mu), wl.translation_classes_honeycomb(a, b)[:2]
    return wl.square_lattice(a, b, tp=tp, mu=mu), wl.translation_classes_square(a, b)[:2]


def _chains(case):
    """Per chain (lattice index, U, L), and the lattices' (hopping, (class map, number of classes))."""
    lat = [_lattice(t.strip(), case["tp"], case["mu"]) for t in case["lattices"].split(",")]
    Us = [float(u) for u in case["U"].split()]
    Ls = [int(v) for v in case["slices"].split()]
    n = case["chains"]
    return [(c * len(lat) // n, Us[c % len(Us)], Ls[c % len(Ls)]) for c in range(n)], lat


def _fields(case, seed):
    """Seeded uniform field configurations [L, N] of every chain."""
    chains, lat = _chains(case)
    return [wl.random_fields(FIELD[case["field"]], L, lat[i][0].shape[0], 1000003 * seed + c)
            for c, (i, _, L) in enumerate(chains)]


def prepare(case, seed):
    chains, lat = _chains(case)
    fields = _fields(case, seed)
    keys = sorted(set(chains))
    index = [keys.index(k) for k in chains]
    classes = [lat[k[0]][1][0] for k in keys]
    n_class = [lat[k[0]][1][1] for k in keys]
    if case["kind"] == "su2":
        models = [dqmc.Su2Model(lat[i][0], U, case["dtau"], L, case["n_wrap"]) for i, U, L in keys]
        ens = dqmc.Su2Ensemble(models, index, fields=fields, seed=seed)
    else:
        models = [wl.ModelSpec(lat[i][0], U=U, dtau=case["dtau"], L=L, n_wrap=case["n_wrap"],
                               field_type=FIELD[case["field"]]) for i, U, L in keys]
        if case["kind"] in ("logdet", "energy"):
            ens = dqmc.Ensemble(models, [0], precision="fp64")
            fields = np.stack(fields)
        else:
            ens = dqmc.Ensemble(models, index, fields=fields, precision=case["precision"],
                                delay_k=case.get("delay_k", 16), seed=seed)
    return {"kind": case["kind"], "ens": ens, "fields": fields, "classes": classes, "n_class": n_class,
            "n_tau": max(L for _, _, L in chains)}


def run(state):
    ens, kind = state["ens"], state["kind"]
    if kind == "logdet":
        logdet, grad_K, grad_U = ens.logdet_backward(0, state["fields"])
        return {"logdet": logdet, "grad_K": grad_K, "grad_U": grad_U}
    if kind == "energy":
        energy, grad_K, grad_U = ens.energy_backward(0, state["fields"])
        return {"energy": energy, "grad_K": grad_K, "grad_U": grad_U}
    if kind == "tau":
        corr, sign = ens.measure_tau_corr(state["n_tau"], state["classes"], state["n_class"])
        return {"corr": corr, "sign": sign}
    # a restart from the caller's fields, so that every pass sweeps the same configurations
    ens.set_fields(state["fields"], 0)
    if kind == "su2":
        ens.sweep(1)
        corr, phase = ens.measure_corr(state["classes"], state["n_class"])
        return {"corr": np.stack([corr.real, corr.imag], -1), "phase": np.array([phase.real, phase.imag]),
                "fields": np.concatenate([f.ravel() for f in ens.get_fields()[0]])}
    ens.sweep(1, stats=False)
    corr, sign = ens.measure_corr(state["classes"], state["n_class"])
    return {"corr": corr, "sign": sign, "fields": np.concatenate([f.ravel() for f in ens.get_fields()[0]])}


def work(case):
    """Operations of the dense algorithm (a product of two N x N matrices: 2 N^3) and the bytes of the inputs and outputs."""
    chains, lat = _chains(case)
    flops = byts = 0.0
    for i, _, L in chains:
        N, ncls = lat[i][0].shape[0], lat[i][1][1]
        nst, n3 = L // case["n_wrap"], float(lat[i][0].shape[0]) ** 3
        chain = 2 * L * n3 + nst * (8 / 3 + 1) * n3        # slice products, QR with Q, T
        green = (2 + 2 + 2 / 3 + 2 + 2) * n3               # Q^T Q, T T^T, LU, solve, last product
        kind = case["kind"]
        if kind == "tau":
            f = chain + nst * 2 * green + L * 8 * n3
            b = L * N + 8.0 * (L + 1) * ncls * 3
        elif kind == "logdet":
            f = 2 * chain + nst * green + L * 4 * n3
            b = L * N + 8.0 * 2 * (N * N + 2)
        elif kind == "energy":
            f = 2 * chain + nst * 1.5 * green + L * 8 * n3
            b = L * N + 8.0 * 2 * (N * N + 3)
        else:
            # the restart's left chain; per sweep two visits of every slice: a wrap, about half of the proposals
            # accepted with a rank-1 update each, and the chains and G at the stabilisation points
            f = chain + green + 2 * (chain + nst * green) + 2 * L * (4 * n3 + 0.5 * N * 2 * N * N)
            b = 2.0 * L * N + 8.0 * ncls * 4
        flops += f * (4 if kind == "su2" else 2)           # complex arithmetic on one color, or two flavors
        byts += b
    byts += sum(8.0 * k.shape[0] ** 2 for k, _ in lat)
    return {"bytes": byts, "flops": flops}


# ---- the same results in 64 bits ------------------------------------------------------------------
# Green functions come from the block-cyclic space-time matrix M of the slice propagators (rows
# x_0 + P_p x_{p-1} = b_0, x_j - P_j x_{j-1} = b_j): its inverse holds G(tau, tau'), its determinant
# is det(1 + B(beta,0)), and it needs no decomposition of the propagators' products.
DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _cyclic(P):
    """M of the blocks P [..., p, N, N]."""
    p, N = P.shape[-3], P.shape[-1]
    eye = torch.eye(N, dtype=P.dtype, device=P.device).expand(P.shape[:-3] + (N, N))
    if p == 1:
        return eye + P[..., 0, :, :]
    zero = torch.zeros_like(eye)
    rows = []
    for j in range(p):
        row = [zero] * p
        row[j] = eye
        row[(j - 1) % p] = P[..., p - 1, :, :] if j == 0 else -P[..., j - 1, :, :]
        rows.append(torch.cat(row, -1))
    return torch.cat(rows, -2)


def _merge(B, w):
    """Products of w consecutive slice propagators B [..., L, N, N]."""
    out = []
    for j in range(0, B.shape[-3], w):
        P = B[..., j, :, :]
        for q in range(j + 1, min(j + w, B.shape[-3])):
            P = B[..., q, :, :] @ P
        out.append(P)
    return torch.stack(out, -3)


def _green(B, tau, w):
    """G(tau) = (1 + B(tau,0) B(beta,tau))^-1 from the slice propagators, merged in groups of w slices."""
    P = _merge(torch.roll(B, -tau, -3), w)
    N = B.shape[-1]
    M = _cyclic(P)
    rhs = torch.zeros(M.shape[:-1] + (N,), dtype=B.dtype, device=B.device)
    rhs[..., range(N), range(N)] = 1.0
    return torch.linalg.solve(M, rhs)[..., :N, :]


def _uniforms(seed, chain, L, N):
    """(u1, u2) [2, L, N] of sweep 0 (direction, slice, vertex): Philox4x32-10 of (sweep, 2 tau + dir, vertex, 0)."""
    d, t, k = np.meshgrid(np.arange(2), np.arange(1, L + 1), np.arange(N), indexing="ij")
    c = [np.zeros(d.shape, np.uint64), (2 * t + d).astype(np.uint64), k.astype(np.uint64), np.zeros(d.shape, np.uint64)]
    m32 = np.uint64(0xFFFFFFFF)
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) ^ chain
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    w = lambda hi, lo: (((hi << np.uint64(32)) | lo) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
    return w(c[0], c[1]), w(c[2], c[3])


def _propose(f, u1, ising):
    """Proposed fields: the flip, or one of the three other values of (-2, -1, 1, 2) in ascending order."""
    if ising:
        return -f
    vals = np.array([-2, -1, 1, 2])
    at = np.searchsorted(vals, f)
    i = np.minimum(np.floor(3.0 * u1).astype(int), 2)
    return vals[i + (i >= at)]


def _eta(f):
    s6 = math.sqrt(6.0)
    return np.sign(f) * np.where(np.abs(f) == 1, math.sqrt(2 * (3 - s6)), math.sqrt(2 * (3 + s6)))


def _gamma(f):
    return np.where(np.abs(f) == 1, 1 + math.sqrt(6.0) / 3, 1 - math.sqrt(6.0) / 3)


def _sweep64(K, Us, fields, case, seed, ids):
    """One sweep of chains that share a lattice and L, in plain 64-bit arithmetic with an immediate rank-1 update
    per accepted proposal: (G(0) [chains, flavors, N, N], fields [chains, L, N], sign or phase [chains])."""
    su2, ising = case["kind"] == "su2", case["field"] == "ising"
    dt, w = case["dtau"], case["n_wrap"]
    f = np.stack(fields).astype(int)
    n, L, N = f.shape
    u = [_uniforms(seed, c, L, N) for c in ids]
    u1, u2 = np.stack([a for a, _ in u]), np.stack([a for _, a in u])
    lam = np.array([math.acosh(math.exp(0.5 * dt * U)) if ising else math.sqrt(0.5 * dt * U) for U in Us])
    kind = torch.complex128 if su2 else torch.float64
    unit = 1j if su2 else 1.0
    flav = torch.tensor([1.0] if su2 else [1.0, -1.0], dtype=kind, device=DEV)
    val = (lambda a: a) if ising else _eta
    dev = lambda a, t=None: torch.as_tensor(np.ascontiguousarray(a), dtype=t, device=DEV)
    h, V = torch.linalg.eigh(dev(K))
    E = ((V * torch.exp(-dt * h)) @ V.T).to(kind)
    Ei = ((V * torch.exp(dt * h)) @ V.T).to(kind)
    v = unit * flav[:, None, None] * dev(lam[:, None, None] * val(f))[:, None]           # [n, flavors, L, N]
    B = E * torch.exp(v)[..., None, :]
    def fresh(tau, w):
        return _green(B, tau, w)
    def phase():
        if not su2:
            s, _ = torch.linalg.slogdet(_cyclic(_merge(B, w)))
            return torch.sign(s).prod(-1)
        s, _ = torch.linalg.slogdet(_cyclic(_merge(B, w)))
        p = s[:, 0] ** 2 * torch.exp(-v.sum((1, 2, 3)))
        return p / p.abs()
    G, P = fresh(0, w), phase()
    for d in range(2):
        for tau in (range(1, L + 1) if d == 0 else range(L, 0, -1)):
            if d == 0:
                e = torch.exp(v[:, :, tau - 1])
                G = e[..., :, None] * G / e[..., None, :]
            else:
                G = Ei @ G @ E
            fo = f[:, tau - 1]
            fn = _propose(fo, u1[:, d, tau - 1], ising)
            dth = unit * flav[:, None] * dev(lam[:, None] * (val(fn) - val(fo)))[:, None]    # [n, flavors, N]
            delta = torch.exp(dth) - 1.0
            gam = dev(np.ones(fo.shape) if ising else _gamma(fn) / _gamma(fo)).to(kind)
            if su2:
                gam = gam * torch.exp(-dth[:, 0])
            uu = dev(u2[:, d, tau - 1])
            took = torch.zeros(n, N, dtype=torch.bool, device=DEV)
            for k in (range(N) if d == 0 else range(N - 1, -1, -1)):
                Rs = 1.0 + delta[:, :, k] * (1.0 - G[:, :, k, k])
                R = gam[:, k] * (Rs[:, 0] ** 2 if su2 else Rs.prod(-1))
                ok = uu[:, k] < ((P * R).real.abs() / P.real.abs() if su2 else R.abs())
                took[:, k] = ok
                a = G[:, :, :, k] * (-(delta[:, :, k] / Rs) * ok[:, None])[..., None]
                b = -G[:, :, k, :]
                b[:, :, k] += 1.0
                G.view(-1, N, N).baddbmm_(a.reshape(-1, N, 1), b.reshape(-1, 1, N))
                P = torch.where(ok, P * R / (P * R).abs() if su2 else P * torch.sign(R), P)
            f[:, tau - 1] = np.where(took.cpu().numpy(), fn, fo)
            vt = unit * flav[:, None] * dev(lam[:, None] * val(f[:, tau - 1]))[:, None]
            v[:, :, tau - 1] = vt
            B[:, :, tau - 1] = E * torch.exp(vt)[..., None, :]
            if d == 0:
                G = E @ G @ Ei
            else:
                e = torch.exp(-vt)
                G = e[..., :, None] * G / e[..., None, :]
            at = tau if d == 0 else tau - 1
            if at % w == 0:
                G, P = fresh(at % L, w), phase()
    # the final G from shorter products, as far as M's size allows
    return fresh(0, min(w, max(1, w // 5, -(-L * N // 2400)))), f, P


def _classes(x, cls, ncls):
    """Sums of x [..., N, N] over the pair classes."""
    out = torch.zeros(x.shape[:-2] + (ncls,), dtype=x.dtype, device=x.device)
    return out.index_add_(-1, torch.as_tensor(cls, dtype=torch.long, device=x.device), x.flatten(-2))


def _corr(G0, G1, cls, ncls):
    """[chains, classes, 4]: S^z S^z, n n, S^+ S^-, sum_s c^+ c of the two flavors' G(0)."""
    one = torch.eye(G0.shape[-1], dtype=G0.dtype, device=G0.device)
    h0, h1 = one - G0.mT, one - G1.mT
    X = h0 * G0 + h1 * G1
    d0, d1 = G0.diagonal(dim1=-2, dim2=-1), G1.diagonal(dim1=-2, dim2=-1)
    m, r = d1 - d0, 2.0 - d0 - d1
    q = (0.25 * (m[..., :, None] * m[..., None, :] + X), r[..., :, None] * r[..., None, :] + X, h0 * G1, h0 + h1)
    return torch.stack([_classes(x, cls, ncls) for x in q], -1)


def _groups(case):
    chains, lat = _chains(case)
    ids = {}
    for c, (i, U, L) in enumerate(chains):
        ids.setdefault((i, L), []).append(c)
    return chains, lat, ids


def _exact_sweep(case, seed):
    chains, lat, ids = _groups(case)
    fields = _fields(case, seed)
    su2 = case["kind"] == "su2"
    top = max(ncls for _, (_, ncls) in lat)
    corr = np.zeros((len(chains), top, 4), dtype=complex if su2 else float)
    sign = np.zeros(len(chains), dtype=complex if su2 else np.int32)
    out = list(fields)
    for (i, L), cs in ids.items():
        K, (cls, ncls) = lat[i]
        G, f, P = _sweep64(K, [chains[c][1] for c in cs], [fields[c] for c in cs], case, seed, cs)
        corr[cs, :ncls] = _corr(G[:, 0], G[:, -1], cls, ncls).cpu().numpy()
        sign[cs] = P.cpu().numpy()
        for q, c in enumerate(cs):
            out[c] = f[q].astype(np.int8)
    flat = np.concatenate([f.ravel() for f in out])
    if su2:
        return {"corr": np.stack([corr.real, corr.imag], -1), "phase": np.array([sign.real, sign.imag]), "fields": flat}
    return {"corr": corr, "sign": sign, "fields": flat}


def _slices64(case, K, U, f):
    """The slice propagators [flavors, L, N, N] of one configuration as a function of K [flavors, N, N] and U."""
    if case["field"] == "ising":
        v = torch.acosh(torch.exp(0.5 * case["dtau"] * U)) * torch.as_tensor(f, dtype=torch.float64, device=DEV)
    else:
        v = torch.sqrt(0.5 * case["dtau"] * U) * torch.as_tensor(_eta(f), dtype=torch.float64, device=DEV)
    E = torch.linalg.matrix_exp(-case["dtau"] * K)
    return E[:, None] * torch.exp(torch.stack([v, -v]))[..., None, :]


def _exact_gradient(case, seed):
    chains, lat = _chains(case)
    K0 = torch.as_tensor(lat[0][0], device=DEV)
    N, dlog = K0.shape[0], case["kind"] == "logdet"
    res = {"logdet" if dlog else "energy": [], "grad_K": [], "grad_U": []}
    for f in _fields(case, seed):
        K = K0.expand(2, N, N).clone().requires_grad_(True)
        U = torch.tensor([chains[0][1]] * 2, dtype=torch.float64, device=DEV, requires_grad=True)
        # U of each flavor on its own: the first row of flavor 0, the second of flavor 1
        B = torch.stack([_slices64(case, K, U[s], f)[s] for s in range(2)])
        if dlog:
            val = torch.linalg.slogdet(_cyclic(_merge(B, 2)))[1]
            total = val.sum()
        else:
            G = _green(B, 0, 2)
            n = 1.0 - G.diagonal(dim1=-2, dim2=-1)
            kin = (K * (torch.eye(N, device=DEV) - G.mT)).sum()
            pot = 0.5 * U.sum() * (n[0] * n[1]).sum()
            val, total = torch.stack([kin, pot, n.sum(), kin + pot]), kin + pot
        gK, gU = torch.autograd.grad(total, (K, U))
        both = gK + gK.mT
        both = both - torch.diag_embed(gK.diagonal(dim1=-2, dim2=-1))
        res["logdet" if dlog else "energy"].append(val.detach().cpu().numpy())
        res["grad_K"].append(both.cpu().numpy())
        res["grad_U"].append((gU if dlog else gU.sum()).cpu().numpy())
    return {k: np.stack(v) for k, v in res.items()}


def _exact_tau(case, seed):
    chains, lat, _ = _groups(case)
    nt = max(L for _, _, L in chains)
    top = max(ncls for _, (_, ncls) in lat)
    corr, sign = np.zeros((len(chains), nt + 1, top, 3)), np.zeros(len(chains), dtype=np.int32)
    for c, f in enumerate(_fields(case, seed)):
        i, U, L = chains[c]
        K, (cls, ncls) = lat[i]
        N = K.shape[0]
        B = _slices64(case, torch.as_tensor(K, device=DEV).expand(2, N, N), torch.tensor(U, dtype=torch.float64, device=DEV), f)
        M = _cyclic(B)
        sign[c] = int(torch.linalg.slogdet(M)[0].prod().item())
        X = torch.linalg.inv(M).reshape(2, L, N, L, N)
        one = torch.eye(N, dtype=torch.float64, device=DEV)
        Gt0 = torch.cat([X[:, :, :, 0], (one - X[:, 0, :, 0])[:, None]], 1)
        G0t = torch.cat([X[:, 0].transpose(1, 2), -X[:, 0, :, 0][:, None]], 1)
        G0t[:, 0] -= one
        n = 1.0 - torch.stack([X[:, t % L, :, t % L].diagonal(dim1=-2, dim2=-1) for t in range(L + 1)], 1)
        Xc = (-G0t.mT * Gt0).sum(0)
        m, r = n[0] - n[1], n[0] + n[1]
        q = (Gt0.sum(0), 0.25 * (m[:, :, None] * m[0][None, None] + Xc), r[:, :, None] * r[0][None, None] + Xc)
        corr[c, :L + 1, :ncls] = torch.stack([_classes(x, cls, ncls) for x in q], -1).cpu().numpy()
    return {"corr": corr, "sign": sign}


def exact(case, seed):
    chains, lat = _chains(case)
    size = max(lat[i][0].shape[0] * L for i, _, L in chains)
    cost = sum(L * lat[i][0].shape[0] for i, _, L in chains)
    if case["kind"] in ("logdet", "energy"):
        return _exact_gradient(case, seed) if size <= 6000 else None
    if case["kind"] == "tau":
        return _exact_tau(case, seed) if size <= 4000 and len(chains) <= 64 else None
    return _exact_sweep(case, seed) if size <= 12000 and cost <= 2500000 else None
