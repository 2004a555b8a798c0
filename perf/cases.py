"""Performance cases: what programs that propagate density matrices ask of the library.

A pass is what such a program does with a context it has built: it sets the
field of every trajectory (which restarts the clock), propagates, and reads the
series J, E, q and the final densities (or, with the Crank-Nicolson integrator,
the occupied states).  One case reads spectra and group charges of a finished
propagation instead.  The systems are diamond-Si supercells of the shapes and
sizes of the repository's own workloads (8, 64, 216 and 512 atoms, Gamma and the
shifted 2x2x2 grid) with Gaussian displacements; a case with `light` > 0 gives
that share of the atoms a single s orbital, so the orbital counts are uneven and
N is any number.  Everything a seed changes is an input: positions, prefactors,
start density, field strength and polarisation.

The split form (BF16x3 products, FP32 derivative) is a single-precision
propagation, so its programs keep the series and densities in single precision;
the FP64 forms keep double precision.
"""
import math

import numpy as np
import torch

from paper_2308_09782_gb300 import inputs, vgtb

C_LIGHT = inputs.C_LIGHT
FRAC = np.array([[0.00, 0.00, 0.00], [0.00, 0.50, 0.50], [0.50, 0.00, 0.50], [0.50, 0.50, 0.00],
                 [0.25, 0.25, 0.25], [0.25, 0.75, 0.75], [0.75, 0.25, 0.75], [0.75, 0.75, 0.25]])


def _case(name, form, cells, kgrid, steps, traj="0", field="pulse", sigma=0.05, light=0.0, autotune=0, obs_stride=1,
          frozen=False, delta=False):
    c = {"form": form, "cells": cells, "kgrid": kgrid, "steps": steps, "traj": traj, "field": field, "sigma": sigma,
         "light": light, "autotune": autotune, "obs_stride": obs_stride, "frozen": frozen, "delta": delta}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the unit cell on a k grid under a pulse, full double precision: the smallest run, a check or a
        # convergence study, where launches and latency count
        _case("si8_fp64", "fp64", "1x1x1", "mp2", 100, sigma=0.0),
        # the same in the split form
        _case("si8_split", "split", "1x1x1", "mp2", 200),
        # a small supercell on a k grid in double precision, the reference run of a production study
        _case("si64_fp64", "fp64", "2x2x2", "mp2", 50, sigma=0.03),
        # its split-form twin, with the charges kept at every fourth step
        _case("si64_split", "split", "2x2x2", "mp2", 200, obs_stride=4),
        # a cell with light atoms (one orbital each) in the double-precision delta form: uneven blocks, odd N
        _case("mixed144_fp64_delta", "fp64", "3x3x2", "gamma", 20, light=0.25, delta=True, field="kick"),
        # an orbital count that is no multiple of a tile (N = 864), Gamma only, kick spectrum, split form
        _case("si216_split", "split", "3x3x3", "gamma", 300, field="kick", sigma=0.15),
        # the headline run: 512 atoms at Gamma after a kick, tile schedules timed at create
        _case("si512_split", "split", "4x4x4", "gamma", 250, field="kick", sigma=0.15, autotune=1),
        # the laser experiment: three pulses on one 512-atom cell advance together
        _case("si512_laser_split", "split", "4x4x4", "gamma", 64, traj="0,0,0", sigma=0.15, autotune=1),
        # systems of different sizes and several trajectories in one batch
        _case("batch_split", "split", "2x2x2;3x3x3", "mp2;gamma", 100, traj="0,1,0,1", sigma=0.15, autotune=1),
        # the 512-atom run in double precision, the reference of the split form
        _case("si512_fp64", "fp64", "4x4x4", "gamma", 8, field="kick", sigma=0.03),
        # Crank-Nicolson states of a small supercell on a k grid
        _case("si64_cn", "cn", "2x2x2", "mp2", 12, sigma=0.03),
        # spectra and charge transfer between atom groups of a finished propagation
        _case("si8_post", "post", "1x1x1", "mp2", 1200, field="kick"),
    ]


def draw(rng):
    form = rng.choice(["fp64", "fp64", "split", "split", "split", "cn", "post"])
    if form == "post":
        return _case("", form, rng.choice(["1x1x1", "2x1x1"]), rng.choice(["gamma", "mp2"]), rng.randrange(200, 1200),
                     field="kick", sigma=round(rng.uniform(0.0, 0.15), 3), obs_stride=rng.choice([1, 2, 5]))
    top = {"fp64": 216, "split": 512, "cn": 128}[form]
    while True:  # supercells over the logarithm of the atom count
        want = 8.0 * math.exp(rng.uniform(0.0, math.log(top / 8.0)))
        shape = [rng.randint(1, 4) for _ in range(3)]
        nat = 8 * shape[0] * shape[1] * shape[2]
        if 0.8 * want <= nat <= min(top, 1.25 * want):
            break
    light = round(rng.uniform(0.05, 0.5), 3) if rng.random() < 0.35 and nat <= 216 else 0.0
    kgrid = rng.choice(["gamma", "mp2"]) if nat <= 64 else "gamma"
    n = 4 * nat
    # steps so that a pass stays within the largest listed one
    cap = {"fp64": 2.0e11, "split": 4.0e13, "cn": 1.0e10}[form] / (8.0 * n ** 3 * (8 if kgrid == "mp2" else 1))
    steps = max(2, min(int(cap), rng.randrange(24, 250)))
    if form == "cn":
        steps = min(steps, 24)
    traj = rng.choice(["0", "0", "0,0"]) if form == "split" else "0"
    # amorphous cells are a split-form workload; the double-precision runs here are crystals with thermal displacements
    sigma = round(rng.uniform(0.0, 0.15 if form == "split" or light else 0.034), 3)
    return _case("", form, "x".join(str(s) for s in shape), kgrid, steps, traj=traj, field=rng.choice(["pulse", "kick"]),
                 sigma=sigma, light=light, autotune=rng.choice([0, 1]) if form == "split" else 0,
                 obs_stride=rng.choice([1, 1, 3]), frozen=rng.random() < 0.15 and form != "cn",
                 delta=form == "fp64" and rng.random() < 0.25)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _two_centre(d, v, onsite):
    """Two-centre sp3 blocks [n, 4, 4] and their gradients [3, n, 4, 4] at distance vectors d [n, 3]."""
    r = np.sqrt((d * d).sum(1))
    zero = r == 0.0
    u = d / np.where(zero, 1.0, r)[:, None]
    f = v[None, :] * np.exp(-r / inputs.R_DECAY)[:, None]
    fp = -f / inputs.R_DECAY
    inv = 1.0 / np.where(zero, 1.0, r)
    n = len(r)
    b = np.zeros((n, 4, 4))
    g = np.zeros((3, n, 4, 4))
    eye = np.eye(3)
    dn = (eye[None] - u[:, :, None] * u[:, None, :]) * inv[:, None, None]  # d u_a / d d_c
    b[:, 0, 0] = f[:, 0]
    pps, ppp, dps, dpp = f[:, 2] - f[:, 3], f[:, 3], fp[:, 2] - fp[:, 3], fp[:, 3]
    for c in range(3):
        g[c, :, 0, 0] = fp[:, 0] * u[:, c]
    for p in range(3):
        b[:, 0, 1 + p] = u[:, p] * f[:, 1]
        b[:, 1 + p, 0] = -u[:, p] * f[:, 1]
        for c in range(3):
            x = dn[:, p, c] * f[:, 1] + u[:, p] * fp[:, 1] * u[:, c]
            g[c, :, 0, 1 + p] = x
            g[c, :, 1 + p, 0] = -x
        for q in range(3):
            b[:, 1 + p, 1 + q] = u[:, p] * u[:, q] * pps + eye[p, q] * ppp
            for c in range(3):
                g[c, :, 1 + p, 1 + q] = ((dn[:, p, c] * u[:, q] + u[:, p] * dn[:, q, c]) * pps
                                         + (u[:, p] * u[:, q] * dps + eye[p, q] * dpp) * u[:, c])
    b[zero] = np.diag(onsite)
    g[:, zero] = 0.0
    return b, g


def _gamma(lat, pos, dev):
    """Klopman-Ohno kernel over all periodic images, summed in reciprocal space without its G = 0 term."""
    a = 1.0 / inputs.U_HUBBARD
    gmax = 18.0 / a
    rec = 2.0 * np.pi * np.linalg.inv(lat).T
    m = [int(gmax / np.linalg.norm(rec[i])) + 1 for i in range(3)]
    grid = np.stack(np.meshgrid(*[np.arange(-k, k + 1) for k in m], indexing="ij"), -1).reshape(-1, 3)
    first = np.where(grid[:, 0] != 0, grid[:, 0], np.where(grid[:, 1] != 0, grid[:, 1], grid[:, 2]))
    gv = grid[first > 0] @ rec
    gn = np.sqrt((gv ** 2).sum(1))
    gv, gn = gv[gn <= gmax], gn[gn <= gmax]
    gt = torch.from_numpy(gn).to(dev)
    w = 8.0 * math.pi * a * torch.special.modified_bessel_k1(a * gt) / gt / abs(np.linalg.det(lat))
    x = torch.from_numpy(pos).to(dev) @ torch.from_numpy(gv).to(dev).T
    c, s = torch.cos(x) * w.sqrt(), torch.sin(x) * w.sqrt()
    t = c @ c.T + s @ s.T
    return (0.5 * (t + t.T)).cpu().numpy()


def _system(case, which, seed, dev):
    """System dictionary of the binding (keys as in inputs.diamond_si) of the case's system `which`."""
    rng = np.random.default_rng([seed, which])
    shape = np.array([int(s) for s in case["cells"].split(";")[which].split("x")])
    lat = np.diag(inputs.A_SI * shape.astype(float))
    cell = np.stack(np.meshgrid(*[np.arange(s) for s in shape], indexing="ij"), -1).reshape(-1, 3)
    pos = (cell[:, None, :] + FRAC[None]).reshape(-1, 3) * inputs.A_SI
    pos = pos + np.clip(rng.normal(0.0, 1.0, pos.shape), -2.0, 2.0) * case["sigma"]  # keeps S well conditioned
    nat = len(pos)
    light = np.zeros(nat, bool)
    light[rng.permutation(nat)[:2 * int(round(0.5 * case["light"] * nat))]] = True
    norb = np.where(light, 1, 4)
    lmax = np.ceil(inputs.R_CUT / np.diag(lat)).astype(int) + 1
    shift = np.stack(np.meshgrid(*[np.arange(-k, k + 1) for k in lmax], indexing="ij"), -1).reshape(-1, 3)
    lv = shift @ lat
    found = []
    for i in range(nat):
        dv = pos[None] - pos[i] - lv[:, None]
        s, j = np.nonzero((dv * dv).sum(-1) <= inputs.R_CUT ** 2)
        o = np.lexsort((s, j))
        found.append((np.full(len(o), i), j[o], s[o]))
    bi, bj, bs = (np.concatenate(x) for x in zip(*found))
    d = pos[bj] - pos[bi] - lv[bs]
    vs = inputs.BASE_S * (1.0 + 0.1 * rng.uniform(-1.0, 1.0, 4))
    vh = inputs.BASE_H * (1.0 + 0.1 * rng.uniform(-1.0, 1.0, 4))
    on = np.array([inputs.ONSITE_S] + [inputs.ONSITE_P] * 3)
    sb, sg = _two_centre(d, vs, np.ones(4))
    hb, _ = _two_centre(d, vh, on)
    keep = (np.arange(4)[None, :, None] < norb[bi][:, None, None]) & (np.arange(4)[None, None, :] < norb[bj][:, None, None])
    kpt, wk = inputs.kpoints(case["kgrid"].split(";")[which])
    z = np.where(light, 1.0, 4.0)
    return {"lattice": lat, "pos": pos, "orb_offset": np.concatenate([[0], np.cumsum(norb)]).astype(np.int32), "z_ref": z,
            "blk_ijl": np.column_stack([bi, bj, shift[bs]]).astype(np.int32), "h0": hb[keep], "s": sb[keep],
            "ds": np.stack([sg[c][keep] for c in range(3)]), "gamma": _gamma(lat, pos, dev), "kpt": kpt, "wk": wk,
            "n_electrons": float(z.sum()), "dt": 0.2}


def _field(case, t, seed, dt):
    rng = np.random.default_rng([seed, 1000 + t])
    pol = np.array([1.0, 0.0, 0.0]) if case["field"] == "kick" else rng.normal(0.0, 1.0, 3)
    n = case["steps"]
    if case["field"] == "kick":  # stronger where the charges that follow are the result
        return inputs.kick_field(n, (0.2 if case["form"] == "post" else 0.001) * rng.uniform(0.8, 1.2), pol)
    return inputs.pulse_field(n, dt, 0.01 * rng.uniform(0.8, 1.2), rng.uniform(0.08, 0.22), pol, duration=max(n * dt, 40.0))


def _pattern(sysd):
    """Row, column, block and block element of every stored value of the real-space blocks."""
    off = np.asarray(sysd["orb_offset"], np.int64)
    ijl = np.asarray(sysd["blk_ijl"])
    ni, nj = np.diff(off)[ijl[:, 0]], np.diff(off)[ijl[:, 1]]
    size = ni * nj
    blk = np.repeat(np.arange(len(ijl)), size)
    e = np.arange(size.sum()) - np.repeat(np.cumsum(size) - size, size)
    return off[ijl[blk, 0]] + e // nj[blk], off[ijl[blk, 1]] + e % nj[blk], blk


def _bloch(sysd, k, values, dev):
    """Dense sum over blocks of exp(-i k.L) values, on the device in complex128."""
    row, col, blk = _pattern(sysd)
    n = int(sysd["orb_offset"][-1])
    ph = np.exp(-2j * np.pi * (np.asarray(sysd["blk_ijl"])[:, 2:5] @ np.asarray(sysd["kpt"])[k]))
    out = torch.zeros(n * n, dtype=torch.complex128, device=dev)
    out.index_put_((torch.from_numpy(row * n + col).to(dev),), torch.from_numpy(ph[blk] * values).to(dev), accumulate=True)
    return out.reshape(n, n)


def _start(sysd, k, dev, states):
    """Density (or the occupied states) of the lowest N_el / 2 states of H0_k: the ground state without charge feedback."""
    S, H = _bloch(sysd, k, sysd["s"], dev), _bloch(sysd, k, sysd["h0"], dev)
    if not np.any(sysd["kpt"][k]):
        S, H = S.real.contiguous(), H.real.contiguous()
    nocc = int(round(sysd["n_electrons"] / 2))
    Lc = torch.linalg.cholesky(S)
    F = torch.linalg.solve_triangular(Lc, H, upper=False)
    F = torch.linalg.solve_triangular(Lc, F.mH.contiguous(), upper=False)
    F = 0.5 * (F + F.mH)
    if states or len(S) <= 900:
        C = torch.linalg.solve_triangular(Lc.mH, torch.linalg.eigh(F)[1][:, :nocc].contiguous(), upper=True)
        if not states:
            return 2.0 * (C @ C.mH)
        # any orthonormal basis of the occupied space is a start: one that does not depend on how
        # degenerate eigenvectors came out
        G = torch.from_numpy(np.random.default_rng(len(S)).normal(0.0, 1.0, (len(S), nocc))).to(dev).to(C.dtype)
        B = C @ (C.mH @ G)
        R = torch.linalg.cholesky(B.mH @ (S @ B))
        return torch.linalg.solve_triangular(R, B.mH.contiguous(), upper=False).mH.resolve_conj().contiguous()
    # a large cell: purification of the orthogonalised matrix in single precision, polished in double
    ev = torch.linalg.norm(F, ord=1).item()
    P = (0.5 * (torch.eye(len(F), dtype=F.dtype, device=dev) - F / ev)).to(torch.complex64 if F.is_complex() else torch.float32)
    for _ in range(60):
        Q = P @ P
        t, q = P.diagonal().real.sum().item(), Q.diagonal().real.sum().item()
        if abs(t - q) < 1e-3 and abs(t - nocc) < 1e-2:
            break
        P = Q if abs(q - nocc) < abs(2.0 * t - q - nocc) else 2.0 * P - Q
    P = P.to(F.dtype)
    for _ in range(3):
        Q = P @ P
        P = 3.0 * Q - 2.0 * (Q @ P)
        P = 0.5 * (P + P.mH)
    X = torch.linalg.solve_triangular(Lc.mH, P, upper=True)
    D = torch.linalg.solve_triangular(Lc.mH, X.mH.contiguous(), upper=True)
    return D + D.mH


def _inputs(case, seed):
    dev = torch.device("cuda")
    systems = [_system(case, s, seed, dev) for s in range(len(case["cells"].split(";")))]
    traj = [int(t) for t in case["traj"].split(",")]
    start = [[_start(s, k, dev, case["form"] == "cn") for k in range(len(s["wk"]))] for s in systems]
    for s, per_k in zip(systems, start):
        # reference populations equal to the start's: the start is then the self-consistent ground state
        q = np.zeros(len(s["z_ref"]))
        for k, x in enumerate(per_k):
            S = _bloch(s, k, s["s"], dev).to(torch.complex128)
            x = x.to(torch.complex128)
            diag = (2.0 * (x * (S @ x).conj()) if case["form"] == "cn" else x * S.conj()).real.sum(1).cpu().numpy()
            q += s["wk"][k] * np.add.reduceat(diag, s["orb_offset"][:-1])
        s["z_ref"] = q
    fields = [_field(case, t, seed, systems[0]["dt"]) for t in range(len(traj))]
    return systems, traj, start, fields


def _omegas():
    return np.linspace(0.01, 0.5, 400)


def prepare(case, seed):
    systems, traj, start, fields = _inputs(case, seed)
    form = case["form"]
    opt = {"init": vgtb.INIT_USER, "obs_stride": case["obs_stride"], "autotune": case["autotune"],
           "precision": vgtb.SPLIT_BF16X3 if form == "split" else vgtb.FP64, "delta_form": 1 if case["delta"] else 0,
           "integrator": vgtb.CRANK_NICOLSON if form == "cn" else vgtb.LEAPFROG,
           "scc": vgtb.SCC_FROZEN if case["frozen"] else vgtb.SCC_ON}
    ctx = vgtb.Context(systems, traj_sys=traj, **opt)
    for s, per_k in enumerate(start):
        for k, x in enumerate(per_k):
            (ctx.set_coefficients if form == "cn" else ctx.set_density)(s, k, x.cpu().numpy())
    state = {"ctx": ctx, "form": form, "steps": case["steps"], "fields": fields, "traj": traj,
             "nk": [len(s["wk"]) for s in systems], "nocc": [int(round(s["n_electrons"] / 2)) for s in systems]}
    if form == "post":
        ctx.set_field(0, fields[0])
        ctx.propagate(case["steps"])
        state["e0"] = -float(fields[0][0, 0]) / C_LIGHT
        state["group"] = np.arange(len(systems[0]["z_ref"]), dtype=np.int32) % 3
    return state


def run(state):
    ctx, form = state["ctx"], state["form"]
    if form == "post":
        sigma, eps = ctx.spectrum(0, state["e0"], _omegas())
        return {"sigma": sigma, "eps": eps, "dq": ctx.group_charges(0, state["group"], 3)}
    for t, a in enumerate(state["fields"]):
        ctx.set_field(t, a)
    ctx.propagate(state["steps"])
    out = []
    for t, s in enumerate(state["traj"]):
        J, E, q = ctx.observables(t)
        if form == "cn":
            x = [ctx.get_coefficients(t, k, state["nocc"][s]) for k in range(state["nk"][s])]
        else:
            x = [ctx.get_density(t, k) for k in range(state["nk"][s])]
        if form == "split":
            J, E, q = (v.astype(np.float32) for v in (J, E, q))
            x = [v.astype(np.complex64) for v in x]
        out.append({"J": J, "E": E, "q": q, "x": np.stack(x)})
    return out


def _sizes(case, s):
    """Orbitals, occupied states, real-space values, distinct matrix elements, atoms and k-points of system s (expected over seeds)."""
    shape = [int(c) for c in case["cells"].split(";")[s].split("x")]
    nat = 8 * shape[0] * shape[1] * shape[2]
    nl = 2 * int(round(0.5 * case["light"] * nat))
    n = 4 * (nat - nl) + nl
    per_pair = (n / nat) ** 2
    # pairs within the cutoff per atom, counting images (4/3 pi R^3 times the density, and the atom itself)
    pairs = nat * (4.0 / 3.0 * math.pi * inputs.R_CUT ** 3 * 8.0 / inputs.A_SI ** 3)
    nel = (4 * (nat - nl) + nl) // 2
    return n, nel, pairs * per_pair, min(pairs * per_pair, float(n * n)), nat, 8 if case["kgrid"].split(";")[s] == "mp2" else 1


def work(case):
    """Flops: per step, k-point and trajectory the product of the sparse H with D and the dense product with S^-1
    (8 real flops per complex multiply-add); Crank-Nicolson: S^-1 H once and twelve sweeps over the occupied states.
    Bytes: the blocks, S^-1 and the start read once, the series and the final state written once."""
    word = 8 if case["form"] == "split" else 16
    steps, flops, byts = case["steps"], 0.0, 0.0
    if case["form"] == "post":
        levels, nat = steps + 1, _sizes(case, 0)[4]
        return {"bytes": 8.0 * (3 * levels + levels // case["obs_stride"] * (nat + 3) + 13 * 400), "flops": 400.0 * levels * 30.0}
    for t in case["traj"].split(","):
        n, nocc, real, nnz, nat, nk = _sizes(case, int(t))
        if case["form"] == "cn":
            flops += steps * nk * (8.0 * nnz * n + 12 * 8.0 * nocc * n * n + 8.0 * nnz * nocc)
            state = nocc * n
        else:
            flops += steps * nk * (8.0 * n * n * n + 8.0 * nnz * n)
            state = n * n
        byts += 5 * 8.0 * real + 8.0 * nat * nat + word * nk * (n * n + 2.0 * state) + 8.0 * (steps + 1) * (4 + nat / case["obs_stride"])
    return {"bytes": byts, "flops": flops}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the equations
# ---------------------------------------------------------------------------
def _exact_traj(case, sysd, start, A):
    dev = start[0].device
    dt, wk, nk = sysd["dt"], sysd["wk"], len(sysd["wk"])
    off = np.asarray(sysd["orb_offset"])
    n, nat = int(off[-1]), len(off) - 1
    atom = torch.from_numpy(np.repeat(np.arange(nat), np.diff(off))).to(dev)
    gam = torch.from_numpy(np.asarray(sysd["gamma"])).to(dev)
    z = torch.from_numpy(np.asarray(sysd["z_ref"])).to(dev)
    vol = abs(np.linalg.det(sysd["lattice"]))
    row, col, _ = _pattern(sysd)
    flat = torch.from_numpy(np.unique(row * n + col)).to(dev)
    ri, ci = flat // n, flat % n
    crow = torch.searchsorted(ri, torch.arange(n + 1, device=dev))
    S, V, Si = [], [], []
    for k in range(nk):
        full = [_bloch(sysd, k, v, dev) for v in (sysd["s"], sysd["h0"], 1j * sysd["ds"][0], 1j * sysd["ds"][1], 1j * sysd["ds"][2])]
        V.append(torch.stack([f.reshape(-1)[flat] for f in full]))
        Si.append(torch.linalg.inv(full[0]))
        Si[-1] = 0.5 * (Si[-1] + Si[-1].mH)
        if not np.any(sysd["kpt"][k]):
            Si[-1] = Si[-1].real.contiguous()
        S.append(full[0] if case["form"] == "cn" else None)

    def density(x):
        return 2.0 * (x @ x.mH) if case["form"] == "cn" else x

    def times(a, b):  # a may be real
        return a @ b if a.is_complex() else torch.complex(a @ b.real.contiguous(), a @ b.imag.contiguous())

    def observe(X, a):
        q = torch.zeros(nat, dtype=torch.float64, device=dev)
        T = torch.zeros(4, dtype=torch.float64, device=dev)
        for k in range(nk):
            d = density(X[k]).reshape(-1)[flat]
            sums = (d[None] * V[k].conj()).real
            q.index_add_(0, atom[ri], wk[k] * sums[0])
            tot = sums.sum(1)
            T[:3] += wk[k] * (tot[2:] + a * tot[0])
            T[3] += wk[k] * (tot[1] + (a * tot[2:]).sum() + 0.5 * (a @ a) * tot[0])
        dq = q - z
        eps = gam @ dq
        return q, -T[:3] / vol, T[3] + 0.5 * dq @ eps, eps

    def hamilton(k, a, eps):
        s, h, px, py, pz = V[k]
        e = eps[atom]
        # Crank-Nicolson states leave out the |A|^2 term, an overall phase
        return h + 0.5 * (e[ri] + e[ci] + (0.0 if case["form"] == "cn" else a @ a)) * s + a[0] * px + a[1] * py + a[2] * pz

    At = torch.from_numpy(A / C_LIGHT).to(dev)
    X = [x.to(torch.complex128).clone() for x in start]
    if case["form"] != "cn":
        X = [0.5 * (x + x.mH) for x in X]
    J, E, Q, prev, eps0, eprev = [], [], [], None, None, None
    for m in range(case["steps"] + 1):
        q, j, e, eps = observe(X, At[m])
        J.append(j)
        E.append(e)
        if m % case["obs_stride"] == 0:
            Q.append(q)
        if m == case["steps"]:
            break
        if case["frozen"]:
            eps0 = eps if eps0 is None else eps0
            eps = eps0
        new = []
        for k in range(nk):
            if case["form"] == "cn":
                v = hamilton(k, 0.5 * (At[m] + At[m + 1]), 1.5 * eps - 0.5 * (eps if eprev is None else eprev))
                H = torch.zeros(n * n, dtype=torch.complex128, device=dev)
                H[flat] = v
                H = 0.5j * dt * H.reshape(n, n)
                new.append(torch.linalg.solve(S[k] + H, (S[k] - H) @ X[k]))
                continue
            v = hamilton(k, At[m], eps)
            if n > 1000:
                HD = torch.sparse_csr_tensor(crow, ci, v, (n, n)) @ X[k]
            else:
                H = torch.zeros(n * n, dtype=torch.complex128, device=dev)
                H[flat] = v
                HD = H.reshape(n, n) @ X[k]
            Y = times(Si[k], HD)
            dD = -1j * (Y - Y.mH)
            new.append(X[k] + dt * dD if prev is None else prev[k] + 2.0 * dt * dD)
        prev, eprev, X = X, eps, new
    return {"J": torch.stack(J), "E": torch.stack(E), "q": torch.stack(Q), "x": torch.stack(X)}


def exact(case, seed):
    systems, traj, start, fields = _inputs(case, seed)
    out = [_exact_traj(case, systems[s], start[s], fields[t]) for t, s in enumerate(traj)]
    if case["form"] != "post":
        return [{k: v.cpu().numpy() for k, v in r.items()} for r in out]
    J, q = out[0]["J"].cpu().numpy(), out[0]["q"].cpu().numpy()
    dt, w = systems[0]["dt"], _omegas()
    t = np.arange(case["steps"] + 1) * dt
    weight = np.full(len(t), dt)
    weight[[0, -1]] *= 0.5
    e0 = -float(fields[0][0, 0]) / C_LIGHT
    sigma = np.exp(1j * w[:, None] * t[None]) @ (J * (weight * np.exp(-t / 200.0))[:, None]) / e0
    group = np.arange(q.shape[1]) % 3
    dq = np.stack([-(q - q[0])[:, group == g].sum(1) for g in range(3)], 1)
    return {"sigma": sigma, "eps": 1.0 + 4j * np.pi * sigma / w[:, None], "dq": dq}
