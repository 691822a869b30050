"""The work this framework is measured on: force evaluations, DPD steps and
batches through the public binding (paper_1303_4523_gb300.enuf), over the sizes
of the repository's own workloads (electrolytes of density 3 from 1000 to 3 M
beads, the 81000-bead polyelectrolyte, the 64-system sweep).

exact() restates the same sums in plain torch float64 (window loops, torch.fft,
cell-list pairs, the Philox draw), sharing no code with the package.
"""
import math
import random

import numpy as np
import torch

from paper_1303_4523_gb300 import enuf

DEV = "cuda"
DENSITY = 3.0
# Ewald sets: "bench" (p from the case), and the paper's own Table 1 set
SETS = {
    "bench": dict(alpha=0.975, r_cut=3.0, beta=4.0, kappa=13.87 / (4.0 * math.pi)),
    "paper": dict(alpha=1.566, r_cut=3.0, beta=1.125, kappa=1.0 / (4.0 * math.pi)),
}
DPD = dict(a=25.0, gamma=4.5, sigma=3.0, dt=0.04, lambda_vv=0.65, K_bond=4.0, r0_bond=0.0, seed=1303)
NTYPES = 5          # solvent, monomer, counterion, salt cation, salt anion
CHAIN = 50


def _eval(name, N, prec="fp32", p=4, pset="bench", frac=0.1, valency=1, deriv=0, energy=True, host=False):
    return dict(name=name, kind="eval", N=N, prec=prec, p=p, pset=pset, frac=frac, valency=valency, deriv=deriv,
                energy=energy, host=host)


def _step(name, N, prec="fp32", nsteps=4, chains=10, valency=1, host=False):
    return dict(name=name, kind="step", N=N, prec=prec, nsteps=nsteps, chains=chains, valency=valency, host=host)


def _batch(name, systems, n_min, n_max, layout, prec="fp32"):
    return dict(name=name, kind="batch", systems=systems, n_min=n_min, n_max=n_max, layout=layout, prec=prec)


def listed():
    return [
        # the smallest call: one configuration of the simple electrolyte (L = 10, 300 charged) for its
        # forces, the paper's parameter set, inside another program's loop
        _eval("eval_3k_fp32_p2", 3000, p=2, pset="paper", energy=False),
        # the same box in double, energies read: reference-accuracy single evaluations
        _eval("eval_3k_fp64", 3000, prec="fp64"),
        # a CPU code that hands its host arrays over every step (pinned buffers)
        _eval("eval_24k_fp32_host", 24000, host=True),
        # the size sweep's middle, energies read at every evaluation
        _eval("eval_81k_fp32", 81000),
        # gradient-mode forces (one inverse transform), 2:1 salt
        _eval("eval_192k_fp32_grad", 192000, valency=2, deriv=1, energy=False),
        # a served request of odd size: its grid (n = 180) has no power-of-two length
        _eval("eval_524287_fp32", 524287),
        # the largest served system
        _eval("eval_3m_fp32", 3000000),
        # the sweep's largest size in double
        _eval("eval_375k_fp64", 375000, prec="fp64"),
        # the headline run: polyelectrolyte DPD, blocks of 4 steps, energies sampled once a block
        # (short blocks: rounding differences grow along a trajectory)
        _step("step_poly81k_fp32", 81000),
        # the same run in double
        _step("step_poly81k_fp64", 81000, prec="fp64"),
        # the same run with the state on the host, in and out at every step
        _step("step_poly81k_fp32_host", 81000, nsteps=1, host=True),
        # parameter sweeps: 64 uneven systems evaluated at once
        _batch("batch_64_fp32", 64, 3000, 81000, layout=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["eval", "host", "step", "batch"], [10, 2, 6, 2])[0]
    if kind == "eval" or kind == "host":
        prec = rng.choices(["fp32", "fp64"], [4, 1])[0]
        hi = 375000 if prec == "fp64" or kind == "host" else 3000000
        N = _log_int(rng, 1000, hi)
        pset, p = rng.choices([("bench", 4), ("bench", 3), ("bench", 6), ("paper", 2)], [7, 1, 1, 1])[0]
        if p == 6:
            N = min(N, 150000)
        c = _eval("", N, prec=prec, p=p, pset=pset, frac=rng.choice([0.1, 0.1, 0.25]) if N < 100000 else 0.1,
                  valency=rng.choice([1, 1, 2]), deriv=rng.choice([0, 0, 0, 1]), energy=rng.random() < 0.6,
                  host=kind == "host")
    elif kind == "step":
        prec = rng.choices(["fp32", "fp64"], [4, 1])[0]
        N = _log_int(rng, 1000, 300000 if prec == "fp32" else 81000)
        host = rng.random() < 0.25
        c = _step("", N, prec=prec, nsteps=1 if host else rng.randint(1, 4), chains=max(1, int(0.006 * N / CHAIN)),
                  valency=rng.choice([1, 2]), host=host)
    else:
        c = _batch("", rng.randint(4, 64), 3000, _log_int(rng, 10000, 81000), layout=rng.randrange(1 << 20))
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _box(N):
    return (N / DENSITY) ** (1.0 / 3.0)


def _grid(L):
    """Base grid: 1.6 L rounded to the nearest even 2^a 3^b 5^c integer, at least 8."""
    def smooth(m):
        for f in (2, 3, 5):
            while m % f == 0:
                m //= f
        return m == 1
    target, best = 1.6 * L, None
    for m in range(2, int(4 * target) + 8, 2):
        if smooth(m) and (best is None or abs(m - target) < abs(best - target) - 1e-12):
            best = m
    return max(best, 8)


def _dtype(prec):
    return torch.float32 if prec == "fp32" else torch.float64


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _electrolyte(N, frac, valency, dtype, gen):
    """Uniform beads; cations +valency and anions -1 (neutral) on a random subset."""
    pos = torch.rand((N, 3), generator=gen, device=DEV, dtype=torch.float64).mul_(_box(N)).to(dtype)
    order = torch.randperm(N, generator=gen, device=DEV)
    n_cat = int(round(frac * N)) // (1 + valency)
    q = torch.zeros(N, device=DEV, dtype=dtype)
    q[order[:n_cat]] = float(valency)
    q[order[n_cat:n_cat + valency * n_cat]] = -1.0
    return pos, q


def _polyelectrolyte(case, seed):
    """Chains of 50 beads (random walk of step 0.5, every second monomer -1), their counterions,
    z:1 salt at 0.1 bead fraction, the rest neutral solvent; Maxwell velocities. Host arrays."""
    rng = np.random.default_rng(seed)
    N, L, z, nc = case["N"], _box(case["N"]), case["valency"], case["chains"]
    pos = rng.uniform(0.0, L, (N, 3))
    d = rng.normal(size=(nc, CHAIN, 3))
    d *= 0.5 / np.linalg.norm(d, axis=2, keepdims=True)
    d[:, 0] = rng.uniform(0.0, L, (nc, 3))
    m = nc * CHAIN
    pos[:m] = np.cumsum(d, axis=1).reshape(m, 3) % L
    q, types = np.zeros(N), np.zeros(N, np.int32)
    types[:m] = 1
    q[0:m:2] = -1.0
    k = m + m // 2
    q[m:k], types[m:k] = 1.0, 2
    n_cat = int(round(0.1 * N)) // (1 + z)
    q[k:k + n_cat], types[k:k + n_cat] = float(z), 3
    q[k + n_cat:k + n_cat * (1 + z)], types[k + n_cat:k + n_cat * (1 + z)] = -1.0, 4
    vel = rng.normal(size=(N, 3))
    vel -= vel.mean(axis=0)
    i = np.arange(m).reshape(nc, CHAIN)
    bonds = np.stack([i[:, :-1], i[:, 1:]], axis=-1).reshape(-1, 2).astype(np.int32)
    real = np.float32 if case["prec"] == "fp32" else np.float64
    return pos.astype(real), vel.astype(real), q.astype(real), types, bonds


def _layout(case):
    """Bead counts, charged fractions and valencies of a batch's systems."""
    r = random.Random(case["layout"])
    return [(_log_int(r, case["n_min"], case["n_max"]), r.choice([0.1, 0.1, 0.12]), r.choice([1, 2]))
            for _ in range(case["systems"])]


def _batch_inputs(case, seed):
    gen = _gen(seed)
    return [_electrolyte(N, frac, z, _dtype(case["prec"]), gen) for N, frac, z in _layout(case)]


class _Resident:
    """A device array that the system owns (which this object keeps alive), for torch.as_tensor."""

    def __init__(self, system, ptr, n, prec):
        self.system = system
        self.__cuda_array_interface__ = dict(shape=(n, 3), typestr="<f4" if prec == "fp32" else "<f8",
                                             data=(ptr, False), version=2)


def _params(case):
    L = _box(case["N"])
    return enuf.make_params(L=L, M=_grid(L), p=case.get("p", 4), prec=case["prec"], deriv=case.get("deriv", 0),
                            **SETS[case.get("pset", "bench")])


def prepare(case, seed):
    dt = _dtype(case["prec"])
    if case["kind"] == "eval":
        pos, q = _electrolyte(case["N"], case["frac"], case["valency"], dt, _gen(seed))
        s = dict(case=case, plan=enuf.Plan(_params(case), case["N"]))
        if case["host"]:
            pos, q, F = (torch.empty(x.shape, dtype=dt, pin_memory=True).copy_(x).numpy() for x in (pos, q, pos))
        else:
            F = torch.empty_like(pos)
        s.update(pos=pos, q=q, F=F)
    elif case["kind"] == "step":
        pos, vel, q, types, bonds = _polyelectrolyte(case, seed)
        plan = enuf.Plan(_params(case), case["N"])
        sim = enuf.DpdSystem(plan, np.full((NTYPES, NTYPES), DPD["a"]), DPD["gamma"], DPD["sigma"], DPD["dt"], pos, vel,
                             types, q, bonds, lambda_vv=DPD["lambda_vv"], K_bond=DPD["K_bond"],
                             r0_bond=DPD["r0_bond"], seed=DPD["seed"])
        s = dict(case=case, sim=sim)
        if case["host"]:
            s["state"] = [torch.empty((case["N"], 3), dtype=dt, pin_memory=True) for _ in range(3)]
            sim.get_state_into(*s["state"])
        else:
            s["state"] = [torch.as_tensor(_Resident(sim, p, case["N"], case["prec"]), device=DEV)
                          for p in sim.device_state()]
    else:
        inputs = _batch_inputs(case, seed)
        shapes = _layout(case)
        params = [_params(dict(N=N, prec=case["prec"])) for N, _, _ in shapes]
        F = torch.empty((sum(N for N, _, _ in shapes), 3), device=DEV, dtype=dt)
        s = dict(case=case, batch=enuf.Batch(params, [N for N, _, _ in shapes]), pos=[p for p, _ in inputs],
                 q=[q for _, q in inputs], F=F, parts=list(F.split([N for N, _, _ in shapes])))
    return s


def run(s):
    """The forces (or the new state) whole, and the energies in the type the case computes in."""
    case = s["case"]
    real = np.float32 if case["prec"] == "fp32" else np.float64
    if case["kind"] == "eval":
        if case["host"]:
            E, W = s["plan"].energy_forces_host(s["pos"], s["q"], s["F"])
        elif case["energy"]:
            E, W = s["plan"].energy_forces(s["pos"], s["q"], s["F"])
        else:
            s["plan"].energy_forces(s["pos"], s["q"], s["F"], want_energy=False)
            return dict(F=s["F"])
        return dict(F=s["F"], E=E.astype(real), virial=real(W))
    if case["kind"] == "step":
        if case["host"]:
            E = s["sim"].step_host(*s["state"], nsteps=case["nsteps"], want_energy=True)
        else:
            E = s["sim"].step(case["nsteps"], want_energy=True)
        pos, vel, F = s["state"]
        return dict(pos=pos, vel=vel, F=F, E=E.astype(real))
    E = s["batch"].energy_forces(s["pos"], s["q"], s["parts"])
    return dict(F=s["F"], E=E.astype(real))


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _eval_work(N, nq, esz, p, deriv, rc):
    n = 2 * _grid(_box(N))
    nf = 1 if deriv else 3
    pairs = 0.5 * nq * (nq / N) * DENSITY * 4.0 / 3.0 * math.pi * rc ** 3
    fft = (1 + nf) * 2.5 * n ** 3 * math.log2(n ** 3)      # one real transform forward, nf inverse
    taps = (2 * p) ** 3
    return esz * 7 * N, pairs * 60 + fft + nq * taps * 2 * (1 + max(nf, 2))


def work(case):
    esz = 4 if case["prec"] == "fp32" else 8
    if case["kind"] == "batch":
        b = f = 0.0
        for N, frac, _ in _layout(case):
            x, y = _eval_work(N, frac * N, esz, 4, 0, 3.0)
            b, f = b + x, f + y
        return dict(bytes=b, flops=f)
    N = case["N"]
    if case["kind"] == "eval":
        b, f = _eval_work(N, case["frac"] * N, esz, case["p"], case["deriv"], SETS[case["pset"]]["r_cut"])
        return dict(bytes=b, flops=f)
    _, f = _eval_work(N, 0.1 * N + 0.75 * case["chains"] * CHAIN, esz, 4, 0, 3.0)
    f += 0.5 * N * DENSITY * 4.0 / 3.0 * math.pi * 100      # DPD pairs: forces and the random draw
    # the state (positions, velocities, forces) in and out, charges and types in
    return dict(bytes=case["nsteps"] * (18 * esz + esz + 4) * N, flops=case["nsteps"] * f)


# ---------------------------------------------------------------------------
# the same sums in 64 bits
# ---------------------------------------------------------------------------
def _pairs(x, L, rc):
    """All pairs i < j (in some order) closer than rc: indices, minimum-image r_i - r_j, r^2."""
    n = x.shape[0]
    out = []

    def keep(i, j):
        d = x[i] - x[j]
        d = d - L * torch.round(d / L)
        r2 = (d * d).sum(1)
        ok = (r2 < rc * rc) & (r2 > 0)
        out.append((i[ok], j[ok], d[ok], r2[ok]))

    nc = int(L / rc)
    if nc < 3:
        keep(*torch.triu_indices(n, n, 1, device=x.device))
    else:
        c = (x * (nc / L)).long().clamp_(0, nc - 1)
        cell = (c[:, 2] * nc + c[:, 1]) * nc + c[:, 0]
        order = torch.argsort(cell, stable=True)
        count = torch.bincount(cell, minlength=nc ** 3)
        start = torch.cumsum(count, 0) - count
        m = int(count.max())
        slot = torch.arange(n, device=x.device) - start[cell[order]]
        table = torch.full((nc ** 3, m), -1, dtype=torch.long, device=x.device)
        table[cell[order], slot] = order
        cube = torch.arange(nc ** 3, device=x.device).view(nc, nc, nc)
        part = max(1, 20_000_000 // (m * m))
        for k in range(13, 27):      # the cell itself and the 13 after it
            dx, dy, dz = k % 3 - 1, k // 3 % 3 - 1, k // 9 - 1
            other = torch.roll(cube, (-dz, -dy, -dx), (0, 1, 2)).reshape(-1)
            for a in range(0, nc ** 3, part):
                i = table[a:a + part, :, None].expand(-1, m, m)
                j = table[other[a:a + part], None, :].expand(-1, m, m)
                ok = (i >= 0) & (j >= 0)
                if k == 13:
                    ok &= i < j
                keep(i[ok], j[ok])
    return tuple(torch.cat(v) for v in zip(*out))


def _wrap(x, L):
    w = x - L * torch.floor(x / L)
    return torch.where(w >= L, torch.zeros_like(w), w)


def _electrostatics(x, q, P, L, p, deriv):
    """F, (E_real, E_recip, E_self + E_neutral, total), virial of all beads (x wrapped), float64."""
    al, be, kap, rc = P["alpha"], P["beta"], P["kappa"], P["r_cut"]
    F = torch.zeros_like(x)
    ch = torch.nonzero(q).reshape(-1)
    xc, qc = x[ch], q[ch]
    Fc = torch.zeros_like(xc)
    # real space: erfc and the Slater correction
    i, j, d, r2 = _pairs(xc, L, rc)
    r = r2.sqrt()
    e = torch.exp(-2.0 * be * r)
    qq = kap * qc[i] * qc[j]
    B = torch.special.erfc(al * r)
    u = (B - (1.0 + be * r) * e) / r
    f = (B - (1.0 + 2.0 * be * r + 2.0 * (be * r) ** 2) * e) / r2 + 2.0 * al / math.sqrt(math.pi) * torch.exp(-(al * r) ** 2) / r
    E_real, W_real = (qq * u).sum(), (qq * f * r).sum()
    g = (qq * f / r)[:, None] * d
    Fc.index_add_(0, i, g).index_add_(0, j, -g)
    # reciprocal space: the Gaussian-window NFFT sums
    M = _grid(L)
    n, nc = 2 * M, M // 2 - 1
    b = 4.0 * p / (3.0 * math.pi)
    uu = xc * (n / L)
    uu = torch.where(uu >= n, uu - n, uu)
    base = torch.floor(uu)
    l = base.long()[:, :, None] + torch.arange(1 - p, p + 1, device=x.device)      # [nq, 3, 2p]
    dist = uu[:, :, None] - l
    w = torch.exp(-dist * dist / b) / math.sqrt(math.pi * b)
    l = l % n
    dw = -2.0 * dist / b * w
    grid = torch.zeros(n ** 3, dtype=torch.float64, device=x.device)
    part = max(1, 30_000_000 // (2 * p) ** 3)
    for a in range(0, len(qc), part):
        s = slice(a, a + part)
        idx = (l[s, 2, :, None, None] * n + l[s, 1, None, :, None]) * n + l[s, 0, None, None, :]
        v = w[s, 2, :, None, None] * w[s, 1, None, :, None] * w[s, 0, None, None, :] * qc[s, None, None, None]
        grid.index_add_(0, idx.reshape(-1), v.reshape(-1))
    S = torch.fft.fftn(grid.view(n, n, n))
    k = torch.fft.fftfreq(n, 1.0 / n, device=x.device, dtype=torch.float64)
    in1 = (k.abs() <= nc).double()
    c2 = in1 * torch.exp(2.0 * b * (math.pi * k / n) ** 2)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2
    D = c2[:, None, None] * c2[None, :, None] * c2[None, None, :] * torch.exp(-math.pi ** 2 * k2 / (al * L) ** 2)
    D = torch.where(k2 > 0, D / k2.clamp(min=1.0), torch.zeros_like(D))
    Ek = kap / (2.0 * math.pi * L) * D * (S.real ** 2 + S.imag ** 2)
    E_recip = Ek.sum()
    W_recip = (Ek * (1.0 - 2.0 * math.pi ** 2 * k2 / (al * L) ** 2)).sum()
    G = D * S
    del Ek, k2, S, D

    def gather(h, wx, wy, wz):
        got = torch.empty_like(qc)
        for a in range(0, len(qc), part):
            s = slice(a, a + part)
            idx = (l[s, 2, :, None, None] * n + l[s, 1, None, :, None]) * n + l[s, 0, None, None, :]
            v = wz[s, :, None, None] * wy[s, None, :, None] * wx[s, None, None, :]
            got[s] = (h.reshape(-1)[idx] * v).sum((1, 2, 3))
        return got

    if deriv:
        h = torch.fft.ifftn(G, norm="forward").real
        for t in range(3):
            ws = [dw[:, t2] if t2 == t else w[:, t2] for t2 in range(3)]
            Fc[:, t] += -kap * n / (math.pi * L * L) * qc * gather(h, *ws)
    else:
        for t in range(3):
            kt = k.view(*(n if 2 - t == dim else 1 for dim in range(3)))
            h = torch.fft.ifftn(-1j * kt * G, norm="forward").real
            Fc[:, t] += 2.0 * kap / (L * L) * qc * gather(h, w[:, 0], w[:, 1], w[:, 2])
    Q = qc.sum()
    E_neut = -kap * math.pi / (2.0 * L ** 3 * al * al) * Q * Q
    E_self = -kap * al / math.sqrt(math.pi) * (qc * qc).sum() + E_neut
    F[ch] = Fc
    return F, torch.stack([E_real, E_recip, E_self, E_real + E_recip + E_self]), W_real + W_recip + 3.0 * E_neut


def _philox0(c0, c1, step, seed):
    """Word 0 of Philox4x32-10 of the counters (c0, c1, step_lo, step_hi) under key = seed."""
    m32 = 0xFFFFFFFF
    x = [c0, c1, torch.full_like(c0, step & m32), torch.full_like(c0, step >> 32)]
    k0, k1 = seed & m32, seed >> 32
    for _ in range(10):
        a, b = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57        # modulo 2^64
        x = [((b >> 32) & m32) ^ x[1] ^ k0, b & m32, ((a >> 32) & m32) ^ x[3] ^ k1, a & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return x[0]


def _dpd_forces(x, v0, bonds, L, step):
    F = torch.zeros_like(x)
    i, j, d, r2 = _pairs(_wrap(x, L), L, 1.0)
    r = r2.sqrt()
    w = 1.0 - r
    word = _philox0(torch.minimum(i, j), torch.maximum(i, j), step, DPD["seed"])
    theta = math.sqrt(3.0) * (2.0 * (word.double() + 0.5) / 2.0 ** 32 - 1.0)
    vr = ((v0[i] - v0[j]) * d).sum(1) / r
    f = w * (DPD["a"] - DPD["gamma"] * w * vr + DPD["sigma"] * theta / math.sqrt(DPD["dt"])) / r
    g = f[:, None] * d
    F.index_add_(0, i, g).index_add_(0, j, -g)
    i, j = bonds[:, 0], bonds[:, 1]
    d = x[i] - x[j]
    d = d - L * torch.round(d / L)
    rb = (d * d).sum(1).sqrt()
    g = (-DPD["K_bond"] * (rb - DPD["r0_bond"]) / rb.clamp(min=1e-300))[:, None] * d
    F.index_add_(0, i, g).index_add_(0, j, -g)
    return F, 0.5 * DPD["a"] * (w * w).sum(), 0.5 * DPD["K_bond"] * ((rb - DPD["r0_bond"]) ** 2).sum()


def _exact_steps(case, seed):
    pos, vel, q, types, bonds = _polyelectrolyte(case, seed)
    x, v, q = (torch.as_tensor(a, device=DEV).double() for a in (pos, vel, q))
    bonds = torch.as_tensor(bonds, device=DEV).long()
    L, P, dt = _box(case["N"]), SETS["bench"], DPD["dt"]

    def force(v0, step):
        F, Ec, Eb = _dpd_forces(x, v0, bonds, L, step)
        Fe, E, W = _electrostatics(_wrap(x, L), q, P, L, 4, 0)
        return F + Fe, E, Ec, Eb, W

    F, E, Ec, Eb, W = force(v, 0)
    for step in range(1, case["nsteps"] + 1):
        v0 = v + DPD["lambda_vv"] * dt * F
        v = v + 0.5 * dt * F
        x = x + v * dt
        F, E, Ec, Eb, W = force(v0, step)
        v = v + 0.5 * dt * F
    return dict(pos=x, vel=v, F=F, E=torch.cat([E, torch.stack([Ec, Eb, 0.5 * (v * v).sum(), W])]))


def exact(case, seed):
    if case["kind"] == "step":
        return _exact_steps(case, seed)
    if case["kind"] == "eval":
        x, q = _electrolyte(case["N"], case["frac"], case["valency"], _dtype(case["prec"]), _gen(seed))
        L = _box(case["N"])
        F, E, W = _electrostatics(_wrap(x.double(), L), q.double(), SETS[case["pset"]], L, case["p"], case["deriv"])
        return dict(F=F, E=E, virial=np.float64(float(W))) if case["energy"] or case["host"] else dict(F=F)
    Fs, Es = [], []
    for x, q in _batch_inputs(case, seed):
        L = _box(x.shape[0])
        F, E, _ = _electrostatics(_wrap(x.double(), L), q.double(), SETS["bench"], L, 4, 0)
        Fs.append(F)
        Es.append(E)
    return dict(F=torch.cat(Fs), E=torch.stack(Es))
