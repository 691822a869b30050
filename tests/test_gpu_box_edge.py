"""Beads within rounding of a box face: the tile a bead is sorted into and the
coordinate it is stored with agree, whatever the box edge rounds to (round
edges such as 10, 30 or 50 hide the FP32 case), against the FP64 CPU oracle."""
import numpy as np
import pytest

import oracle as orc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_enuf import TOL, Ref, _bead_max, _gpu, _inputs, _oparams, _rel_rms, enuf  # noqa: E402,F401

# edges L with L^3 = N/3 and others, grids n = 2 M: float(L) above and below L, and
# (FP64) boxes where the largest double below L times n/L rounds to n
BOXES = {"14.45": (14.449686898305517, 24), "15": (15.0, 24), "25.54": (25.543647746451768, 40),
         "28.58": (28.57539627437798, 45 * 2), "30": (30.0, 48), "50-": (49.999999999999986, 80),
         "55.9": (55.90911419702041, 90)}


def _face_beads(prec, L, seed=5):
    """Charged beads at, just below and just above a face of each dimension (as
    given, from either side, and some boxes away), each with three charged
    partners on either side of the face within r_c, and uncharged beads."""
    fl = np.float32 if prec == "fp32" else np.float64
    near = [-1e-7, -1e-8, 0.0, float(np.nextafter(L, 0.0)), float(fl(L)), float(np.nextafter(fl(L), fl(0.0)))]
    for k in (1, 3, -2):
        x = fl(k * L)
        near += [float(np.nextafter(x, fl(-np.inf))), float(x), float(np.nextafter(x, fl(np.inf)))]
    if prec == "fp64":
        near += [-1e-15, -1e-17]
    rng = np.random.default_rng(seed)
    pos, q = [], []
    for axis in range(3):
        for x in near:
            c = rng.uniform(0.0, L, 3)
            c[axis] = x
            pos.append(c)
            q.append(rng.choice([-1.0, 1.0]))
            for side in (-1.0, 1.0):
                for _ in range(3):
                    d = rng.uniform(-1.2, 1.2, 3)
                    d[axis] = side * rng.uniform(0.3, 2.0)
                    pos.append(c + d)
                    q.append(rng.choice([-1.0, 1.0, 2.0]))
    pos = np.concatenate([np.array(pos), rng.uniform(0.0, L, (50, 3))])
    return pos, np.concatenate([q, np.zeros(50)])


def _at_face(L, n, pos):
    """FP64 inputs wrapped as documented (x - L floor(x / L), corrected once into
    [0, L), else 0), those whose grid coordinate x (n/L) rounds to n at 0: the oracle,
    which forms n (x/L), then takes the same grid base (the move is at most half a
    unit in the last place of L)."""
    k = np.floor(pos.astype(np.float32) / np.float32(L)).astype(np.float64)   # as the kernels take the quotient
    w = pos - L * k
    w = np.where(w < 0, pos - L * (k - 1), np.where(w >= L, pos - L * (k + 1), w))
    w = np.where((w >= L) | (w < 0), 0.0, w)
    w = np.where((pos >= 0) & (pos < L), pos, w)
    return np.where(w * (n / L) >= n, 0.0, w)


@pytest.mark.parametrize("prec,box", [("fp64", "14.45"), ("fp64", "15"), ("fp64", "25.54"), ("fp64", "28.58"),
                                      ("fp64", "30"), *(("fp32", b) for b in BOXES)])
def test_beads_at_the_faces(enuf, prec, box):
    """Forces bead by bead and E_real. p = 8 (FP64) or 6: a grid base that the two
    sides decide differently for a bead on a face exchanges end taps of relative
    size 7e-9 (6e-7 at p = 6), below the FP32 bounds."""
    L, M = BOXES[box]
    P = dict(L=L, M=M, p=8 if prec == "fp64" else 6, alpha=1.0, r_cut=3.0, beta=4.0, kappa=1.1)
    pos, q = _inputs(prec, *_face_beads(prec, L))
    plan, F, E, Wv = _gpu(enuf, prec, P, pos, q)
    assert plan.info.n // plan.info.tile > 3      # more tiles than the stencil has: shifted images
    ref, t = Ref(P, _at_face(L, 2 * M, pos) if prec == "fp64" else pos, q), TOL[prec]
    assert np.all(np.isfinite(F))
    assert _rel_rms(F, ref.F) < t["F"] and _bead_max(F, ref.F) < 100 * t["F"]
    own = max(abs(ref.E[0]), abs(ref.E[2])) if prec == "fp32" else abs(ref.E[0])
    assert abs(E[0] - ref.E[0]) <= t["E"] * own, (E, ref.E)
    plan.close()


def test_beads_at_the_faces_in_a_batch(enuf):
    """The same through one launch sequence, systems of two window widths."""
    P, pos, q, ref = [], [], [], []
    for box, p in (("14.45", 6), ("25.54", 6), ("30", 8)):
        L, M = BOXES[box]
        P.append(dict(L=L, M=M, p=p, alpha=1.0, r_cut=3.0, beta=4.0, kappa=1.1))
        x, c = _inputs("fp32", *_face_beads("fp32", L, seed=9))
        ref.append(Ref(P[-1], x, c))
        pos.append(torch.tensor(x, dtype=torch.float32, device="cuda"))
        q.append(torch.tensor(c, dtype=torch.float32, device="cuda"))
    F = [torch.full_like(x, float("nan")) for x in pos]
    b = enuf.Batch([enuf.make_params(prec="fp32", **p) for p in P], [len(x) for x in pos])
    assert b.mode() == 1
    E = b.energy_forces(pos, q, F)
    for k, r in enumerate(ref):
        Fk = F[k].double().cpu().numpy()
        assert _rel_rms(Fk, r.F) < TOL["fp32"]["F"] and _bead_max(Fk, r.F) < 100 * TOL["fp32"]["F"]
        assert abs(E[k][0] - r.E[0]) <= TOL["fp32"]["E"] * max(abs(r.E[0]), abs(r.E[2]))
    b.close()


@pytest.mark.parametrize("pairs", [1, 2])
@pytest.mark.parametrize("box", ["14.45", "25.54"])
def test_beads_crossing_a_face_in_a_step(enuf, box, pairs):
    """FP32 DPD step whose beads move from 0 to -1e-7 and 1e-7: the step's forces
    (Table 2, at the new positions) against the oracle's step. One step rounds
    positions and velocities once more than a force evaluation: twice its bound."""
    L, M = BOXES[box]
    P = dict(L=L, M=M, p=6, alpha=1.0, r_cut=3.0, beta=4.0, kappa=1.1)
    pos, q = _inputs("fp32", *_face_beads("fp32", L, seed=11))
    dt = 0.04
    vel = np.zeros_like(pos)
    for axis in range(3):
        at0 = np.flatnonzero(pos[:, axis] == 0.0)
        vel[at0, axis] = -1e-7 / dt
    vel = np.asarray(vel, np.float32).astype(np.float64)
    n = len(q)
    types = np.zeros(n, np.int32)
    dp = dict(a=np.full((1, 1), 25.0), gamma=4.5, sigma=3.0, dt=dt, lambda_vv=0.65, K_bond=4.0, r0_bond=0.0, seed=3)
    bonds = np.zeros((0, 2), np.int32)
    plan = enuf.Plan(enuf.make_params(prec="fp32", pairs=pairs, **P), n)
    s = enuf.DpdSystem(plan, dp["a"], dp["gamma"], dp["sigma"], dt, pos, vel, types, q, bonds,
                       lambda_vv=dp["lambda_vv"], K_bond=dp["K_bond"], r0_bond=dp["r0_bond"], seed=dp["seed"])
    Po, Do = _oparams(P), orc.DpdParams(**dp)
    F0, _ = orc.total_forces(Po, Do, pos, vel, types, q, bonds, step=0)
    _, _, F, _ = s.get_state()
    assert _rel_rms(F.astype(np.float64), F0) < 1e-5 and _bead_max(F.astype(np.float64), F0) < 1e-3
    s.set_state(pos, vel, F=np.zeros((n, 3)), step=0)
    s.step(1)
    p1, _, F1, _ = s.get_state()
    assert ((p1 < 0.0) & (p1 > -2e-7)).any()
    _, _, Fr, _, _ = orc.dpd_run(Po, Do, pos, vel, np.zeros((n, 3)), types, q, bonds, step=0, nsteps=1)
    assert _rel_rms(F1.astype(np.float64), Fr) < 2e-5 and _bead_max(F1.astype(np.float64), Fr) < 2e-3
    s.close()
    plan.close()
