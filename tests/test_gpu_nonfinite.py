"""Positions that are not numbers (a diverged integration): they stay with their
bead, index nothing outside the arrays, and leave no trace in the next call."""
import numpy as np
import pytest

import oracle as orc
from paper_1303_4523_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_dpd import _bead_max, _make, _prep, _rel, _system, enuf  # noqa: E402,F401


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("pairs", [1, 2])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("fp32", 1e-5)])
def test_dpd_forces_beside_a_lost_bead(enuf, prec, tol, pairs, bad):
    """An uncharged, unbonded bead without a position: the others' forces are the
    oracle's, which finds no pair of that bead within the cutoffs; and a step runs."""
    s = _system()
    dp = W.dpd_params(5)
    pos, vel, q = _prep(prec, s)
    lost = int(np.flatnonzero((q == 0) & ~np.isin(np.arange(s.N), s.bonds))[7])
    pos[lost] = [bad, 1.0, bad]
    plan, sysm, Po, Do = _make(enuf, prec, s, pos, vel, q, dp, pairs)
    _, _, F, _ = sysm.get_state()
    Fr, _ = orc.total_forces(Po, Do, pos, vel, s.types, q, s.bonds, step=0)
    keep = np.arange(s.N) != lost
    F = np.asarray(F, np.float64)
    assert np.all(np.isfinite(F[keep])) and np.all(F[lost] == 0.0)
    assert _rel(F[keep], Fr[keep]) < tol and _bead_max(F[keep], Fr[keep]) < 100 * tol
    sysm.step(1)
    p, _, F, _ = sysm.get_state()
    assert not np.isfinite(p[lost]).all() and np.all(np.isfinite(F[keep]))
    sysm.close()
    plan.close()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("fp32", 1e-5)])
def test_charged_bead_without_a_position(enuf, prec, tol):
    """A charged bead at NaN makes the reciprocal part of the call NaN (its window has
    no weights) and nothing else: no error, and the next call on the same plan, with
    numbers, is the oracle's."""
    s = W.electrolyte_small("bench")
    P = dict(L=s.L, M=s.M, **s.params)
    dt = torch.float32 if prec == "fp32" else torch.float64
    pos, _, q = _prep(prec, s)
    charged = np.flatnonzero(q != 0)
    plan = enuf.Plan(enuf.make_params(prec=prec, **P), s.N)
    tq = torch.tensor(q, dtype=dt, device="cuda")
    for bad in (np.nan, np.inf, -np.inf):
        x = pos.copy()
        x[charged[3]] = [bad, bad, 1.0]
        F = torch.empty((s.N, 3), dtype=dt, device="cuda")
        E, _ = plan.energy_forces(torch.tensor(x, dtype=dt, device="cuda"), tq, F)
        assert np.isnan(E[1]) and np.isfinite(E[0]) and bool((F[tq == 0] == 0).all())
    E, _ = plan.energy_forces(torch.tensor(pos, dtype=dt, device="cuda"), tq, F)
    Fr, Er = orc.real_space(orc.EwaldParams(**P), pos, q)
    Fk, Ek, _, _ = orc.recip_enuf(orc.EwaldParams(**P), pos, q)
    assert _rel(F.double().cpu().numpy(), Fr + Fk) < tol
    assert abs(E[1] - Ek[0]) <= tol * abs(Ek[0])
    plan.close()
