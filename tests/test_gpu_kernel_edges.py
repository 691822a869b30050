"""The evaluation's kernels at the sizes where their work split can go wrong
(lists that fill, rows across the box face, few beads, few tiles), against the
FP64 CPU oracle with the parity tests' bounds."""
import numpy as np
import pytest

import oracle as orc  # noqa: F401  (the oracle is built with the library)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_enuf import TOL, Ref, _bead_max, _check, _gpu, _inputs, _oparams, _rel_rms, enuf  # noqa: E402,F401


def _beads(L, nq, cluster, seed, solvent=37):
    """nq charged beads, the first `cluster` of them in a unit ball around a box
    corner (each within r_c of all others, across three faces), the rest
    uniform, some on the faces; uncharged beads mixed in."""
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0.0, L, (nq, 3))
    pos[:cluster] = rng.uniform(-0.6, 0.6, (cluster, 3)) % L
    if nq > cluster + 4:
        pos[cluster] = [0.0, 0.5 * L, np.nextafter(L, 0.0)]
        pos[cluster + 1] = [-0.25 * L, 1.5 * L, 2.0 * L]      # wrapped inside the library
    q = np.where(np.arange(nq) % 2 == 0, 1.0, -1.0)
    pos = np.concatenate([pos, rng.uniform(0.0, L, (solvent, 3))])
    q = np.concatenate([q, np.zeros(solvent)])
    order = rng.permutation(len(q))
    return pos[order], q[order]


BASE = dict(alpha=1.0, r_cut=3.0, beta=4.0, kappa=1.1, p=4)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name,box", [
    ("stencil_3_of_4", dict(L=12.0, M=20, tile=10)),      # rs = 1, 4 tiles: rows wrapped tile by tile
    ("stencil_5_of_4", dict(L=9.0, M=16, tile=8)),        # rs = 2, 4 tiles: whole rows, minimum image
    ("stencil_5_of_8", dict(L=20.0, M=32, tile=8)),       # rs = 2 with room
    ("stencil_3_of_3", dict(L=9.0, M=18, tile=12)),       # exactly the tiles there are
])
@pytest.mark.parametrize("nq,cluster", [(2, 2), (33, 33), (200, 150), (1500, 90)])
def test_real_space_lists(enuf, prec, name, box, nq, cluster):
    """Lists that fill several times (150 beads within r_c of one another),
    lanes per bead from 32 down, beads on and outside the faces: forces and the
    real-space energy (beads on grid lines may take the other grid base in FP32,
    which moves E_recip by the window's truncation)."""
    P = dict(BASE, **box)
    pos, q = _inputs(prec, *_beads(P["L"], nq, cluster, seed=nq + 7))
    plan, F, E, Wv = _gpu(enuf, prec, P, pos, q)
    assert plan.info.tile == P["tile"]
    ref, t = Ref(P, pos, q), TOL[prec]
    assert np.all(np.isfinite(F)) and np.all(F[q == 0] == 0.0)
    assert _rel_rms(F, ref.F) < t["F"] and _bead_max(F, ref.F) < 100 * t["F"]
    own = max(abs(ref.E[0]), abs(ref.E[2])) if prec == "fp32" else abs(ref.E[0])
    assert abs(E[0] - ref.E[0]) <= t["E"] * own, (E, ref.E)
    plan.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 8])
@pytest.mark.parametrize("L,M,nq", [(8.0, 12, 300), (9.0, 16, 33), (28.8, 48, 7)])
def test_reduction_spread_grid(enuf, prec, p, L, M, nq):
    """The automatic spreading's grid for every window width (unrolled and not),
    windows across all faces, a grid cleared by the count kernel and one large for
    its beads (cleared by a memset), and the same again on the used workspace."""
    P = dict(L=L, M=M, p=p, alpha=1.0, r_cut=3.0, beta=4.0, kappa=1.1)
    rng = np.random.default_rng(100 * M + p)
    pos = rng.uniform(-0.02 * L, 1.02 * L, (nq + 20, 3))
    q = np.where(np.arange(nq + 20) < nq, rng.choice([-1.0, 1.0, 2.0], nq + 20), 0.0)
    pos, q = _inputs(prec, pos, q)
    plan, F, E, Wv = _gpu(enuf, prec, P, pos, q)
    dt = torch.float32 if prec == "fp32" else torch.float64
    again = torch.empty((nq + 20, 3), dtype=dt, device="cuda")
    plan.energy_forces(torch.tensor(pos, dtype=dt, device="cuda"), torch.tensor(q, dtype=dt, device="cuda"), again)
    grid = plan.debug_buffer(enuf.ENUF_BUF_GRID).astype(np.float64)
    _, _, g_ref, _ = orc.recip_enuf(_oparams(P), pos, q, want_grid=True)
    assert np.abs(grid - g_ref).max() < TOL[prec]["stage"] * np.abs(g_ref).max()
    plan.close()


@pytest.mark.parametrize("deriv", [0, 1])
@pytest.mark.parametrize("n,fft_path", [(108, 0), (108, 1), (180, 0), (216, 0), (288, 0), (300, 0), (360, 0)])
def test_fft_radices_9_15_18(enuf, n, fft_path, deriv):
    """FP32 grids that split into two register radices only with 9, 15 or 18: the
    fields against the Stockham stages' on the same beads (FP32 FFT rounding,
    ~1e-6 of the largest value), forces and energies against the oracle's up to
    n = 216 (its plain DFTs take n^4 steps)."""
    L = n / 5.0
    P = dict(L=L, M=n // 2, p=4, alpha=1.0, r_cut=3.0, beta=4.0, kappa=1.1, fft_path=fft_path, deriv=deriv)
    rng = np.random.default_rng(n)
    pos = rng.uniform(0.0, L, (300, 3))
    q = np.where(np.arange(300) % 2 == 0, 1.0, -1.0)
    pos, q = _inputs("fp32", pos, q)
    plan, F, E, Wv = _gpu(enuf, "fp32", P, pos, q)
    other, F2, E2, _ = _gpu(enuf, "fp32", dict(P, fft_radix=2), pos, q)
    assert plan.info.fft_two_factor == 0 and plan.info.fft_kernels == other.info.fft_kernels
    h, h2 = (x.debug_buffer(enuf.ENUF_BUF_FIELD).astype(np.float64) for x in (plan, other))
    assert np.abs(h - h2).max() < TOL["fp32"]["stage"] * np.abs(h2).max()
    assert _rel_rms(F, F2) < TOL["fp32"]["F"] and abs(E[1] - E2[1]) < TOL["fp32"]["E"] * abs(E2[1])
    if n <= 216:
        _check("fp32", F, E, Wv, Ref(P, pos, q))
    plan.close()
    other.close()


@pytest.mark.parametrize("deriv", [0, 1])
@pytest.mark.parametrize("n", [20, 24, 36, 40, 96, 100, 108])
def test_fft_half_spectrum(enuf, n, deriv):
    """FP64 line passes whose inverse transforms skip the empty half of the spectrum:
    radix 8 (24, 40, 96), 4 (36, 108), and 4 after others in the plan's list (20, 100)."""
    L = n / 5.0
    rc = min(3.0, 0.45 * L)
    P = dict(L=L, M=n // 2, p=3, alpha=3.0 / rc, r_cut=rc, beta=4.0, kappa=1.1, deriv=deriv)
    rng = np.random.default_rng(n)
    pos = rng.uniform(0.0, L, (200, 3))
    q = np.where(np.arange(200) % 2 == 0, 1.0, -1.0)
    plan, F, E, Wv = _gpu(enuf, "fp64", P, pos, q)
    _check("fp64", F, E, Wv, Ref(P, pos, q))
    plan.close()
