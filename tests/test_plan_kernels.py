"""The kernels a plan runs, from the host logic alone (enuf_plan_kernels), and the
autotuner's choice between them. CPU only."""
import pytest


@pytest.fixture(scope="module")
def mods():
    from paper_1303_4523_gb300 import build
    build.build()
    from paper_1303_4523_gb300 import autotune, enuf
    return autotune, enuf


BASE = dict(alpha=1.0, r_cut=3.0, beta=4.0, kappa=1.0, p=4)
EXT = {108: (9, 12), 180: (12, 15), 216: (12, 18), 288: (16, 18), 300: (15, 20), 324: (18, 18), 360: (18, 20)}


def _kernels(E, n, **kw):
    k = E.plan_kernels(E.make_params(L=n / 3.2, M=n // 2, **dict(BASE, **kw)), 1000)
    return (k.fft_f1, k.fft_f2), k.spread


def test_two_factor_splits_that_run(mods):
    """Every length with a split over 4, 5, 6, 8, 10, 12, 16, 20, or else with 9, 15 and
    18, runs the two-factor kernels unless Stockham stages are asked for."""
    _, E = mods
    for n, f in {**EXT, 96: (8, 12), 320: (16, 20)}.items():
        assert _kernels(E, n, prec="fp32")[0] == f
        for kw in (dict(prec="fp32", fft_radix=1), dict(prec="fp32", fft_radix=2), dict(prec="fp64")):
            assert _kernels(E, n, **kw)[0] == (0, 0)
    for n in (12, 512):   # no split
        assert _kernels(E, n, prec="fp32", r_cut=1.5)[0] == (0, 0)


def test_spreading_form_that_runs(mods):
    """0 runs reductions in both precisions; a form asked for runs itself."""
    _, E = mods
    assert _kernels(E, 96, prec="fp32")[1] == 5 and _kernels(E, 160, prec="fp32")[1] == 5
    assert _kernels(E, 96, prec="fp64")[1] == 5 and _kernels(E, 96, prec="fp64", spread=1)[1] == 1
    for form in (1, 2, 3, 4):
        assert _kernels(E, 160, prec="fp32", spread=form)[1] == form
    with pytest.raises(E.EnufError):
        _kernels(E, 96, prec="fp64", spread=2)


def test_autotuner_offers_both_line_transforms(mods):
    """A grid that splits with 9, 15 or 18 only: the two-factor kernels (0) and the
    Stockham stages (2) are different candidates, as on the other split lengths."""
    A, E = mods
    for n in EXT:
        c = A.candidates(E.make_params(L=n / 3.2, M=n // 2, prec="fp32", **BASE), 1000)
        tiles = {x["tile"] for x in c}
        assert tiles
        for t in tiles:
            assert {0, 2} <= {x["fft_radix"] for x in c if x["tile"] == t}, (n, t)
