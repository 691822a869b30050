"""The block rules of a batched launch (FP32): systems with no, few and all beads
charged, and batches on both sides of the block order's size line, against single
plans (the bound of test_batch_equals_single_plans: both sides round in FP32)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_enuf import _rel_rms, enuf  # noqa: E402,F401


@pytest.mark.parametrize("name,systems", [
    # (beads, charged): blocks without beads, a system of one block, every block full
    ("mixed", [(600, 600), (3000, 0), (5000, 2), (1024, 1), (4100, 4100), (20000, 150)]),
    # more blocks than two to a place: a system's blocks together
    ("large", [(81000, 8100)] * 7 + [(81000, 81000), (3000, 3000)]),
])
def test_charged_fractions(enuf, name, systems):
    rng = np.random.default_rng(len(systems))
    params, pos, q, F, ref = [], [], [], [], []
    for N, nq in systems:
        L = (N / 3.0) ** (1.0 / 3.0)
        params.append(enuf.make_params(prec="fp32", L=L, M=0, p=4, alpha=0.975, r_cut=min(3.0, 0.5 * L), beta=4.0,
                                       kappa=1.1))
        c = np.zeros(N)
        c[:nq] = np.where(np.arange(nq) % 2 == 0, 1.0, -1.0)
        pos.append(torch.tensor(rng.uniform(0.0, L, (N, 3)), dtype=torch.float32, device="cuda"))
        q.append(torch.tensor(rng.permutation(c), dtype=torch.float32, device="cuda"))
        F.append(torch.full_like(pos[-1], float("nan")))
        one = enuf.Plan(params[-1], N)
        Fs = torch.empty_like(pos[-1])
        E, _ = one.energy_forces(pos[-1], q[-1], Fs)
        ref.append((Fs.double().cpu().numpy(), E))
        one.close()
    b = enuf.Batch(params, [N for N, _ in systems])
    assert b.mode() == 1
    for _ in range(2):
        E = b.energy_forces(pos, q, F)
        for k, (Fs, Es) in enumerate(ref):
            Fb = F[k].double().cpu().numpy()
            assert np.all(np.isfinite(Fb)) and (_rel_rms(Fb, Fs) < 1e-6 or not Fs.any())
            assert np.allclose(E[k], Es, rtol=1e-6, atol=1e-6 * np.abs(Es).max())
    b.close()
