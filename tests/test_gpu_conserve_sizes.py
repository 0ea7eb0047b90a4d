"""Projection and species sum at the grid sizes whose blocks are shared by one CTA (N = 4 to 8) and by eight
(N = 24 to 48): the oracle's projection of the operators the library itself returns without the flag."""

import numpy as np
import pytest

from gpu_helpers import TOL_FP64
from oracle import fast_spectral as fs, moments
from paper_1903_03056_gb300 import dgfs, synth

pytestmark = pytest.mark.gpu

# FP32: sums and projection are in FP64, so one rounding of the result (2^-24 of the largest value)
ROUNDING = 1.2e-7


def evaluate(f, precision, flags, **kw):
    import torch
    plan = dgfs.Plan(kw["N"], 6.0, kw["masses"], 0.7, M=6, N_rho=2, precision=precision, flags=flags,
                     kappa=kw.get("kappa"), max_batch=f.shape[0])
    Q = plan.eval(torch.from_numpy(f).to(device="cuda", dtype=torch.float64 if precision == "fp64" else torch.float32))
    torch.cuda.synchronize()
    out = Q.double().cpu().numpy()
    plan.close()
    return out


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N,s", [(4, 3), (6, 2), (8, 2), (24, 2), (32, 2), (48, 2)])
def test_projection_and_sum(N, s, precision):
    masses = [1.0, 2.3, 1.6][:s]
    f = np.random.default_rng(N).random((2, s, N, N, N))
    b = fs.make_problem(N, 6.0, masses, omega=0.7, M=6, N_rho=2).b
    raw = evaluate(f, precision, 0, N=N, masses=masses)
    ref = np.stack([moments.conservation_projection(q, masses, 6.0, b) for q in raw])
    tol = TOL_FP64 if precision == "fp64" else ROUNDING
    got = evaluate(f, precision, dgfs.DGFS_CONSERVE, N=N, masses=masses)
    assert np.max(np.abs(got - ref)) <= tol * np.max(np.abs(ref))
    assert np.max(np.abs(raw - ref)) > 100 * tol * np.max(np.abs(ref))  # there is something to project
    kappa = np.random.default_rng(s).uniform(0.3, 2.0, (s, s))
    for flags, q in ((dgfs.DGFS_SUM_SPECIES, raw), (dgfs.DGFS_SUM_SPECIES | dgfs.DGFS_CONSERVE, ref)):
        want = np.stack([moments.species_sum(x, kappa) for x in q])
        got = evaluate(f, precision, flags, N=N, masses=masses, kappa=kappa)
        assert np.max(np.abs(got - want)) <= tol * np.max(np.abs(want))
