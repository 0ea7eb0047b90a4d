"""Collision kernel on states that fill every mode: white noise on the grid has as much in the
unpaired modes (index N/2 of an axis) as anywhere else, so every face and edge term of the real
transforms enters at full size.  Rules with shifts of zero along an axis, with and without antipodes,
one to three species; every grid size the library supports; VHS, and VSS, whose products stay complex and
whose weights differ between a mode and its negative on the faces of the unpaired modes."""

import numpy as np
import pytest

from gpu_helpers import TOL_FP32, TOL_FP64, gpu_collision, max_rel_error, oracle_collision

pytestmark = pytest.mark.gpu


def _rule(kind):
    """(sigma [M, 3], weights [M]) or (None, None) for the built-in icosahedron."""
    if kind == "icosahedron":
        return None, None
    if kind == "axes":      # zero shift along two axes of every direction
        return np.array([[1, 0, 0], [0, 1, 0], [0, 0, -1]], float), np.array([4.0, 5.0, 3.0])
    rng = np.random.default_rng(7)   # no antipodes, two directions of one sigma_x group, uneven weights
    s = rng.normal(size=(3, 3))
    s /= np.linalg.norm(s, axis=1, keepdims=True)
    s = np.concatenate([s, s[:1] * [1.0, -1.0, 1.0]])
    return s, np.array([3.0, 5.5, 2.0, 2.5])


CASES = [(N, kind, s, n_rho) for N in (4, 6, 8, 12) for kind, s, n_rho in
         (("icosahedron", 2, 3), ("axes", 3, 2), ("general", 2, 3), ("general", 1, 1))]
CASES += [(N, "general", 2, 2) for N in (16, 24, 32, 48)]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N,kind,s,n_rho", CASES)
def test_white_noise_state_matches_the_oracle(N, kind, s, n_rho, precision):
    f = np.random.default_rng(N + s).random((2 if N <= 12 else 1, s, N, N, N))
    sigma, w = _rule(kind)
    kw = dict(N=N, L=5.0, masses=[1.0, 2.3, 1.6][:s], omega=0.7, M=12, N_rho=n_rho, sigma=sigma, w_sigma=w)
    if precision == "fp32":
        f = f.astype(np.float32).astype(np.float64)
    got, ref = gpu_collision(f, precision=precision, **kw), oracle_collision(f, **kw)
    # the bounds of the parity tests: FP64 per pair, FP32 per node
    if precision == "fp64":
        assert max_rel_error(got, ref, "pair") < TOL_FP64
    else:
        assert max_rel_error(got, ref, "node") < TOL_FP32


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N,kind,s,n_rho", [(N, kind, s, 2) for N in (4, 6, 8, 12)
                                            for kind, s in (("icosahedron", 2), ("axes", 2), ("general", 1))]
                         + [(16, "general", 2, 1), (24, "general", 2, 1)])
def test_white_noise_state_with_vss_matches_the_oracle(N, kind, s, n_rho, precision):
    f = np.random.default_rng(10 * N + s).random((1, s, N, N, N))
    sigma, w = _rule(kind)
    kw = dict(N=N, L=5.0, masses=[1.0, 2.3][:s], omega=0.7, alpha=1.4, M=12, N_rho=n_rho, sigma=sigma, w_sigma=w)
    if precision == "fp32":
        f = f.astype(np.float32).astype(np.float64)
    got, ref = gpu_collision(f, precision=precision, **kw), oracle_collision(f, **kw)
    if precision == "fp64":
        assert max_rel_error(got, ref, "pair") < TOL_FP64
    else:
        assert max_rel_error(got, ref, "node") < TOL_FP32
