"""Split and whole work items on states that fill every mode and sphere rules with shifts along all axes, so
that every face, edge and corner term enters: a node has the same bits alone and in a batch that certainly
runs whole (more items than any device could hold parts of), and VSS sums of several parts meet the oracle."""

import numpy as np
import pytest

from gpu_helpers import TOL_FP32, TOL_FP64, gpu_collision, max_rel_error, oracle_collision
from paper_1903_03056_gb300 import dgfs

pytestmark = pytest.mark.gpu

# at most 32 CTAs on each of 152 SMs
MOST_CLUSTERS = 32 * 152


def general_rule(M=4):
    rng = np.random.default_rng(7)
    s = rng.normal(size=(M - 1, 3))
    s /= np.linalg.norm(s, axis=1, keepdims=True)
    return np.concatenate([s, s[:1] * [1.0, -1.0, 1.0]]), rng.uniform(2.0, 5.0, M)


@pytest.mark.parametrize("N,batch,precision,alpha,n_rho", [
    (8, 5000, "fp32", 1.0, 8), (12, 3000, "fp32", 1.0, 5), (16, 1500, "fp32", 1.0, 5), (24, 600, "fp32", 1.0, 5),
    (32, 500, "fp32", 1.0, 5), (48, 160, "fp32", 1.0, 5), (8, 5000, "fp64", 1.0, 8), (16, 1500, "fp64", 1.0, 5),
    (32, 100, "fp64", 1.0, 5), (8, 3700, "fp32", 1.4, 10), (8, 10000, "fp64", 1.4, 3), (16, 3700, "fp32", 1.4, 8),
    (32, 600, "fp32", 1.4, 8), (48, 250, "fp32", 1.4, 8),
])
def test_a_node_has_the_same_bits_split_and_whole(N, batch, precision, alpha, n_rho):
    import torch
    sigma, w = general_rule()
    dt = torch.float32 if precision == "fp32" else torch.float64
    few = torch.from_numpy(np.random.default_rng(N).random((2, 2, N, N, N))).to(device="cuda", dtype=dt)
    plan = dgfs.Plan(N, 5.0, [1.0, 2.3], 0.7, alpha=alpha, N_rho=n_rho, precision=precision, sigma=sigma, w_sigma=w)
    if N <= 16:  # (larger grids hold at most 4 CTAs an SM: their batches are far beyond the room for parts)
        assert 4 * batch * min(8, n_rho) > (24 if alpha != 1.0 else 6) * MOST_CLUSTERS
    whole = plan.eval(few.repeat(batch // 2, 1, 1, 1, 1))
    torch.cuda.synchronize()
    assert bool((whole[::2] == whole[0]).all()) and bool((whole[1::2] == whole[1]).all())
    for b in (1, 2):
        assert torch.equal(plan.eval(few[:b].contiguous()), whole[:b])
    torch.cuda.synchronize()
    assert plan.check()
    plan.close()


_ORACLE = {}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N,n_rho", [(16, 3), (32, 2), (48, 2)])
def test_vss_sum_of_parts_matches_the_oracle(N, n_rho, precision):
    f = np.random.default_rng(10 * N).random((1, 1, N, N, N)).astype(np.float32).astype(np.float64)
    sigma, w = general_rule()
    kw = dict(N=N, L=5.0, masses=[1.0], omega=0.7, alpha=1.4, N_rho=n_rho, sigma=sigma, w_sigma=w)
    if (N, n_rho) not in _ORACLE:
        _ORACLE[N, n_rho] = oracle_collision(f, **kw)
    got = gpu_collision(f, precision=precision, **kw)
    if precision == "fp64":
        assert max_rel_error(got, _ORACLE[N, n_rho], "pair") < TOL_FP64
    else:
        assert max_rel_error(got, _ORACLE[N, n_rho], "node") < TOL_FP32
