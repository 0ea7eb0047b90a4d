"""Small VHS batches run with their radial nodes split into chunks, and on some grids in a launch
shape of their own; a node's result is bit for bit the one it has inside a batch that fills the
device and runs unsplit."""

import numpy as np
import pytest

from paper_1903_03056_gb300 import dgfs, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("N,batch", [(4, 20000), (6, 8000), (8, 4000), (12, 1500), (16, 1000), (24, 400),
                                     (32, 400), (48, 140)])
def test_a_node_alone_and_in_a_full_batch_give_the_same_bits(N, batch, precision):
    import torch
    dt = torch.float32 if precision == "fp32" else torch.float64
    # N_rho = 5 does not divide into the chunks evenly; the full batch's products outnumber any
    # parts buffer, so it runs unsplit
    w = synth.Workload("split", 3, N, 5.0, (1.0, 2.1), 0.7, 1.0, 6, 5, "bimaxwellian", 0.05, 90)
    few = torch.from_numpy(synth.batch_distribution(w)).to(device="cuda", dtype=dt)
    full = few.repeat((batch + 2) // 3, 1, 1, 1, 1)[:batch].contiguous()
    plan = dgfs.Plan(N, 5.0, [1.0, 2.1], 0.7, M=6, N_rho=5, precision=precision)
    ref = plan.eval(full)
    for b in (1, 2, 3):
        assert torch.equal(plan.eval(few[:b].contiguous()), ref[:b])
    plan.set_sm_share(0.1)  # fewer clusters: another split of the same items
    assert torch.equal(plan.eval(few), ref[:3])
    torch.cuda.synchronize()
    assert plan.check()
    plan.close()


def test_a_split_evaluation_replays_from_a_graph():
    import torch
    w = synth.Workload("split", 2, 16, 5.0, (1.0, 2.1), 0.7, 1.0, 6, 5, "bimaxwellian", 0.05, 91)
    f = torch.from_numpy(synth.batch_distribution(w)).to(device="cuda", dtype=torch.float32)
    plan = dgfs.Plan(16, 5.0, [1.0, 2.1], 0.7, M=6, N_rho=5, precision="fp32")
    ref = plan.eval(f)
    Q = torch.zeros_like(ref)
    g = plan.capture(f, Q)
    for _ in range(3):
        Q.fill_(np.nan)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(Q, ref)
    plan.close()


def test_plans_of_one_shape_with_different_sphere_rules_stay_usable():
    """Two plans share a kernel and differ in its shared memory (phase blocks of 32 and 6 directions):
    creating and running the smaller one leaves the larger one usable."""
    import torch
    w = synth.Workload("split", 2, 16, 5.0, (1.0, 2.1), 0.7, 1.0, 6, 3, "bimaxwellian", 0.05, 92)
    f = torch.from_numpy(synth.batch_distribution(w)).to(device="cuda", dtype=torch.float32)
    large = dgfs.Plan(16, 5.0, [1.0, 2.1], 0.7, M=32, N_rho=3, precision="fp32")
    ref = large.eval(f)
    small = dgfs.Plan(16, 5.0, [1.0, 2.1], 0.7, M=6, N_rho=3, precision="fp32")
    small.eval(f)
    assert torch.equal(large.eval(f), ref)
    torch.cuda.synchronize()
    large.close()
    small.close()


@pytest.mark.parametrize("N,N_rho,s,M,few,many,precision", [
    (8, 10, 2, 6, 3, 1500, "fp32"),   # parts of one and two radial nodes
    (8, 3, 2, 12, 2, 3000, "fp64"),    # fewer radial nodes than parts
    (12, 9, 2, 6, 40, 1200, "fp32"),  # groups that share a barrier
    (16, 8, 3, 32, 1, 400, "fp32"),   # clusters of two, three species
    (24, 17, 2, 12, 2, 700, "fp32"),
    (6, 1, 1, 6, 1, 5, "fp32"),       # one radial node: never split
])
def test_vss_nodes_do_not_depend_on_the_split(N, N_rho, s, M, few, many, precision):
    """A VSS node's bits are the same alone, where its items split over the parts of the radial sum,
    and in a batch whose items run whole."""
    import torch
    masses = [1.0, 2.1, 0.6][:s]
    w = synth.Workload("vss_split", few, N, 5.0, tuple(masses), 0.7, 1.4, M, N_rho, "bimaxwellian", 0.05, 17)
    dt = torch.float64 if precision == "fp64" else torch.float32
    f = torch.from_numpy(synth.batch_distribution(w)).to(device="cuda", dtype=dt)
    plan = dgfs.Plan(N, 5.0, masses, 0.7, alpha=1.4, M=M, N_rho=N_rho, precision=precision)
    ref = plan.eval(f)
    batch = f.repeat((many + few - 1) // few, 1, 1, 1, 1)[:many].contiguous()
    Q = plan.eval(batch)
    torch.cuda.synchronize()
    for b in range(many):
        assert torch.equal(Q[b], ref[b % few])
    assert torch.equal(plan.eval(f), ref)
    plan.close()
