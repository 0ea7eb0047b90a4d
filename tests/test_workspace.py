"""The collision workspaces under short memory and the bytes a plan reports, with an allocator that refuses
what passes a limit (CPU): a plan is refused only when the smallest workspace does not fit."""

import json
import os
import shutil
import subprocess

import pytest

from paper_1903_03056_gb300 import build, dgfs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
GUARDS = 2 * 4096
# the VSS workspace of three species at N = 48 (M = 32): 76 clusters, 24 parts each
VSS48 = dict(N=48, s=3, precision=1, flags=0, max_batch=0, c0=76, c1=0, slot=1200000, slots=1824, size=117456, tasks=6,
             n_rho=24, vss=1)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs g++ and the CUDA headers")
    libdir = os.path.dirname(build.build())
    exe = str(tmp_path_factory.mktemp("probe") / "workspace_probe")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", build.CSRC, "-I", CUDA_INC,
                    os.path.join(ROOT, "tests", "workspace_probe.cpp"), "-o", exe, "-L", libdir, "-ldgfs",
                    "-Wl,-rpath," + libdir], check=True)

    def run(limit=1 << 60, batch=0, **kw):
        words = list(kw.values()) + [limit, batch]
        return json.loads(subprocess.run([exe], input=" ".join(map(str, words)), capture_output=True, text=True,
                                         check=True).stdout)

    return run


def test_enough_memory_keeps_the_whole_workspace(probe):
    r = probe(**VSS48)
    assert r["rc"] == 0 and r["scratch"] == r["wanted"] == (76 * 1200000 + 1824 * 117456) * 8
    assert r["clusters"] == [76, 0] and r["part_slots"] == 1824


@pytest.mark.parametrize("limit,clusters,slots", [
    (2_300_000_000, 76, 0),   # no room for split items
    (400_000_000, 38, 0),     # half the clusters
    (10_000_000, 1, 0),       # one
])
def test_short_memory_shrinks_the_workspace(probe, limit, clusters, slots):
    r = probe(limit=limit, **VSS48)
    assert r["rc"] == 0 and r["clusters"] == [clusters, 0] and r["part_slots"] == slots
    assert r["scratch"] == clusters * 1200000 * 8 and r["used"] == r["scratch"] + GUARDS + r["counters"] <= limit


def test_two_shapes_share_the_smaller_workspace(probe):
    r = probe(limit=200 << 20, N=32, s=2, precision=1, flags=0, max_batch=0, c0=228, c1=57, slot=254000, slots=1368,
              size=16384, tasks=3, n_rho=16, vss=0)
    assert r["rc"] == 0 and r["clusters"] == [57, 15] and r["part_off"] == 57 * 254000


def test_less_than_one_cluster_is_refused(probe):
    assert probe(limit=9_000_000, **VSS48)["rc"] == dgfs.DGFS_ERR_OOM


@pytest.mark.parametrize("batch", [0, 700])
def test_reported_bytes_hold_every_array_of_the_workspace(probe, batch):
    """Workspace, guards and counters, the staged operators and the projection's multipliers; for a host-buffer
    call the second workspace and its counters, inputs and outputs."""
    flags = dgfs.DGFS_CONSERVE | dgfs.DGFS_SUM_SPECIES
    r = probe(batch=batch, N=24, s=2, precision=1, flags=flags, max_batch=1000, c0=304, c1=90, slot=100000, slots=1824,
              size=6912, tasks=3, n_rho=12, vss=0)
    n3 = 24 ** 3 * 4
    one = r["scratch"] + GUARDS + (64 + 1824) * 4
    want = one + 1000 * 4 * n3 + 1000 * 3 * 6 * 8
    if batch:  # chunks of a pipelined batch are too large to split: no room for split items there
        want += one - 1824 * (6912 * 8 + 4) + batch * (2 + 2) * n3
    assert r["reported"] == want


def test_the_second_workspace_has_room_for_split_items_only_where_chunks_can_split(probe):
    r = probe(**VSS48)  # 249 nodes are 1494 items of 8 parts
    assert r["part_slots2"] == 0 and r["second"] == 76 * 1200000 * 8
    small = dict(N=4, s=1, precision=1, flags=0, max_batch=0, c0=1216, c1=0, slot=880, slots=7296, size=32, tasks=1, n_rho=2, vss=0)
    r = probe(**small)  # 249 items of two radial nodes
    assert r["part_slots2"] == 7296 and r["second"] == r["scratch"]
    assert probe(**dict(small, n_rho=30))["part_slots2"] == 0
