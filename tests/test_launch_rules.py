"""The rules that split work items (launch_plan.h) against launches timed on the device with every split
forced, FP32: the split a rule takes is within a quarter of the best one measured, and a batch that runs
faster whole is not split."""

import os
import shutil
import subprocess

import pytest

from paper_1903_03056_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

# (N, species, directions, radial nodes, nodes): us by number of chunks
VSS = {
    (4, 1, 6, 2, 600): {1: 31.5, 2: 41.6}, (4, 2, 7, 2, 1000): {1: 144.1, 2: 166.6},
    (4, 1, 6, 2, 60): {1: 30.9, 2: 27.9}, (6, 1, 6, 3, 600): {1: 47.4, 2: 68.0, 3: 57.5},
    (6, 2, 12, 3, 1): {1: 101.4, 2: 75.5, 3: 53.1}, (8, 1, 6, 3, 600): {1: 49.6, 2: 70.6, 3: 59.0},
    (8, 2, 12, 3, 100): {1: 127.4, 2: 101.9, 3: 74.5}, (8, 1, 6, 4, 2000): {1: 125.0, 2: 137.9, 4: 148.7},
    (12, 1, 6, 6, 400): {1: 155.6, 2: 185.2, 4: 188.6, 6: 189.5},
    (12, 2, 12, 6, 30): {1: 434.7, 2: 273.4, 4: 213.1, 6: 159.8},
    (16, 1, 6, 5, 200): {1: 160.7, 2: 184.8, 4: 186.9, 5: 180.2},
    (16, 2, 12, 5, 1): {1: 407.6, 2: 270.5, 4: 202.6, 5: 134.5},
    (16, 1, 6, 8, 600): {1: 459.2, 2: 547.1, 4: 552.3, 8: 593.3},
    (24, 2, 12, 12, 20): {1: 3122.3, 2: 1831.0, 4: 1439.3, 8: 1431.6},
    (24, 1, 6, 12, 400): {1: 2000.3, 2: 1995.5, 4: 1992.2, 8: 2076.9},
    (32, 1, 6, 9, 20): {1: 390.2, 2: 325.8, 4: 490.8, 8: 452.4},
    (32, 1, 6, 9, 40): {1: 463.6, 2: 649.7, 4: 558.7, 8: 592.9},
    (32, 2, 12, 16, 1): {1: 2411.2, 2: 1415.7, 4: 818.9, 8: 541.3},
    (48, 2, 12, 24, 1): {1: 11791.1, 2: 6342.0, 4: 3795.1, 8: 2597.7},
    (48, 1, 6, 13, 60): {1: 2938.8, 2: 3473.4, 4: 3513.7, 8: 3697.1},
}
VHS = {
    (4, 1, 6, 2, 400): {1: 23.2, 2: 30.0}, (4, 2, 12, 2, 600): {1: 52.7, 2: 61.8},
    (6, 1, 6, 3, 400): {1: 32.0, 2: 43.3, 3: 39.9}, (6, 2, 12, 3, 1): {1: 46.7, 2: 39.7, 3: 29.8},
    (8, 1, 6, 4, 400): {1: 38.1, 2: 45.6, 4: 45.7}, (8, 2, 12, 4, 100): {1: 67.0, 2: 51.4, 4: 54.6},
}
CLUSTERS = {"vss": {4: 1216, 6: 1216, 8: 1216, 12: 608, 16: 304, 24: 304, 32: 76, 48: 76}, "vhs": {4: 1216, 6: 608, 8: 608}}


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("probe") / "launch_probe")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", build.CSRC, "-I", CUDA_INC,
                    os.path.join(ROOT, "tests", "launch_probe.cpp"), "-o", exe], check=True)

    def run(kind, N, s, M, n_rho, nodes):
        antipodal = M in (6, 12, 32)
        tasks = s * (s + 1) // 2 if antipodal else s * s
        most = M if s > 1 or not antipodal else M // 2
        total = s * (s - 1) // 2 * M + s * M // 2 if antipodal else tasks * M
        c = CLUSTERS[kind][N]
        line = ["vss", nodes * tasks, n_rho, c] if kind == "vss" else ["vhs", nodes * tasks, n_rho, c, 0, 1.0]
        line += [most, total / (tasks * most), (24 if kind == "vss" else 6) * c]
        out = subprocess.run([exe], input=" ".join(map(str, line)), capture_output=True, text=True, check=True).stdout
        return int(out.split()[1])

    return run


@pytest.mark.parametrize("kind,case", [("vss", c) for c in VSS] + [("vhs", c) for c in VHS])
def test_the_split_is_near_the_best_measured_one(probe, kind, case):
    times = (VSS if kind == "vss" else VHS)[case]
    got = probe(kind, *case)
    assert got in times and times[got] <= 1.25 * min(times.values()), got
    if times[1] == min(times.values()):
        assert got == 1
