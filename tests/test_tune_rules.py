"""The tuner's rules on the CPU: which objects a variant links, which shapes it tries, which radix
schedule it keeps; the shape table."""

import os
import re

from paper_1903_03056_gb300 import build, tune


def test_a_variant_links_the_librarys_own_objects_only(tmp_path, monkeypatch):
    monkeypatch.setattr(build, "BUILD", str(tmp_path))
    names = [os.path.splitext(f)[0] for f in build.SOURCES]
    for n in names + ["left_over"]:  # the object of a source that is no longer there
        (tmp_path / (n + ".o")).write_bytes(b"")
    linked = [os.path.splitext(os.path.basename(f))[0] for f in tune.other_objects("collision_f32")]
    assert sorted(linked) == sorted(n for n in names if n != "collision_f32")


def test_equal_times_are_decided_by_the_error():
    # the largest error of a few nodes says little: the 2-norm decides
    rows = [{"radix": 28, "ms": 145.5, "err_vs_fp64": 1.8e-6, "l2_vs_fp64": 1.32e-6},
            {"radix": 44, "ms": 148.0, "err_vs_fp64": 2.7e-6, "l2_vs_fp64": 1.21e-6},
            {"radix": 422, "ms": 149.5, "err_vs_fp64": 1.0e-6, "l2_vs_fp64": 1.0e-6}]
    assert tune.best_radix(rows)["radix"] == 44
    assert tune.best_radix(rows[::2])["radix"] == 28
    rows[0]["l2_vs_fp64"] = 1.23e-6  # 2 % more than the best: the present order stays
    assert tune.best_radix(rows, current=28)["radix"] == 28 and tune.best_radix(rows, current=422)["radix"] == 44


def test_a_run_tries_the_librarys_own_shape():
    for precision in ("fp32", "fp64"):
        for N in tune.WORKLOAD_FOR_N:
            tried = tune.shape_candidates(precision, N)
            assert tune.current_shape(precision, N) in tried and set(tune.CANDIDATES[N]) <= set(tried)


def test_small_grids_are_sized_for_enough_warps():
    """FP32 shapes whose CTAs are a few warps name the CTAs per SM: sized for one, the compiler takes up to
    255 registers a thread and an SM holds 4 to 10 warps of 64."""
    text = open(tune.SHAPES_H).read()
    rows = re.findall(r"^DGFS_(SHAPE3|VSS)\(float, (\d+), (\d+), (\d+), (\d+)\)$", text, re.M)
    assert len(rows) == 16
    for kind, N, cluster, groups, ctas in rows:
        if kind == "VSS" and N == "4":
            continue  # one warp a CTA: 8 CTAs fit whatever it is sized for, more measured 3 to 8 % slower
        warps = (int(groups) * int(N) + 31) // 32
        assert warps * int(ctas) >= 8, (kind, N)
