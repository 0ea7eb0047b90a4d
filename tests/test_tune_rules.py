"""The tuner's rules on the CPU: which objects a variant links and which radix schedule it keeps."""

import os

from paper_1903_03056_gb300 import build, tune


def test_a_variant_links_the_librarys_own_objects_only(tmp_path, monkeypatch):
    monkeypatch.setattr(build, "BUILD", str(tmp_path))
    names = [os.path.splitext(f)[0] for f in build.SOURCES]
    for n in names + ["left_over"]:  # the object of a source that is no longer there
        (tmp_path / (n + ".o")).write_bytes(b"")
    linked = [os.path.splitext(os.path.basename(f))[0] for f in tune.other_objects("collision_f32")]
    assert sorted(linked) == sorted(n for n in names if n != "collision_f32")


def test_equal_times_are_decided_by_the_error():
    rows = [{"radix": 28, "ms": 145.5, "err_vs_fp64": 1.32e-6}, {"radix": 44, "ms": 146.0, "err_vs_fp64": 1.21e-6},
            {"radix": 422, "ms": 147.5, "err_vs_fp64": 1.0e-6}]
    assert tune.best_radix(rows)["radix"] == 44
    assert tune.best_radix(rows[::2])["radix"] == 28
