"""What a cached launch shape is keyed by, and which shapes are timed.  No GPU needed."""
import os
import shutil

from paper_1509_08391_gb300 import autotune, build, workloads


def test_a_shape_tuned_for_another_kernel_is_not_found(tmp_path, monkeypatch):
    w = workloads.small_l4()
    autotune._kernel_version.cache_clear()
    here = autotune._key(w, "GPU")
    assert here != "GPU|L=4|n=8"            # the key of a cache without a version
    assert here.endswith("|n=%d" % w.n_lattices)
    src = tmp_path / "csrc"
    shutil.copytree(build.CSRC, src)
    monkeypatch.setattr(build, "CSRC", str(src))
    try:
        autotune._kernel_version.cache_clear()
        assert autotune._key(w, "GPU") == here
        with open(os.path.join(src, "llr_chain.cu"), "a") as f:
            f.write("// another kernel\n")
        autotune._kernel_version.cache_clear()
        assert autotune._key(w, "GPU") != here
    finally:
        autotune._kernel_version.cache_clear()


def test_no_launch_is_timed_twice():
    assert not {160, 192} <= set(autotune.SHAPES)
    assert not {2, 4} <= set(autotune.RINGS)
