"""A cached tuning is used only for the kernel sources that it was measured on
(CPU), and complex64 is not tuned over the march option, whose values -1 and 1
run the same kernels there."""
from paper_2308_13476_gb300 import autotune


def test_entry_of_other_sources_is_not_used():
    key = autotune.cache_key("GPU", 8, 8, 2, "mixed", "gmres3", "V", 2)
    best = {"best": {"tile_rows": 1}, "results": []}
    assert autotune.cached({}, key) is None
    assert autotune.cached({key: best}, key) is None                          # written before sources were recorded
    assert autotune.cached({key: dict(best, sources="0" * 16)}, key) is None
    hit = dict(best, sources=autotune.sources_digest())
    assert autotune.cached({key: hit}, key) == hit


def test_digest_follows_the_sources(tmp_path, monkeypatch):
    import os
    import shutil
    d = tmp_path / "pkg"
    shutil.copytree(os.path.join(os.path.dirname(autotune.__file__), "csrc"), d / "csrc")
    monkeypatch.setattr(autotune, "__file__", str(d / "autotune.py"))
    a = autotune.sources_digest()
    assert a == autotune.sources_digest()
    with open(d / "csrc" / "common.cuh", "a") as f:
        f.write("\n")
    assert a != autotune.sources_digest()


def test_march_is_tuned_in_complex128_only():
    assert any("march" in s for s in autotune.default_stages("fp64"))
    for precision in ("mixed", "mixed-ff"):
        stages = autotune.default_stages(precision)
        assert not any("march" in s for s in stages) and any("kron_chunk" in s for s in stages)
