"""bench.py's labels and profile figures: the histogram path from the stages that
the library reports, and a kernel's figures only for the source they are of."""
import os
import shutil
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_path_labels_follow_the_stages():
    own = {"range": 1.0, "prep": 1.0, "integral_image": 1.0, "lookup": 1.0}
    assert bench.path_of({**own, "fused_sweep": 1.0}) == "fused"
    assert bench.path_of({**own, "compact_histogram": 1.0}) == "compact"
    assert bench.path_of({**own, "integral_histogram": 1.0}) == "materialised"
    assert bench.batch_passes({"batch": 1.0}) == ["fused"]
    assert bench.batch_passes({"batch_materialised": 1.0}) == ["materialised"]
    assert bench.batch_passes({"batch": 1.0, "batch_materialised": 1.0}) == ["fused", "materialised"]
    assert bench.batch_passes({"batch_materialised": 1.0, "batch_compact": 1.0}) == ["compact"]


def test_a_kernels_hash_covers_its_headers(tmp_path, monkeypatch):
    """Most of the lookup's arithmetic is in headers: an edit there drops its figures."""
    import paper_2102_01289_gb300 as tm

    shutil.copytree(os.path.join(tm.PKG, "csrc"), tmp_path / "csrc")
    monkeypatch.setattr(tm, "PKG", str(tmp_path))
    before = {k: bench.kernel_source_hash(k) for k in ("lookup_compact", "fused_sweep", "bwd_pixel")}
    assert None not in before.values() and bench.kernel_source_hash("no_such_kernel") is None
    for name in ("tm_common.cuh", "tm_lookup.cuh", "tm_compact.cu"):
        with open(tmp_path / "csrc" / name, "a") as fh:
            fh.write("\n// edited\n")
        after = {k: bench.kernel_source_hash(k) for k in before}
        assert after["lookup_compact"] != before["lookup_compact"]
        assert (after["fused_sweep"] == before["fused_sweep"]) == (name == "tm_compact.cu")
        before = after
