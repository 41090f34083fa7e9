"""bench.py names the histogram path from the stages that the library reports."""
import os
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
