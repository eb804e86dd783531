"""bench.py's roofline counts the bytes that the traversal reads: a child slot
of the default tree is a quarter of the node that the library's header lays
out, and the records of both workloads are counted with it."""
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_slot_bytes_are_the_nodes():
    src = open(os.path.join(ROOT, "paper_1912_04000_gb300", "csrc", "rt_internal.h")).read()
    node = int(re.search(r"kNode4Bytes = (\d+)", src).group(1))
    assert bench.NODE4_SLOT_BYTES == node / 4
    calls = [c for c in re.findall(r"= trace_roofline\((.*)\)", open(os.path.join(ROOT, "bench.py")).read())]
    assert len(calls) == 2 and all("NODE4_SLOT_BYTES" in c for c in calls)


def test_slot_bytes_counted():
    class Probe:
        def probe_l2(self):
            return 20_000.0

    counts = {"nodes_visited": 41_000, "tris_tested": 2_000, "ext_rays": 1_000,
              "shadow_nodes_visited": 20_000, "shadow_tris_tested": 1_500, "shadow_rays": 1_000}
    roof = bench.trace_roofline(Probe(), counts, 13.0, 10, 2e7, slot_bytes=bench.NODE4_SLOT_BYTES)
    assert roof["algorithmic_bytes_per_ray"] == 41.0 * 24 + 2.0 * 48 + 32 + 8
