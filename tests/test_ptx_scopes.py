"""Ordering between the CTAs of a cluster, read from the kernels' sources on CPU:
an mbarrier arrive on another CTA's barrier orders that CTA's reads only if it
names the cluster scope (the default scope is the CTA's own).  A stale operand
would be a wrong result without an error, on no particular input, so the rule is
checked where it is written."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_2408_14070_gb300", "csrc", "*.cu*")))


def _arrives(text):
    return re.findall(r"mbarrier\.arrive(?!\.expect_tx)[\w.:]*shared::cluster[\w.:]*", text)


def test_remote_arrives_name_the_cluster_scope():
    seen = 0
    for path in SOURCES:
        for op in _arrives(open(path).read()):
            seen += 1
            assert re.match(r"mbarrier\.arrive\.(release|relaxed)\.cluster\.shared::cluster", op), (path, op)
    assert seen >= 2


def test_relaxed_arrives_follow_a_release_fence():
    for path in SOURCES:
        lines = [l.strip() for l in open(path).read().splitlines()]
        for i, l in enumerate(lines):
            if "mbarrier.arrive.relaxed.cluster" in l:
                assert "fence.release" in lines[i - 1] and ".cluster" in lines[i - 1], (path, i + 1)
