"""Kernels that write into other CTAs' shared memory: every CTA of the cluster has to have
started before the first such store and must not exit before the last one has landed, so a
cluster barrier comes before the first and after the last store (read from the sources)."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def cluster_kernels():
    found = []
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2211_15383_gb300", "csrc", "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__cluster_dims__\([^)]*\)\s*(\w+)\s*\(", text):
            start = text.index("{", m.end())
            depth, i = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            found.append((m.group(1), text[start:i]))
    return found


@pytest.mark.parametrize("name,body", cluster_kernels(), ids=[k for k, _ in cluster_kernels()])
def test_barriers_around_remote_stores(name, body):
    stores = [m.start() for m in re.finditer(r"\bcluster_store\(", body)]
    barriers = [m.start() for m in re.finditer(r"\bcluster_barrier\(\)", body)]
    assert stores and barriers
    assert barriers[0] < stores[0], f"{name}: remote store before every CTA is known to have started"
    assert barriers[-1] > stores[-1], f"{name}: CTAs may exit before a remote store has landed"
