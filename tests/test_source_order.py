"""Orders that the kernels' sources have to keep and that no run can be relied on to show: another CTA's shared
memory is written only after a cluster barrier has shown that every CTA of the cluster runs."""
import os
import re

import pytest

from paper_2607_15498_gb300 import build

REMOTE = r"map_shared_rank\(|mapa\.|cluster_addr\("
START = r"cluster\.sync\(\)|cluster\.barrier_wait\(\)|cluster_barrier\(\)"


def kernel_body(file, kernel):
    """Body of a kernel, without comments."""
    text = open(os.path.join(build.CSRC, file)).read()
    text = re.sub(r"//[^\n]*", "", text)
    at = text.index("{", text.index(f"{kernel}("))
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at + 1:i]
    raise AssertionError("unbalanced braces")


@pytest.mark.parametrize("file, kernel", [("allocate.cu", "allocate_kernel"), ("pack.cu", "pack_tables_kernel"),
                                          ("anchor_search.cu", "anchor_search_tc_kernel")])
def test_remote_shared_memory_after_a_cluster_barrier(file, kernel):
    body = kernel_body(file, kernel)
    remote = re.search(REMOTE, body).start()
    before = body[:remote]
    starts = [m.start() for m in re.finditer(START, before)]
    assert starts, "no cluster barrier before the first access to another CTA's shared memory"
    # and one that every thread passes: not inside a conditional block
    assert any(before[:s].count("{") == before[:s].count("}") for s in starts)
