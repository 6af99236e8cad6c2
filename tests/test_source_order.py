"""Orders that the kernels' sources have to keep and that no run can be relied on to show: another CTA's shared
memory is written only after a cluster barrier has shown that every CTA of the cluster runs, and no shared array
is written by one warp while another may still read it."""
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


def _accesses(statement):
    """(array, index, is_write) of the combine's shared arrays in one statement: what stands left of an assignment,
    or is a destination of `stage`, is written."""
    left, eq, right = statement.partition(" = ")
    found = []
    for part, write in ((left, bool(eq)), (right, False)):
        for m in re.finditer(r"cs\.(\w+)(?:\[([^\]]*)\])?", part):
            found.append((m.group(1), m.group(2), write or part[:m.start()].rstrip().endswith("stage(")))
    return found


def test_window_combine_shared_arrays_between_barriers():
    """Run the source of the combine by statements, its loop over the tail twice, and collect what each stretch
    between two block barriers touches. A thread-private place (the warp's own row) may be written and read in one
    stretch; anything else that is written in a stretch may not be read in it. The barrier at the end of the loop's
    body stands in a condition that holds on every pass but the last."""
    body = kernel_body("decode_window.cu", "window_combine_kernel")
    loop = body.index("for (int t0 = 0;")
    end, depth = body.index("{", loop), 0
    for end in range(end, len(body)):
        depth += {"{": 1, "}": -1}.get(body[end], 0)
        if depth == 0:
            break
    head, step, rest = body[:loop], body[body.index("{", loop) + 1:end], body[end + 1:]
    again = step.index("if (t0 + kTT < vis_max)")
    stretches = [[]]
    for text in (head, step, step[:again], rest):
        for statement in re.split(r"[;{}]", text):
            if "__syncthreads()" in statement:
                stretches.append([])
            else:
                stretches[-1] += _accesses(statement)
    assert sum(len(s) for s in stretches) > 20 and len(stretches) > 7
    for s in stretches:
        for array, index, _ in (a for a in s if a[2]):
            read = [i for x, i, written in s if x == array and i != index and not written]
            assert not read, f"cs.{array}[{index}] is written while cs.{array}{read} may be read"
