"""Thread-block clusters: a block's shared memory may be accessed by another block only
once that block has started.  Every kernel of the library that maps remote shared memory
has a cluster-wide barrier (a sync, or the wait of an arrival at its entry) before the
first such access.  Read from the source: the faulty order is undefined on a GPU."""
import os
import re

import pytest

from paper_2208_12737_gb300 import build


def _cluster_kernels():
    out = []
    for path in build.sources():
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__cluster_dims__", text):
            i = text.index("{", text.index(")", text.index("kernel(", m.end())))
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[j], 0)
                j += 1
            name = re.search(r"(\w+kernel)\(", text[m.end():i]).group(1)
            out.append(pytest.param(text[i:j], id=f"{os.path.basename(path)}:{name}"))
    return out


@pytest.mark.parametrize("body", _cluster_kernels())
def test_barrier_before_the_first_remote_access(body):
    remote = body.find("map_shared_rank")
    waits = [body.find(x) for x in ("cluster.sync()", "cluster.barrier_wait()") if x in body]
    assert remote < 0 or (waits and min(waits) < remote)


def test_the_cluster_kernels_are_found():
    assert len(_cluster_kernels()) >= 2
