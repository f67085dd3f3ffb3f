"""Source check of the rule for distributed shared memory: a block may touch
another block's shared memory only once all blocks of the cluster have
started.  Every kernel that maps another block's shared memory therefore
passes a cluster barrier (cl.sync(), or cl.barrier_arrive() and
cl.barrier_wait()) before the first mapping, which no thread can return in
front of once it has arrived, and one more after the last access."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2010_12879_gb300", "csrc")


def _kernels():
    """(name, body) of every kernel, comments left out."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\([^{]*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield m.group(1), text[m.end():i]


def test_cluster_blocks_have_started_before_remote_shared_memory():
    mapped = [(n, b) for n, b in _kernels() if "map_shared_rank" in b]
    assert mapped
    for name, body in mapped:
        before, after = body.split("map_shared_rank", 1)
        if "cl.sync();" not in before:
            assert before.count("cl.barrier_arrive();") == 1, name
            assert before.count("cl.barrier_wait();") == 1, name
            arrive, wait = before.index("cl.barrier_arrive();"), before.index("cl.barrier_wait();")
            assert arrive < wait, name
            assert "return" not in before[arrive:], name
        assert "cl.sync();" in after, name


def test_no_cluster_access_outside_kernels():
    uses = sum(re.sub(r"//[^\n]*", "", open(p).read()).count("map_shared_rank")
               for p in glob.glob(os.path.join(CSRC, "*.cu*")))
    assert uses == sum(b.count("map_shared_rank") for _, b in _kernels())
