"""A CTA of a cluster may touch another's shared memory only once that CTA is known to run, which
the programming model guarantees after a cluster barrier alone. An access without one is not an
error that a run shows, so the kernels' source is read instead."""
import glob
import os
import re

from conftest import ROOT


def kernels(text):
    """(name, body) of every __global__ function."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    for m in re.finditer(r"__global__", text):
        start = text.index("{", m.end())
        depth, i = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        names = re.findall(r"(\w+)\s*\(", text[m.end():start])
        yield next(n for n in names if not n.startswith("__")), text[start:i]


def test_remote_shared_memory_follows_a_cluster_barrier():
    remote = []
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_0910_2918_gb300", "csrc", "*.cu*"))):
        for name, body in kernels(open(path).read()):
            at = body.find("map_shared_rank")
            if at < 0:
                continue
            remote.append(name)
            assert re.search(r"cluster\.(barrier_wait\(|sync\(\))", body[:at]), name + " does not wait for its cluster first"
            assert re.search(r"cluster\.sync\(\)", body[at:]), name + " does not wait for the remote writes"
    assert remote == ["k_combine"]
