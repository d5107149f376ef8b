"""Distributed shared memory in the kernels' sources: a CTA's shared memory may
be read or written by another CTA of its cluster only once a cluster barrier
has shown that it runs, so every kernel's first remote access stands after a
wait on that barrier.  (On a device a missing barrier shows only by chance.)
And a kernel that is handed one array as two pointers declares neither of them
free of aliases."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
REMOTE = re.compile(r"\b(?:ld|st|atom|red)(?:\.\w+)*\.shared::cluster|\bld_cluster_\w+\(")
WAIT = re.compile(r"barrier\.cluster\.wait|\bcluster_sync\(\)")


def _kernels():
    """(file:kernel, signature, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2504_00959_gb300", "csrc", "*.cu"))):
        src = re.sub(r"/\*.*?\*/|//[^\n]*", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"__global__", src):
            start = src.index("{", m.end())
            depth, i = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            sig = src[m.end():start]
            name = [w for w in re.findall(r"\b(k_\w+)", sig)]
            if name:
                yield f"{os.path.basename(path)}:{name[0]}", sig, src[start:i]


def test_remote_shared_memory_after_a_cluster_barrier():
    remote = {name: body for name, _, body in _kernels() if REMOTE.search(body)}
    assert {"rick_prep.cu:k_scan_one", "rick_grid.cu:k_grid_heavy"} <= set(remote)
    for name, body in remote.items():
        wait = WAIT.search(body)
        assert wait and wait.start() < REMOTE.search(body).start(), name


def test_scan_in_place_declares_no_restrict():
    sig = {name: sig for name, sig, _ in _kernels()}["rick_prep.cu:k_scan_one"]
    args = {a.split()[-1].lstrip("*"): a for a in sig[sig.index("k_scan_one") + 11:].rstrip().rstrip(")").split(",")}
    assert "__restrict__" not in args["in"] and "__restrict__" not in args["cursor"]
