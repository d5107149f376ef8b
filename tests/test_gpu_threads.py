"""Handles on several threads, each on a stream of its own and each kernel's first
launch on the device among them: every thread's images are the ones that a
single thread makes afterwards.  (What is set up once per device and kernel is
published after it is complete.)"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import threading
import torch
import synth
import paper_2504_00959_gb300 as rick

def image(n, nw, seed, out, i, gate):
    with torch.cuda.stream(torch.cuda.Stream()):
        prob = synth.disk_problem(n, nw, 3000, synth.KERNEL_KB, 7, 3.0, 60.0, seed, fill=0.4)
        g = {k: prob[k].cuda() for k in ("vis", "u", "v", "w", "wt")}
        im = rick.Imager(dict(prob["params"], flags=synth.FLAG_REAL))
        gate.wait()
        im.grid(g["vis"], g["u"], g["v"], g["w"], g["wt"])
        img = im.image()
        grad = im.degrid(img, g["u"], g["v"], g["w"], g["wt"])
        torch.cuda.current_stream().synchronize()
        im.stats()
        out[i] = (img, grad)
        im.close()

torch.zeros(1, device="cuda")
jobs = [(n, nw, s) for s in (1, 2) for n, nw in ((1024, 12), (2048, 4), (4096, 2), (8192, 1))]
both = []
for together in (True, False):
    out = [None] * len(jobs)
    gate = threading.Barrier(len(jobs) if together else 1, timeout=60)
    threads = [threading.Thread(target=image, args=(*j, out, i, gate)) for i, j in enumerate(jobs)]
    for t in threads:
        t.start()
        if not together:
            t.join()
    for t in threads:
        t.join()
    both.append(out)
for a, b in zip(*both):
    for x, y in zip(a, b):
        assert (x - y).abs().max().item() <= 1e-5 * y.abs().max().item()
print("ok")
"""


def test_first_launches_on_several_threads():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_00959_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
