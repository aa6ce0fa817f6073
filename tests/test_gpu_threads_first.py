"""The first calls of a process, from several host threads at once, each with a handle and a stream of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import threading, torch
import paper_1504_06443_gb300 as gep
gep.load()
torch.cuda.init()
out, start = {}, threading.Barrier(8)
def work(i):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        g = torch.Generator(device="cuda").manual_seed(i % 2)
        M = (300, 650)[i % 2]
        A = torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda")
        A = A + A.t()
        B = torch.eye(M, dtype=torch.float64, device="cuda")
        h = gep.Handle(stream=s)
        s.synchronize()
        start.wait()
        w, Y, info = gep.solve(A, B, precision=("fp64", "fp64_emulated")[i % 2], sep=("1stage", "2stage")[i % 2], handle=h)
        bs = gep.BatchedSolver([A, A[:40, :40].contiguous()], [B, B[:40, :40].contiguous()], nstreams=2)
        bs.run()
        torch.cuda.synchronize()
        out[i] = (info, bs.info(), w.cpu(), bs.results()[0][0].cpu())
t = [threading.Thread(target=work, args=(i,)) for i in range(8)]
[x.start() for x in t]
[x.join() for x in t]
assert len(out) == 8
for i in range(8):
    assert out[i][0] == 0 and out[i][1] == 0
    assert torch.equal(out[i][2], out[i % 2][2]) and torch.equal(out[i][3], out[i % 2][3])
print("ok")
"""


def test_first_calls_from_threads():
    from paper_1504_06443_gb300 import build
    build.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.stdout.strip().endswith("ok"), r.stderr[-2000:]
