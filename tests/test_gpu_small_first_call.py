"""The device is asked once whether it takes the one-cluster iterations of small clouds, at the first call that wants
them: also where that call is being captured into a caller's CUDA graph, and from several threads at once."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
COMMON = """
import threading
import torch
from paper_2512_04996_gb300 import synth, vicp
p = synth.sphere_plane(seed=3, n=3000)
s, t = torch.from_numpy(p.source).cuda(), torch.from_numpy(p.target).cuda()

def tracker(stream=None):
    c = vicp.Context(grid_divisions=64, dilation_layers=10, flags=vicp.VICP_FLAG_KEEP_GRID, stream=stream)
    c.build_grid(t)
    c.dilate()
    assert c.sync() == 0
    return c, torch.eye(4, dtype=torch.float64, device="cuda")
"""
CAPTURED = COMMON + """
st = torch.cuda.Stream()
st.wait_stream(torch.cuda.current_stream())
with torch.cuda.stream(st):
    c, pose = tracker()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        c.step(s, pose)
    pose.copy_(torch.eye(4))
    g.replay()
    g.replay()
torch.cuda.synchronize()
ref, eager = tracker()
ref.step(s, eager)
ref.step(s, eager)
assert ref.sync() == 0
assert torch.equal(pose, eager)
"""
CAPTURED_IN_A_LOOP = COMMON + """
st = torch.cuda.Stream()
st.wait_stream(torch.cuda.current_stream())
with torch.cuda.stream(st):
    c, pose = tracker()
    c.step(s, pose)
    c.build_grid(t)   # (a step would now take the separate kernels, whose buffers do not exist yet)
    c.dilate()
    assert c.sync() == 0
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        c.step(s, pose)
    g.replay()
torch.cuda.synchronize()
ref, eager = tracker()
ref.step(s, eager)
ref.step(s, eager)
assert ref.sync() == 0
assert torch.equal(pose, eager)
"""
THREADS = COMMON + """
out = [None] * 4

def work(k):
    with torch.cuda.stream(torch.cuda.Stream()):
        c, pose = tracker()
        c.step(s, pose)
        assert c.sync() == 0
        out[k] = pose.cpu()

torch.cuda.synchronize()
threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
for x in threads:
    x.start()
for x in threads:
    x.join()
assert all(x is not None and torch.equal(x, out[0]) for x in out)
"""


@pytest.mark.parametrize("code", [CAPTURED, CAPTURED_IN_A_LOOP, THREADS], ids=["captured", "loop", "threads"])
def test_first_small_step_of_a_process(code):
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
