"""Calls that set something up at their first use, made first of all under or beside
the capture of a stream (each in a process of its own)."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEAD = """
import torch
from paper_2001_08250_gb300 import synth, talekpir
g, s, s2 = torch.cuda.CUDAGraph(), torch.cuda.Stream(), torch.cuda.Stream()
rnd = lambda *shape: torch.randint(-2**62, 2**62, shape, dtype=torch.int64, device="cuda")
"""


def run(body):
    r = subprocess.run([sys.executable, "-c", HEAD + body], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr


def test_the_first_rice_encode_of_a_process_is_captured():
    run("""
m = 1 << 20
v, out, res = rnd(m // 64), torch.zeros(8 * m, dtype=torch.uint8, device="cuda"), torch.zeros(3, dtype=torch.int64, device="cuda")
torch.cuda.synchronize()
with torch.cuda.graph(g, stream=s):
    talekpir.rice_encode_async(v, m, out, out.numel(), res, -1, s)
g.replay()
torch.cuda.synchronize()
a = res.clone(), out.clone()
out.fill_(255)
torch.cuda.synchronize()
talekpir.rice_encode_async(v, m, out, out.numel(), res, -1, s)
torch.cuda.synchronize()
assert (a[0] == res).all() and (a[1] == out).all() and res[0] > 0
print("ok")
""")
