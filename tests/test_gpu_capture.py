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


@pytest.mark.parametrize("B,d", [(8, 4), (64, 4), (64, 1)])
def test_reads_that_make_the_transposed_copy_beside_a_capture(B, d):
    """Reads on another stream, among them the one that makes their table's copy (of
    small batches, of large ones, on narrow rows), leave the capture as it is."""
    run(f"""
B, n, z = {B}, 4096, 64
db = talekpir.DB(n, {d}, z * (4 if {d} > 1 else 1))
db.load_async(rnd(n, db.row_bytes // 8))
R, out, x = rnd(B, n // 64), torch.zeros(B, db.row_bytes, dtype=torch.uint8, device="cuda"), torch.zeros(8, device="cuda")
db.set_kernel(2)
db.read_batch_async(R, B, out)
db.set_kernel(0)
torch.cuda.synchronize()
expected = out.clone()
out.zero_()
torch.cuda.synchronize()
counts = []
with torch.cuda.graph(g, stream=s):
    x += 1
    for _ in range(100):
        before = talekpir.kernel_launches()
        db.read_batch_async(R, B, out, s2)
        counts.append(talekpir.kernel_launches() - before)
g.replay()
torch.cuda.synchronize()
assert (out == expected).all() and x[0] == 1
assert set(counts) != {{2}}  # (the register-tiled kernel alone takes two launches each)
print("ok")
""")
