"""Reads where the device has little room for the transposed copy of the tensor-core
read.  The device is filled with one allocation, so that the copy of a 256 MiB
table is refused to smaller batches (more than a quarter of what is free) or to
all.  Routes are told apart by launches: the register-tiled read takes two (replies
zeroed, scan), the tensor-core read of these few buckets one."""

import numpy as np
import pytest

from gpu_helpers import dev_out, require_cuda, to_dev
from paper_2001_08250_gb300 import synth, talekpir

pytestmark = pytest.mark.gpu

N, D, Z = 1000, 4, 65536  # 250 MiB; one k-chunk
ROW = D * Z
MID, LARGE = 16, 64


def fill(torch, leave):
    """All but `leave` bytes of the device's free memory."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    x = torch.empty(free - leave, dtype=torch.uint8, device="cuda")
    left, _ = torch.cuda.mem_get_info()
    assert abs(left - leave) < 64 << 20
    return x


class Table:
    def __init__(self):
        torch = require_cuda()
        self.db = talekpir.DB(N, D, Z)
        g = torch.Generator(device="cuda")
        g.manual_seed(210)
        t = torch.empty(N, ROW // 8, dtype=torch.int64, device="cuda").random_(generator=g)
        self.db.load_async(t)
        self.R = to_dev(synth.random_bits(LARGE, N, seed=211))
        self.out = dev_out(LARGE, ROW)
        self.db.set_kernel(2)
        self.db.read_batch_async(self.R, LARGE, self.out)
        self.expected = self.out.clone()
        self.db.set_kernel(0)
        torch.cuda.synchronize()

    def read(self, B):
        """One read of B requests: its launches (replies checked)."""
        self.out.zero_()
        before = talekpir.kernel_launches()
        self.db.read_batch_async(self.R, B, self.out)
        launches = talekpir.kernel_launches() - before
        assert (self.out[:B] == self.expected[:B]).all()
        return launches


def test_a_refusal_for_small_batches_leaves_large_ones_their_copy():
    torch = require_cuda()
    t = Table()
    x = fill(torch, 640 << 20)
    try:
        assert [t.read(MID) for _ in range(4)] == [2] * 4  # refused: over a quarter of 640 MiB
        assert t.read(LARGE) == 2  # copy and scan
        assert t.read(LARGE) == 1
        assert t.read(MID) == 1
    finally:
        del x
        torch.cuda.empty_cache()
        t.db.close()
    assert talekpir.device_status() == talekpir.OK
