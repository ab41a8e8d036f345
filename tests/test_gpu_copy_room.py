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
MID, LARGE = 32, 64


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
        self.table = torch.empty(N, ROW // 8, dtype=torch.int64, device="cuda").random_(generator=g)
        self.load()
        self.R = to_dev(synth.random_bits(LARGE, N, seed=211))
        self.out = dev_out(LARGE, ROW)
        self.expect()
        torch.cuda.synchronize()

    def load(self):
        """The same content again."""
        self.db.load_async(self.table)

    def expect(self):
        """Replies of the table as it now is, by the register-tiled kernel."""
        self.db.set_kernel(2)
        self.db.read_batch_async(self.R, LARGE, self.out)
        self.expected = self.out.clone()
        self.db.set_kernel(0)

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
        assert [t.read(MID) for _ in range(8)] == [2] * 8  # refused: over a quarter of 640 MiB
        assert t.read(LARGE) == 2  # copy and scan
        assert t.read(LARGE) == 1
        assert t.read(MID) == 1
    finally:
        del x
        torch.cuda.empty_cache()
        t.db.close()
    assert talekpir.device_status() == talekpir.OK


def test_a_tuned_tensor_kernel_without_room_for_its_copy(tmp_path):
    """Reads, many-table calls and captured graphs run on the register-tiled kernel,
    and the refused copy is not asked for by each of them."""
    torch = require_cuda()
    t = Table()
    plan = tmp_path / "plan.json"
    plan.write_text('{"plans": [\n' + "".join(
        '{"row_words": %d, "batch_class": %d, "n_class": 10, "kernel": 5, "tensor_mode": 1, '
        '"tensor_kc_rows": 0, "tensor_loads": 0}\n' % (ROW // 4, c) for c in (5, 6)) + "]}\n")
    talekpir.tune_load(str(plan))
    x = fill(torch, 160 << 20)
    try:
        for B in (LARGE, MID):
            job = (t.db, B, t.R, t.out)
            t.out.zero_()
            g = talekpir.MultiGraph([job])
            g.launch()
            torch.cuda.synchronize()
            assert (t.out[:B] == t.expected[:B]).all()
            g.close()
            assert t.read(B) == 2
            t.out.zero_()
            talekpir.read_multi_async([job])
            assert (t.out[:B] == t.expected[:B]).all()
    finally:
        talekpir.tune_clear()
        del x
        torch.cuda.empty_cache()
        t.db.close()
    assert talekpir.device_status() == talekpir.OK


def test_a_tuned_small_batch_has_its_copy_as_a_large_one(tmp_path):
    """A plan that names the tensor-core kernel for a small batch asks for the copy:
    it is made at the first read, and kept at a load."""
    torch = require_cuda()
    t = Table()
    plan = tmp_path / "plan.json"
    plan.write_text('{"plans": [\n{"row_words": %d, "batch_class": 5, "n_class": 10, "kernel": 5, '
                    '"tensor_mode": 1, "tensor_kc_rows": 0, "tensor_loads": 0}\n]}\n' % (ROW // 4))
    talekpir.tune_load(str(plan))
    x = fill(torch, 640 << 20)
    try:
        assert [t.read(MID) for _ in range(2)] == [2, 1]  # copy and scan, scan
        t.load()
        assert t.read(MID) == 1
    finally:
        talekpir.tune_clear()
        del x
        torch.cuda.empty_cache()
        t.db.close()
    assert talekpir.device_status() == talekpir.OK


def test_a_copy_there_was_no_room_for_is_asked_for_again():
    """Once memory has been given back, a table whose copy was refused gets it, by
    single reads as by many-table calls, without a load in between."""
    torch = require_cuda()
    t = Table()
    x = fill(torch, 160 << 20)
    try:
        assert [t.read(LARGE) for _ in range(3)] == [2] * 3
        del x
        torch.cuda.empty_cache()
        for i in range(300):
            if i % 2:
                t.db.read_batch_async(t.R, LARGE, t.out)
            else:
                talekpir.read_multi_async([(t.db, LARGE, t.R, t.out)])
        assert t.read(LARGE) == 1
    finally:
        t.db.close()
    assert talekpir.device_status() == talekpir.OK
