"""The kernel by which the serve loop reads a batch: forced and tuned choices hold,
and a copy that could not be made takes nothing of the budget."""

import numpy as np
import pytest

import oracle
from gpu_helpers import require_cuda
from paper_2001_08250_gb300 import synth, talekpir

pytestmark = pytest.mark.gpu

N, D, Z, B = 3000, 4, 256, 32


def burst(server, tid, R, out):
    """All rows of R in one unit (within one batching window)."""
    for i in range(len(R)):
        server.submit_read(tid, R[i], out[i], i)
    server.drain()
    done = server.poll(len(R))
    assert len(done) == len(R) and all(c.status == talekpir.OK for c in done)


@pytest.mark.parametrize("kernel,tuned", [(1, False), (3, False), (4, False), (5, False), (4, True), (5, True)])
def test_small_batches_run_on_the_forced_or_tuned_kernel(kernel, tuned, tmp_path):
    require_cuda()
    T = synth.table_bytes(N, D, Z, seed=220, table=0)
    R = synth.random_bits(B, N, seed=221)
    exp = oracle.read_batch(T, N, D, Z, R)
    server = talekpir.Server(tick_us=200000)
    try:
        tid = server.add_table(N, D, Z)
        db = server.table(tid)
        db.load(T)
        if tuned:
            plan = tmp_path / "plan.json"
            plan.write_text('{"plans": [\n' + "".join(
                '{"row_words": %d, "batch_class": %d, "n_class": 12, "kernel": %d, "tensor_mode": 0, '
                '"tensor_kc_rows": 0, "tensor_loads": 0}\n' % (D * Z // 4, c, kernel) for c in range(7)) + "]}\n")
            talekpir.tune_load(str(plan))
        else:
            db.set_kernel(kernel)
        out = np.empty((B, D * Z), dtype=np.uint8)
        burst(server, tid, R, out)
        assert np.array_equal(out, exp)
        by_kernel = list(server.stats().kernel_launches)
        assert by_kernel[kernel] == sum(by_kernel) > 0
    finally:
        talekpir.tune_clear()
        server.close()


def test_a_copy_that_was_not_made_takes_nothing_of_the_budget():
    """Large batches whose copy the device has no room for, after each of several
    loads; then a table that the budget holds only without those copies."""
    torch = require_cuda()
    n, z, reads = 1000, 65536, 64  # a table of 250 MiB, a copy of 256 MiB
    server = talekpir.Server(hbm_budget_bytes=(256 + 250 + 256 + 60) << 20, max_inflight=1, tick_us=200000)
    try:
        tid = server.add_table(n, D, z)
        db = server.table(tid)
        g = torch.Generator(device="cuda")
        g.manual_seed(230)
        t = torch.empty(n, D * z // 8, dtype=torch.int64, device="cuda").random_(generator=g)
        R = synth.random_bits(reads, n, seed=231)
        out = np.empty((reads, D * z), dtype=np.uint8)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        x = torch.empty(torch.cuda.mem_get_info()[0] - (192 << 20), dtype=torch.uint8, device="cuda")
        for _ in range(3):
            db.load_async(t)
            db.sync()
            burst(server, tid, R, out)
        assert server.stats().kernel_launches[2] == 3
        del x
        torch.cuda.empty_cache()
        server.add_table(1000, 4, 100 * 256)  # 98 MiB
    finally:
        server.close()
