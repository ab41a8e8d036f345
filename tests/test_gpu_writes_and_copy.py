"""GPU parity of the transposed copy after batches of writes: few slots, more slots
than are listed one by one in few blocks, more blocks than are listed."""

import numpy as np
import pytest

import oracle
from gpu_helpers import dev_out, require_cuda, to_dev, to_host
from paper_2001_08250_gb300 import synth, talekpir

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,z,counts", [
    (200, 4, 16, [1, 30, 200]), (700, 8, 48, [600, 900, 5]), (3000, 1, 144, [300, 700]),
    (64 * 500, 2, 16, [400, 2000, 3]),
])
def test_tensor_reads_after_batches_of_writes(n, d, z, counts):
    require_cuda()
    B, row = 60, d * z
    R = synth.random_bits(B, n, seed=191, table=n)
    dR = to_dev(R)
    with talekpir.DB(n, d, z) as db:
        db.set_kernel(5)
        db.read_batch_async(dR, B, dev_out(B, row))
        oc = oracle.Cuckoo(n, d, z, 0, 500, seed=3)
        db.set_policy(0, 500, 3)
        for i, count in enumerate(counts):
            keys = synth.write_keys(count, seed=192 + i)
            b1, b2 = synth.bucket_pairs(keys, n)
            M = synth.messages(count, z, seed=192 + i)
            status, _ = db.write_batch(b1, b2, M)
            for j in range(count):
                rc, _ = oc.insert(int(b1[j]), int(b2[j]), M[j])
                assert rc == status[j]
            out = dev_out(B, row)
            db.read_batch_async(dR, B, out)
            db.sync()
            T = oc.table()
            assert np.array_equal(db.dump(), T.reshape(n, row))
            assert np.array_equal(to_host(out), oracle.read_batch(T, n, d, z, R)), i
    assert talekpir.device_status() == talekpir.OK


@pytest.mark.parametrize("n,d,z,counts", [
    (40, 2, 65536, [1, 20, 60]), (6, 4, 1 << 20, [1, 15]), (12, 2, 20496, [1, 14, 12]), (30, 3, 16400, [50, 40]),
    (9, 1, (1 << 24) + 16, [3, 4]),
])
def test_batches_of_writes_of_large_slots(n, d, z, counts):
    """Slots of one CTA, of several, and of more than the widest grid (16 MiB), whose
    last threads have less to do; tables that fill up, so that slots move."""
    require_cuda()
    with talekpir.DB(n, d, z) as db:
        db.set_policy(n * d, 500, 3)
        oc = oracle.Cuckoo(n, d, z, n * d, 500, seed=3)
        for i, count in enumerate(counts):
            keys = synth.write_keys(count, seed=202 + i)
            b1, b2 = synth.bucket_pairs(keys, n)
            M = synth.messages(count, z, seed=202 + i)
            status, _ = db.write_batch(b1, b2, M)
            for j in range(count):
                rc, _ = oc.insert(int(b1[j]), int(b2[j]), M[j])
                assert rc == status[j]
            db.sync()
            assert np.array_equal(db.dump(), oc.table().reshape(n, d * z)), i
    assert talekpir.device_status() == talekpir.OK
