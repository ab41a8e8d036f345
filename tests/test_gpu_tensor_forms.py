"""GPU parity of the tensor-core read with the table operand in tensor memory:
its block, chunk, tile and stage edges, and the batch sizes whose route
changes once a table has its transposed copy."""

import numpy as np
import pytest

import oracle
from gpu_helpers import dev_out, require_cuda, to_dev, to_host
from paper_2001_08250_gb300 import synth, talekpir

pytestmark = pytest.mark.gpu

TENSOR = 5

# one column tile and several; buckets around a word (64) and a stage (256);
# request blocks of 16 .. 128 with and without a second, third, ... block;
# k-chunks that end within a stage; more chunks than one
SHAPES = [
    (1, 1, 16, 1), (64, 1, 16, 16), (65, 1, 32, 17), (255, 1, 48, 33), (257, 2, 64, 64),
    (1000, 1, 112, 65), (2817, 1, 128, 128), (2900, 2, 64, 97), (5700, 1, 64, 113),
    (700, 4, 256, 129), (20011, 1, 16, 70), (513, 1, 80, 300), (90001, 1, 32, 20),
]


@pytest.mark.parametrize("n,d,z,B", SHAPES)
def test_tensor_memory_form_bit_exact(n, d, z, B):
    """Plain and masked replies equal the oracle's, from request rows at an
    8-byte offset (which only this form reads) and at a 16-byte one."""
    require_cuda()
    T = synth.table_bytes(n, d, z, seed=160, table=n)
    R = synth.random_bits(B, n, seed=161, table=n)
    S = synth.mask_seeds(B, seed=162, table=n)
    exp = oracle.read_batch(T, n, d, z, R)
    with talekpir.DB(n, d, z) as db:
        db.load(T)
        db.set_kernel(TENSOR)
        for offset in (0, 1):
            flat = to_dev(np.concatenate([np.zeros(offset, np.uint64), R.reshape(-1)]))
            out = dev_out(B, d * z)
            db.read_batch_async(flat[offset:], B, out)
            assert np.array_equal(to_host(out), exp), offset
        assert np.array_equal(db.read_batch_masked(R, S), oracle.read_batch_masked(T, n, d, z, R, S))
    assert talekpir.device_status() == talekpir.OK


@pytest.mark.parametrize("n,d,z,B", [(3000, 4, 256, 5), (3000, 4, 256, 47), (5000, 1, 64, 9),
                                     (5000, 1, 64, 130), (300, 1, 16, 47)])
def test_smaller_batches_before_and_after_the_transposed_copy(n, d, z, B):
    """The first batch of these sizes runs without the transposed copy, the
    second makes it, the third uses it; all equal the oracle's, also after a
    load and after writes, and through many-table calls and a captured graph."""
    torch = require_cuda()
    R = synth.random_bits(B, n, seed=171, table=n)
    dR = to_dev(R)
    keys = synth.write_keys(40, seed=172)
    b1, b2 = synth.bucket_pairs(keys, n)
    M = synth.messages(40, z, seed=172)
    with talekpir.DB(n, d, z) as db:
        for load in range(2):
            T = synth.table_bytes(n, d, z, seed=173 + load, table=n)
            db.load(T)
            exp = oracle.read_batch(T, n, d, z, R)
            for _ in range(3):
                out = dev_out(B, d * z)
                db.read_batch_async(dR, B, out)
                assert np.array_equal(to_host(out), exp)
        status, _ = db.write_batch(b1, b2, M)
        assert (status == 0).all()
        db.sync()
        T = db.dump()
        exp = oracle.read_batch(T.reshape(n, d * z), n, d, z, R)
        out = dev_out(B, d * z)
        db.read_batch_async(dR, B, out)
        assert np.array_equal(to_host(out), exp)
        job = (db, B, dR, dev_out(B, d * z))
        talekpir.read_multi_async([job])
        assert np.array_equal(to_host(job[3]), exp)
        job[3].zero_()
        g = talekpir.MultiGraph([job])
        g.launch()
        torch.cuda.synchronize()
        assert np.array_equal(to_host(job[3]), exp)
        g.close()
    assert talekpir.device_status() == talekpir.OK


@pytest.mark.parametrize("n,d,z,B", [(200003, 1, 16, 1024), (200003, 1, 16, 784), (120001, 3, 16, 784),
                                     (90001, 1, 16, 769)])
def test_items_of_one_tile_one_after_another(n, d, z, B):
    """Narrow rows with many request blocks and k-chunks: a CTA takes several items
    of one column tile (or of three, one stream with a tile more), in which the
    second stream has none; alone and with another table of such items."""
    require_cuda()
    T = synth.table_bytes(n, d, z, seed=180, table=n)
    R = synth.random_bits(B, n, seed=181, table=n)
    exp = oracle.read_batch(T, n, d, z, R)
    n2, B2 = 70001, 900
    T2 = synth.table_bytes(n2, 1, 48, seed=182, table=n2)
    R2 = synth.random_bits(B2, n2, seed=183, table=n2)
    exp2 = oracle.read_batch(T2, n2, 1, 48, R2)
    with talekpir.DB(n, d, z) as db, talekpir.DB(n2, 1, 48) as db2:
        db.load(T)
        db2.load(T2)
        dR, dR2 = to_dev(R), to_dev(R2)
        for x in (db, db2):
            x.set_kernel(TENSOR)
        outs = [dev_out(B, d * z) for _ in range(12)]
        for out in outs:
            db.read_batch_async(dR, B, out)
        for out in outs:
            assert np.array_equal(to_host(out), exp)
        out, out2 = dev_out(B, d * z), dev_out(B2, 48)
        for _ in range(4):
            talekpir.read_multi_async([(db, B, dR, out), (db2, B2, dR2, out2)])
        assert np.array_equal(to_host(out), exp) and np.array_equal(to_host(out2), exp2)
    assert talekpir.device_status() == talekpir.OK


@pytest.mark.parametrize("n,B,count", [(32768, 128, 2), (32768, 112, 2), (32768, 16, 5), (32768, 256, 7), (2048, 64, 1),
                                       (100000, 16, 5), (100000, 8, 5)])
def test_autotune_times_each_schedule_once(n, B, count):
    """The tensor-memory form's k-chunks hold 2 816 buckets at 128 requests a block,
    3 072 at 112, 21 504 at 16: sizes that it would cut to those are not candidates
    (CTA pairs, above 128 requests, hold all)."""
    require_cuda()
    with talekpir.DB(n, 1, 2048) as db:
        try:
            r = db.autotune(B, 1)
            assert r["tensor_candidates"] == count
        finally:
            talekpir.tune_clear()


@pytest.mark.parametrize("kc", [256, 2048, 16384, 32768])
@pytest.mark.parametrize("B", [16, 100, 128, 200])
def test_given_chunks_bit_exact(kc, B, tmp_path):
    """Plans with k-chunks of a given size, also of one that the form cuts."""
    require_cuda()
    n, d, z = 9000, 2, 80
    T = synth.table_bytes(n, d, z, seed=185, table=n)
    R = synth.random_bits(B, n, seed=186, table=n)
    plan = tmp_path / "plan.json"
    plan.write_text('{"plans": [\n{"row_words": %d, "batch_class": %d, "n_class": 14, "kernel": 5, "tensor_mode": 1, '
                    '"tensor_kc_rows": %d, "tensor_loads": 0}\n]}\n' % (d * z // 4, (B - 1).bit_length(), kc))
    talekpir.tune_load(str(plan))
    try:
        with talekpir.DB(n, d, z) as db:
            db.load(T)
            assert np.array_equal(db.read_batch(R), oracle.read_batch(T, n, d, z, R))
    finally:
        talekpir.tune_clear()
    assert talekpir.device_status() == talekpir.OK
