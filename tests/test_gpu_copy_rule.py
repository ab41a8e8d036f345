"""Routes of batches of 32, 47 and 16 requests of a 250 MiB table (estimated savings 61,
181 and 12 us a batch; copy 125 us, its allocation 126), told apart by launches: 2 on
the register-tiled kernel or with the copy's build, 1 with the copy."""

import numpy as np
import pytest

from gpu_helpers import require_cuda
from paper_2001_08250_gb300 import synth, talekpir
from test_gpu_copy_room import LARGE, N, Z, Table

pytestmark = pytest.mark.gpu


@pytest.fixture()
def t():
    require_cuda()
    t = Table()
    yield t
    t.db.close()
    assert talekpir.device_status() == talekpir.OK


def reads(t, B, count):
    return [t.read(B) for _ in range(count)]


def write(t, count, seed):
    """Launches of a batch of writes."""
    b1, b2 = synth.bucket_pairs(synth.write_keys(count, seed=seed), N)
    before = talekpir.kernel_launches()
    status, _ = t.db.write_batch(b1, b2, synth.messages(count, Z, seed=seed))
    assert (status == 0).all()
    launches = talekpir.kernel_launches() - before
    t.db.sync()
    t.expect()
    return launches


@pytest.mark.parametrize("B,before", [(32, 4), (47, 1)])
def test_the_copy_is_made_once_the_batches_pay_for_it(t, B, before):
    assert reads(t, B, before + 3) == [2] * (before + 1) + [1, 1]
    reads(t, B, 20)
    for _ in range(3):  # a cycle of many batches: at its first one
        t.load()
        assert reads(t, B, 12) == [2] + [1] * 11


def test_cycles_of_few_batches_do_not_pay_for_it(t):
    for _ in range(12):
        t.load()
        assert reads(t, 32, 1) == [2]
        assert reads(t, 16, 3) == [2, 2, 2]
    assert reads(t, LARGE, 2) == [2, 1]  # a large batch asks for it
    t.load()
    assert reads(t, 16, 2) == [1, 1]


def test_small_writes_alone_drop_it(t):
    reads(t, 47, 12)
    assert reads(t, 47, 1) == [1]
    assert [write(t, 1, 240 + i) for i in range(24)] == [2] * 20 + [1] * 4
    assert reads(t, 16, 2) == [2, 1]  # (copies have paid so far: made again, on a guess)
    assert reads(t, 47, 2) == [1, 1]
    assert write(t, 200, 270) == 1  # more slots than are followed: as a load
    assert reads(t, 47, 2) == [2, 1]


def test_replays_of_a_captured_small_batch_follow_the_table(t):
    torch = require_cuda()
    reads(t, 47, 3)
    g = talekpir.MultiGraph([(t.db, 47, t.R, t.out)])

    def replay():
        t.expect()
        t.out.zero_()
        g.launch()
        torch.cuda.synchronize()
        return bool((t.out[:47] == t.expected[:47]).all())

    try:
        assert replay()
        t.table.bitwise_not_()
        t.load()
        assert replay()
        assert write(t, 40, 280) > 1
        assert replay()
        assert write(t, 1, 281) > 1
        assert replay()
    finally:
        g.close()
