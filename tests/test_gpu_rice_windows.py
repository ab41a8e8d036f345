"""GPU parity of the compressed encoding where its blocks change form: codes put
together in shared memory, blocks too long for it, gaps over several blocks,
and calls on two streams at once."""

import numpy as np
import pytest

import oracle
from gpu_helpers import require_cuda
from paper_2001_08250_gb300 import synth, talekpir

pytestmark = pytest.mark.gpu

BLOCK = 65536  # bits of a block of 1024 words


def _bits(m, positions):
    v = np.zeros((m + 63) // 64, dtype=np.uint64)
    np.bitwise_or.at(v, np.asarray(positions) // 64, np.uint64(1) << (np.asarray(positions) % 64).astype(np.uint64))
    return v


def _random(m, density, seed):
    u = synth.uniform01(m, synth.stream_key(seed, 1, 78))
    return _bits(m, np.nonzero(u < density)[0])


CASES = [
    ("dense, long codes: past the window", _random(2 * BLOCK, 0.3, 1), 2 * BLOCK, 12),
    ("64-bit codes", _random(BLOCK, 0.02, 2), BLOCK, 63),
    ("long runs of ones", _random(3 * BLOCK + 17, 0.0005, 3), 3 * BLOCK + 17, 0),
    ("a gap over empty blocks", _bits(9 * BLOCK, [0, 5, 8 * BLOCK + 3, 8 * BLOCK + 4]), 9 * BLOCK, 3),
    ("one bit at the end", _bits(5 * BLOCK, [5 * BLOCK - 1]), 5 * BLOCK, 0),
    ("block edges", _bits(4 * BLOCK, [BLOCK - 1, BLOCK, 2 * BLOCK - 1, 3 * BLOCK]), 4 * BLOCK, -1),
    ("all ones", np.full(2048, 0xFFFFFFFFFFFFFFFF, dtype=np.uint64), 2 * BLOCK, -1),
]


@pytest.mark.parametrize("v,m,k", [c[1:] for c in CASES], ids=[c[0] for c in CASES])
def test_encoding_of_each_block_form(v, m, k):
    torch = require_cuda()
    exp, enb, ecnt, ek = oracle.rice_encode(v, m, None if k < 0 else k)
    cap = (len(exp) + 3) // 4 * 4 + 64
    dv = torch.from_numpy(v.view(np.int64)).cuda()
    outs, ress, streams = [], [], [torch.cuda.Stream() for _ in range(2)]
    for s in streams:
        with torch.cuda.stream(s):
            outs.append(torch.full((cap,), 0xA5, dtype=torch.uint8, device="cuda"))
            ress.append(torch.full((3,), -1, dtype=torch.int64, device="cuda"))
    for _ in range(3):
        for s, o, r in zip(streams, outs, ress):
            s.wait_stream(torch.cuda.default_stream())
            talekpir.rice_encode_async(dv, m, o, cap, r, k, s)
    torch.cuda.synchronize()
    for o, r in zip(outs, ress):
        assert [int(x) & (2**64 - 1) for x in r.cpu()] == [enb, ecnt, ek]
        got = o.cpu().numpy()
        assert np.array_equal(got[:len(exp)], exp)
        assert not got[len(exp):].any()
