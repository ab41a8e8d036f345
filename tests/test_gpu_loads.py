"""GPU parity of bulk loads with the transposed copy in place: from device memory
(one pass for both), from device memory that is not 16-byte aligned, from pinned
and from pageable host memory; tables whose rows and buckets do not fill the
copy's tiles."""

import numpy as np
import pytest

import oracle
from gpu_helpers import dev_out, require_cuda, to_dev, to_host
from paper_2001_08250_gb300 import synth, talekpir

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,z", [(1, 1, 16), (63, 1, 16), (65, 1, 48), (130, 2, 64), (257, 1, 144), (1000, 4, 272)])
def test_loads_reach_the_table_and_its_transposed_copy(n, d, z):
    torch = require_cuda()
    B, row = 70, d * z
    R = synth.random_bits(B, n, seed=181, table=n)
    dR = to_dev(R)
    with talekpir.DB(n, d, z) as db:
        db.set_kernel(5)
        db.read_batch_async(dR, B, dev_out(B, row))  # the copy exists from here on
        for i, kind in enumerate(("device", "offset", "pinned", "pageable", "device")):
            T = synth.table_bytes(n, d, z, seed=182 + i, table=n)
            flat = torch.from_numpy(np.ascontiguousarray(T).reshape(-1))
            if kind == "device":
                src = flat.cuda()
            elif kind == "offset":
                src = torch.cat((torch.zeros(4, dtype=torch.uint8), flat)).cuda()[4:]
            else:
                src = flat.pin_memory() if kind == "pinned" else flat
            if kind in ("pinned", "pageable"):
                db.load(src.numpy().reshape(n, row))
            else:
                db.load_async(src)
            out = dev_out(B, row)
            db.read_batch_async(dR, B, out)
            assert np.array_equal(to_host(out), oracle.read_batch(T, n, d, z, R)), kind
            db.sync()
            assert np.array_equal(db.dump(), T.reshape(n, row)), kind
    assert talekpir.device_status() == talekpir.OK
