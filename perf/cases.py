"""What the speed of this framework is measured on: the server-side work that a
Talek server has it do, each case one call sequence of the public entry points.

Kinds of case (the sizes are those of the benchmark, the tests and the paper's
tables, and odd ones of the same ranges):

  read      one batch of PIR reads of one table, device buffers (masked: the
            replies of serialized PIR)
  many      one call for several tables of uneven sizes and batches
  host      many reads from pinned host buffers to pinned host buffers, in
            batches whose copies overlap the scans
  refresh   a snapshot of the table, a batch of cuckoo writes and a batch of
            reads that sees both
  serve     a burst of reads through the serve loop over several tables
  updates   the compressed interest vector that clients poll

Table payloads are uniform random bytes (ciphertexts), request bits are
Bernoulli(1/2), as a server sees them.
"""

import math

import numpy as np
import torch

from paper_2001_08250_gb300 import synth, talekpir


def listed():
    return [
        # one client's three share rows on the plain-PIR table (4 MiB): the smallest call
        {"name": "read_share", "kind": "read", "n": 1024, "d": 4, "msg": 1024, "B": 3, "masked": False},
        # one read of the paper-scale table (128 MiB): a lone request, no batching
        {"name": "read_one", "kind": "read", "n": 32768, "d": 4, "msg": 1024, "B": 1, "masked": False},
        # the same table under light load: the requests of one short batching window
        {"name": "read_32", "kind": "read", "n": 32768, "d": 4, "msg": 1024, "B": 32, "masked": False},
        # serialized PIR on an odd table of 4.16 KB replies (1 KiB messages with their
        # AEAD overhead): a ragged batch with one-time masks
        {"name": "read_100_masked", "kind": "read", "n": 50021, "d": 4, "msg": 1040, "B": 100, "masked": True},
        # the headline: full batches on the paper-scale table
        {"name": "read_256", "kind": "read", "n": 32768, "d": 4, "msg": 1024, "B": 256, "masked": False},
        # the largest table of the benchmark (4 GiB) with its batch
        {"name": "read_1024_large", "kind": "read", "n": 1 << 20, "d": 4, "msg": 1024, "B": 1024, "masked": False},
        # short messages: many buckets of 128 bytes
        {"name": "read_64_narrow", "kind": "read", "n": 200003, "d": 2, "msg": 64, "B": 64, "masked": False},
        # uneven batching: one call over tables of 2^10 .. 2^17 buckets, 16 .. 512 reads each
        {"name": "many_tables", "kind": "many", "tables": 16, "shapes": 3},
        # end to end through host memory: 4096 reads of the paper-scale table
        {"name": "host_4096", "kind": "host", "n": 32768, "d": 4, "msg": 1024, "B": 4096, "batch": 256},
        # the snapshot cycle of a server: load, 256 writes, a batch of reads
        {"name": "refresh_128", "kind": "refresh", "n": 32768, "d": 4, "msg": 1024, "writes": 256, "B": 128},
        # a burst of 512 reads spread over four tables of the serve loop
        {"name": "serve_burst", "kind": "serve", "n": 32768, "d": 4, "msg": 1024, "tables": 4, "B": 512},
        # GetUpdates: a 2^24-bit interest vector, a fifth of its bits set
        {"name": "updates_16m", "kind": "updates", "m": 1 << 24, "density": 0.2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, most):
    """An odd table shape of at most `most` bytes."""
    d = rng.choice((1, 2, 4, 4, 8))
    msg = rng.choice((64, 256, 528, 1024, 1024, 1040, 4096))
    n = _log(rng, 1000, min(1 << 18, most // (d * msg)))
    return {"n": n, "d": d, "msg": msg}


def draw(rng):
    kind = rng.choice(("read", "read", "read", "read", "many", "host", "refresh", "serve", "updates"))
    if kind == "read":
        return {"kind": kind, **_shape(rng, 1 << 30), "B": _log(rng, 1, 1024), "masked": rng.random() < 0.25}
    if kind == "many":
        return {"kind": kind, "tables": rng.randint(2, 24), "shapes": rng.randint(4, 1 << 20)}
    if kind == "host":
        return {"kind": kind, **_shape(rng, 1 << 28), "B": _log(rng, 256, 8192), "batch": rng.choice((32, 64, 128, 256, 512))}
    if kind == "refresh":
        return {"kind": kind, **_shape(rng, 1 << 28), "writes": _log(rng, 1, 300), "B": _log(rng, 1, 512)}
    if kind == "serve":
        return {"kind": kind, **_shape(rng, 1 << 28), "tables": rng.randint(1, 6), "B": _log(rng, 32, 1024)}
    return {"kind": kind, "m": _log(rng, 1 << 14, 1 << 26), "density": rng.uniform(0.01, 0.4)}


# ---------------------------------------------------------------- inputs

def _bytes(g, *shape):
    """Uniform random bytes of this shape (the last dimension a multiple of 8)."""
    t = torch.empty(*shape[:-1], shape[-1] // 4, dtype=torch.int32, device="cuda")
    t.random_(-(1 << 31), 1 << 31, generator=g)
    return t.view(torch.uint8)


def _requests(g, B, n):
    """B request rows of ceil(n/64) 64-bit words; the bits past n are random too."""
    return _bytes(g, B, 8 * synth.words_per_row(n)).view(torch.int64)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _shapes(case):
    """(n, d, msg, B) of each table of a case."""
    if case["kind"] == "many":
        return synth.multi_table_shapes(case["tables"], case["shapes"])
    tables = case.get("tables", 1)
    share = [case["B"] // tables + (i < case["B"] % tables) for i in range(tables)]
    return [(case["n"], case["d"], case["msg"], b) for b in share]


def _inputs(case, seed):
    """What the case's calls take, on the device: tables, request rows, seeds, writes."""
    g = _gen(seed)
    if case["kind"] == "updates":
        words = (case["m"] + 63) // 64
        bits = torch.rand(words, 64, device="cuda", generator=g) < case["density"]
        bits.view(-1)[case["m"]:] = False
        weight = torch.ones(64, dtype=torch.int64, device="cuda") << torch.arange(64, device="cuda")
        return {"vector": (bits.to(torch.int64) * weight).sum(1)}
    s = {"tables": [_bytes(g, n, d * msg) for n, d, msg, _ in _shapes(case)],
         "requests": [_requests(g, b, n) for n, _, _, b in _shapes(case)]}
    if case.get("masked"):
        s["seeds"] = _bytes(g, case["B"], 32)
    if case["kind"] == "refresh":
        keys = synth.write_keys(case["writes"], seed)
        s["b1"], s["b2"] = synth.bucket_pairs(keys, case["n"])
        s["messages"] = synth.messages(case["writes"], case["msg"], seed)
    return s


class _Table:
    """A table's device memory as an array that torch can wrap; it keeps the table."""

    def __init__(self, db):
        self.db = db
        ptr, shape = db.table_ptr, (db.n, db.row_bytes)
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "|u1", "data": (ptr, False), "version": 2}


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind == "updates":
        words = s["vector"].numel()
        s["out"] = torch.zeros(16 * words + 64, dtype=torch.uint8, device="cuda")
        s["result"] = torch.zeros(3, dtype=torch.int64, device="cuda")
        return s
    if kind == "serve":
        s["server"] = talekpir.Server()
        s["dbs"] = []
        for n, d, msg, _ in _shapes(case):
            s["dbs"].append(s["server"].table(s["server"].add_table(n, d, msg)))
        s["requests"] = [r.cpu().numpy().view(np.uint64) for r in s["requests"]]
        s["out"] = [np.empty((b, d * msg), dtype=np.uint8) for _, d, msg, b in _shapes(case)]
        # clients' reads arrive interleaved over the tables
        s["order"] = sorted((i, t) for t, r in enumerate(s["requests"]) for i in range(len(r)))
    else:
        s["dbs"] = [talekpir.DB(n, d, msg) for n, d, msg, _ in _shapes(case)]
    for db, t in zip(s["dbs"], s["tables"]):
        db.load_async(t)
    torch.cuda.synchronize()
    if kind == "refresh":
        s["table"] = torch.as_tensor(_Table(s["dbs"][0]), device="cuda")
    else:
        del s["tables"]  # the library holds its own copy
    if kind == "host":
        rows = s["requests"][0]
        s["pinned"] = torch.empty(rows.shape, dtype=torch.int64, pin_memory=True).copy_(rows)
        s["replies"] = torch.empty((case["B"], case["d"] * case["msg"]), dtype=torch.uint8, pin_memory=True)
        s["requests"] = s["pinned"].numpy().view(np.uint64)
        s["out"] = s["replies"].numpy()
    elif kind != "serve":
        s["out"] = [torch.empty(b, d * msg, dtype=torch.uint8, device="cuda") for _, d, msg, b in _shapes(case)]
    if kind == "many":
        s["jobs"] = [(db, r.shape[0], r, o) for db, r, o in zip(s["dbs"], s["requests"], s["out"])]
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "read":
        db, rows, out = s["dbs"][0], s["requests"][0], s["out"][0]
        if case["masked"]:
            db.read_batch_masked_async(rows, case["B"], s["seeds"], out)
        else:
            db.read_batch_async(rows, case["B"], out)
        return out
    if kind == "many":
        talekpir.read_multi_async(s["jobs"])
        return s["out"]
    if kind == "host":
        return s["dbs"][0].read_batch_pipelined(s["requests"], case["batch"], s["out"])
    if kind == "refresh":
        db = s["dbs"][0]
        db.load_async(s["tables"][0])
        db.sync()  # the snapshot is in place before the first write to it
        status, evictions = db.write_batch(s["b1"], s["b2"], s["messages"])
        db.read_batch_async(s["requests"][0], case["B"], s["out"][0])
        return {"status": status, "evictions": evictions, "table": s["table"], "replies": s["out"][0]}
    if kind == "serve":
        server, rows, out = s["server"], s["requests"], s["out"]
        for i, t in s["order"]:
            server.submit_read(t, rows[t][i], out[t][i], i)
        server.drain()
        done = server.poll(len(s["order"]))
        return {"done": sum(1 for c in done if c.status == talekpir.OK), "replies": out}
    talekpir.rice_encode_async(s["vector"], case["m"], s["out"], s["out"].numel(), s["result"])
    return {"result": s["result"], "stream": s["out"]}


def work(case):
    """Bytes: each table, request row, seed and reply once.  Flops: one AND and
    one XOR per request and table bit."""
    if case["kind"] == "updates":
        # the vector in, its Golomb-Rice code out (about its entropy)
        p = case["density"]
        h = -p * math.log2(p) - (1 - p) * math.log2(1 - p)
        return {"bytes": case["m"] / 8 * (1 + h), "flops": 0}
    b = f = 0
    for n, d, msg, B in _shapes(case):
        b += n * d * msg + B * (8 * synth.words_per_row(n) + d * msg + (32 if case.get("masked") else 0))
        f += 2.0 * B * n * d * msg * 8
    if case["kind"] == "refresh":  # the snapshot is read and written, the moved slots written
        b += case["n"] * case["d"] * case["msg"] + case["writes"] * case["msg"]
    return {"bytes": float(b), "flops": f}


# ---------------------------------------------------------------- the results in plain torch

def _answers(table, rows):
    """XOR of the selected buckets for each request row, by halving folds of 64-bit words."""
    n = table.shape[0]
    words = table.view(torch.int64)
    out = torch.empty(rows.shape[0], words.shape[1], dtype=torch.int64, device="cuda")
    at = torch.arange(n, device="cuda")
    for i in range(rows.shape[0]):
        picked = words * ((rows[i][at >> 6] >> (at & 63)) & 1)[:, None]
        while picked.shape[0] > 1:
            half = picked.shape[0] // 2
            rest = picked[2 * half:]
            picked = torch.cat((picked[:half] ^ picked[half:2 * half], rest)) if len(rest) else picked[:half] ^ picked[half:]
        out[i] = picked[0]
    return out.view(torch.uint8)


def _masks(seeds, nbytes):
    """ChaCha20 keystreams (RFC 8439) of each seed as the key: zero nonce, blocks from 0."""
    low = 0xFFFFFFFF
    key = seeds.view(torch.int32).to(torch.int64) & low
    blocks = (nbytes + 63) // 64
    start = torch.zeros(seeds.shape[0], blocks, 16, dtype=torch.int64, device="cuda")
    start[..., :4] = torch.tensor([0x61707865, 0x3320646E, 0x79622D32, 0x6B206574], device="cuda")
    start[..., 4:12] = key[:, None]
    start[..., 12] = torch.arange(blocks, device="cuda")
    x = [start[..., i] for i in range(16)]

    def quarter(a, b, c, d):
        for p, q, r, turn in ((a, b, d, 16), (c, d, b, 12), (a, b, d, 8), (c, d, b, 7)):
            x[p] = (x[p] + x[q]) & low
            x[r] = x[r] ^ x[p]
            x[r] = ((x[r] << turn) | (x[r] >> (32 - turn))) & low

    for _ in range(10):
        for i in range(4):
            quarter(i, 4 + i, 8 + i, 12 + i)
        for i in range(4):
            quarter(i, 4 + (i + 1) % 4, 8 + (i + 2) % 4, 12 + (i + 3) % 4)
    words = (torch.stack(x, -1) + start) & low
    stream = torch.stack([(words >> (8 * i)) & 255 for i in range(4)], -1).to(torch.uint8)
    return stream.view(seeds.shape[0], -1)[:, :nbytes]


def exact(case, seed):
    if case["kind"] == "updates":
        return None  # a stream of whole bytes, equal or wrong
    cost = sum(B * n * d * msg for n, d, msg, B in _shapes(case))
    if cost > 1 << 41:
        return None
    s = _inputs(case, seed)
    if case["kind"] == "refresh":
        table = s["tables"][0]
        slots = table.view(case["n"], case["d"], case["msg"])
        used = {}
        for b1, b2, m in zip(s["b1"].tolist(), s["b2"].tolist(), s["messages"]):
            bucket = b1 if used.get(b1, 0) < case["d"] else b2
            at = used.get(bucket, 0)
            if at >= case["d"]:
                return None  # both buckets full: an eviction walk
            used[bucket] = at + 1
            slots[bucket, at] = torch.from_numpy(m).cuda()
        zeros = np.zeros(case["writes"], dtype=np.int32)
        return {"status": zeros, "evictions": zeros.astype(np.uint32), "table": table,
                "replies": _answers(table, s["requests"][0])}
    got = [_answers(t, r) for t, r in zip(s["tables"], s["requests"])]
    if case["kind"] == "serve":
        return {"done": case["B"], "replies": got}
    if case["kind"] == "many":
        return got
    if case.get("masked"):
        got[0] ^= _masks(s["seeds"], got[0].shape[1])
    return got[0]
