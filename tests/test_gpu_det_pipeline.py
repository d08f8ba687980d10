"""The deterministic key-value pipeline at the edges of its parts, against the oracle's serial run in
transaction-id order: the sort's two tile sizes, the fold's tiles and chunks, slots whose accesses run
through several of them, the lane-group widths of the validation pass, invalid transactions over several
tiles of ranks, and op ranges that leave ops out.  Every value is a whole number and must match exactly."""
import numpy as np
import pytest

import oracle
from paper_2406_10158_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_10158_gb300 import engine
    return engine


def run(eng, table, batch, fb, max_ops, times=1):
    nf, nrec = table.shape[:2]
    with eng.Database("kv", n_records=nrec, n_fields=nf, field_bytes=fb, max_ops_per_txn=max_ops,
                      max_batch_txns=batch.n_txns, max_batch_ops=batch.n_ops) as db:
        db.load_kv(table)
        for _ in range(times):
            out = db.run("det", batch)
        return out, db.read_kv()


def make(nrec, nf, fb, **kw):
    table = wl.kv_table_bytes(3, nrec, nf) if fb == 16 else wl.kv_table_splitmix(3, nrec, nf)
    return table, wl.kv_batch(7, nrec=nrec, nfields=nf, field_bytes=fb, **kw)


# op counts around the fold's tiles (512 and 1,024), the sort's tiles (1,024 and 2,048), the switches to
# larger tiles (2^17, 2^19) and a fold chunk (2^20); record counts down to one hot record, up to a power of
# two, and slot counts whose sort keys take digits of more than 8 bits (17 to 20 and 25 to 30 bits)
@pytest.mark.parametrize("fb", [8, 16])
@pytest.mark.parametrize("n,nrec,nf", [
    (1, 1, 1), (511, 1, 1), (513, 2, 3), (1023, 1024, 1), (1024, 1000, 2), (1025, 3, 1), (4097, 1, 2),
    (1 << 17, 1 << 16, 8), ((1 << 17) + 1, 1 << 17, 1), (2049, 1 << 24, 1), (60000, (1 << 22) + 1, 10),
    ((1 << 18) + 77, (1 << 25) - 1, 1), ((1 << 19) - 1, 4096, 4), (1 << 19, 7, 1), ((1 << 19) + 1, 1 << 16, 3),
    ((1 << 20) + 1, 3, 1), ((1 << 21) - 1, 1 << 18, 4), ((1 << 21) + 1, 5, 1), ((1 << 22) + 4097, 1 << 12, 10)])
def test_tile_and_chunk_edges(eng, n, nrec, nf, fb):
    table, batch = make(nrec, nf, fb, n_txns=n, ops_per_txn=1, theta=0.6 if nrec > 8 else 0.0)
    (res, reads, stats), final = run(eng, table, batch, fb, 1)
    ref, ref_reads = oracle.serial(table, batch)
    assert stats["committed"] == n and stats["device_error"] == 0
    assert np.array_equal(res["commit_order"], np.arange(n))
    assert np.array_equal(reads, ref_reads) and np.array_equal(final, ref)


@pytest.mark.parametrize("fb", [8, 16])
@pytest.mark.parametrize("ops_range,max_ops", [((1, 8), 8), ((0, 9), 9), ((16, 16), 16), ((1, 17), 17),
                                               ((30, 33), 33), ((64, 64), 64), ((0, 64), 64)])
def test_group_widths_twice(eng, ops_range, max_ops, fb):
    """Ragged transactions for every lane-group width; the second run starts from the first's table."""
    table, batch = make(5003, 3, fb, n_txns=3001, ops_range=ops_range, theta=0.8)
    (res, reads, _), final = run(eng, table, batch, fb, max_ops, times=2)
    mid, _ = oracle.serial(table, batch)
    ref, ref_reads = oracle.serial(mid, batch)
    assert (res["status"] == oracle.ST_COMMITTED).all()
    assert np.array_equal(reads, ref_reads) and np.array_equal(final, ref)


@pytest.mark.parametrize("n_txns,ops_range", [(5, (1, 16)), (1024, (4, 16)), (40000, (1, 48))])
def test_invalid_and_left_out(eng, n_txns, ops_range):
    """A third of the transactions malformed in one way or another, and stray ops between the ranges: the
    others run as if those were not there, in ranks dense over them."""
    rng = np.random.default_rng(n_txns)
    nrec = 1 << 12
    table, full = make(nrec, 2, 8, n_txns=n_txns, ops_range=ops_range, theta=0.6)
    bad = rng.random(n_txns) < 0.33
    how = rng.integers(0, 4, size=n_txns)
    gaps = rng.integers(0, 3, size=n_txns + 1)
    n_ops = full.n_ops + int(gaps.sum())
    ops, opd = np.zeros(n_ops, dtype=wl.OP_DTYPE), np.zeros((n_ops, 2), dtype=np.uint64)
    ops["kind"], opd[:, 0] = wl.OP_ADD, 1                 # a stray op would add one to record 0
    txns = full.txns.copy()
    txns["first_op"] += np.cumsum(gaps)[:n_txns].astype(np.uint32)
    at = np.repeat(txns["first_op"].astype(np.int64) - full.txns["first_op"], txns["n_ops"]) + np.arange(full.n_ops)
    ops[at], opd[at] = full.ops, full.operands
    for t in np.flatnonzero(bad):
        f, k = int(txns["first_op"][t]), int(txns["n_ops"][t])
        if how[t] == 0:
            ops["key"][f + k - 1] = nrec
        elif how[t] == 1:
            ops["field"][f] = 9
        elif how[t] == 2 and k > 1:
            ops["key"][f] = ops["key"][f + k - 1]
        else:
            txns["type"][t] = wl.TXN_PAYMENT
    batch = wl.KVBatch(txns=txns, ops=ops, operands=opd)
    (res, reads, stats), final = run(eng, table, batch, 8, ops_range[1])
    good = np.flatnonzero(~bad)
    sub = wl.select(full, good)
    ref, ref_reads = oracle.serial(table, sub)
    assert stats["invalid"] == bad.sum() and stats["committed"] == good.size
    assert (res["status"][bad] == 3).all() and (res["commit_order"][bad] == wl.MASK64).all()
    assert np.array_equal(res["commit_order"][good], np.arange(good.size))
    pos = np.concatenate([np.arange(f, f + k) for f, k in zip(txns["first_op"][good], txns["n_ops"][good])])
    assert np.array_equal(reads[pos.astype(np.int64)], ref_reads) and np.array_equal(final, ref)


@pytest.mark.parametrize("k", [2, 7, 8, 15, 16, 17, 32, 33, 64])
def test_every_pair_of_equal_keys(eng, k):
    """A transaction of k ops for every two positions that share a key (record 0 among them, the value of
    an empty lane's descriptor): each is invalid, and the distinct one after it commits."""
    pairs = [(i, j) for i in range(k) for j in range(i + 1, k)]
    n = 2 * len(pairs)
    nrec = 101
    table, batch = make(nrec, 2, 8, n_txns=n, ops_range=(k, k), theta=0.0)
    keys = (np.arange(k)[None, :] + np.arange(n)[:, None] * 7) % nrec
    for p, (i, j) in enumerate(pairs):
        keys[2 * p, j] = keys[2 * p, i]
    batch.ops["key"] = keys.reshape(-1)
    (res, reads, stats), final = run(eng, table, batch, 8, k)
    good = np.arange(1, n, 2)
    ref, ref_reads = oracle.serial(table, wl.select(batch, good))
    assert (res["status"][::2] == 3).all() and (res["status"][good] == oracle.ST_COMMITTED).all()
    assert stats["invalid"] == len(pairs) and stats["committed"] == len(pairs)
    assert np.array_equal(reads.reshape(n, k, -1)[good].reshape(ref_reads.shape), ref_reads)
    assert np.array_equal(final, ref)


def test_slot_ids_of_32_bits(eng):
    """2^31 slots and more leave no spare bit in the sort key: reads of two batches in turn against the
    closed form of the seeded table."""
    nrec, nf, seed = 8421600, 255, 11
    batch = wl.kv_batch(9, nrec=nrec, nfields=nf, n_txns=3000, theta=0.6, permute_keys=True)
    batch.ops["field"][:100] = 254
    with eng.Database("kv", n_records=nrec, n_fields=nf, field_bytes=8, max_batch_txns=3000) as db:
        db.init_seeded(seed)
        got = [db.run("det", batch)[1] for _ in range(2)]
    slot = batch.ops["field"].astype(np.uint64) * np.uint64(nrec) + batch.ops["key"]
    init = wl.splitmix64_init(seed, batch.ops["key"].astype(np.uint64), batch.ops["field"], nf)
    now = dict(zip(slot.tolist(), init.tolist()))
    for reads in got:
        want = []
        for s, add, d in zip(slot.tolist(), batch.ops["kind"] == wl.OP_ADD, batch.operands[:, 0].tolist()):
            want.append(now[s])
            if add:
                now[s] = (now[s] + d) & wl.MASK64
        assert np.array_equal(reads[:, 0], np.array(want, dtype=np.uint64))
