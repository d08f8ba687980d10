"""Paths that only batches of 2^29 and more ops take, at small sizes: sort passes with 64-bit tile descriptors,
and deterministic batches that are sorted and folded in parts, here 2^20 (order entry: 2^22) ops at a time,
against the same batch in one sort."""
import numpy as np
import pytest

from paper_2406_10158_gb300 import workload as wl
from test_gpu_sort_give_up import dev, host, lib, p, u32, u64   # noqa: F401  (lib is the fixture)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    from paper_2406_10158_gb300 import engine
    return engine


@pytest.mark.parametrize("n", [(1 << 19) + 1, (1 << 20) + 4097])
@pytest.mark.parametrize("bits,flagged", [(1, 1), (8, 0), (9, 1), (24, 0), (31, 1), (32, 0)])
def test_sort_with_wide_descriptors(lib, n, bits, flagged):   # noqa: F811
    rng = np.random.default_rng(bits * n)
    key = rng.integers(0, 1 << bits, n, dtype=np.uint64).astype(np.uint32)
    flag = rng.integers(0, 2, n, dtype=np.uint32) << np.uint32(31) if flagged else np.zeros(n, np.uint32)
    ko, vo = dev(np.zeros(n, np.uint32), 16), dev(np.zeros(n, np.uint32), 16)
    assert lib[0].h_sort_wide(p(dev(key | flag)), u32(n), bits, flagged, p(ko), p(vo)) == 0
    at = np.argsort(key, kind="stable").astype(np.uint32)
    assert np.array_equal(host(ko, np.uint32, n), key[at])
    assert np.array_equal(host(vo, np.uint32, n), at | flag[at])


def in_parts(part, db, batch, sort_log2):
    import ctypes
    res = dev(np.zeros(batch.n_txns, dtype=wl.RESULT_DTYPE), 16)
    reads = dev(np.zeros((batch.n_ops, 2), np.uint64), 16)
    assert part.h_batch_in_parts(ctypes.c_void_p(db.handle), p(dev(batch.txns)), u32(batch.n_txns), p(dev(batch.ops)),
                                 p(dev(batch.operands)), u64(batch.n_ops), p(res), p(reads), sort_log2) == 0
    return (host(res, wl.RESULT_DTYPE, batch.n_txns),
            host(reads, np.uint64, 2 * batch.n_ops).reshape(-1, 2))


# two parts and three; chains through all of them (16 records), many records, and slot ids of 32 bits, which leave
# the keys no bit for the op's kind and none for chunks
@pytest.mark.parametrize("fb,n_txns,nrec,nf,form", [
    (fb, n_txns, nrec, nf, form) for fb in (8, 16) for n_txns, nrec, nf in ((350_000, 16, 2), (420_000, 1 << 16, 8))
    for form in ("regular", "gaps", "invalid")] + [(8, 350_000, 1 << 28, 8, "regular")])
def test_kv_batches_in_parts(lib, eng, fb, n_txns, nrec, nf, form):   # noqa: F811
    b = wl.kv_batch(9, nrec=nrec, nfields=nf, field_bytes=fb, n_txns=n_txns, ops_range=(1, 10))
    assert b.n_ops > 1 << 20
    txns, ops = b.txns.copy(), b.ops.copy()
    if form == "gaps":
        txns = txns[np.arange(n_txns) % 7 != 3]
    if form == "invalid":
        ops["key"][::501] = nrec                       # no such record
    b = wl.KVBatch(txns=txns, ops=ops, operands=b.operands)
    out = []
    for parts in (False, True):
        with eng.Database("kv", n_records=nrec, n_fields=nf, field_bytes=fb, max_ops_per_txn=10,
                          max_batch_txns=b.n_txns, max_batch_ops=b.n_ops) as db:
            db.init_seeded(5)
            res, reads = in_parts(lib[4], db, b, 20) if parts else db.run("det", b)[:2]
            out.append((res, reads, db.read_kv() if nrec <= 1 << 16 else None))
    (res, reads, table), (res2, reads2, table2) = out
    ok = res["status"] == 1
    assert ok.all() == (form != "invalid") and ok.sum() > 0.9 * b.n_txns
    assert np.array_equal(res, res2)
    used = np.zeros(b.n_ops, bool)                     # values read by committed transactions
    for t in np.flatnonzero(ok):
        used[txns["first_op"][t]:txns["first_op"][t] + txns["n_ops"][t]] = True
    assert np.array_equal(reads[used], reads2[used])
    if table is not None:
        assert np.array_equal(table, table2)


def test_oe_batches_in_parts(lib, eng):   # noqa: F811
    W, n = 2, 350_000
    b = wl.oe_batch(4, W, n, by_name_frac=0.3)
    assert b.n_ops > 1 << 22
    cap = wl.oe_order_cap([b], W)
    db0 = wl.oe_initial_db(4, W, cap)
    db0["s_quantity"][::97] = 101                       # some rows outside the regular range
    out = []
    for parts in (False, True):
        with eng.Database("oe", n_warehouses=W, order_cap=cap, max_ops_per_txn=33, max_batch_txns=n,
                          max_batch_ops=b.n_ops) as db:
            db.load_oe(db0)
            res, reads = in_parts(lib[3], db, b, 22) if parts else db.run("det", b)[:2]
            out.append((res, reads, db.read_oe()))
    (res, reads, final), (res2, reads2, final2) = out
    assert np.array_equal(res, res2) and np.array_equal(reads, reads2)
    for c in wl.OE_COLUMNS:
        assert np.array_equal(final[c], final2[c]), c
