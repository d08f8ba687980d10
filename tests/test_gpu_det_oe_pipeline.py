"""The deterministic order-entry pipeline where it can go wrong, against the oracle's serial run in
transaction-id order: chains of one warehouse through many tiles and two chunks, stock rows and order
quantities outside the range whose quantities sum, name ids past the index's direct look-ups, and
malformed transactions with stray ops between them.  Every value must match exactly."""
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


def run(eng, db0, batch, W, cap, times=1):
    with eng.Database("oe", n_warehouses=W, order_cap=cap, max_ops_per_txn=33, max_batch_txns=batch.n_txns,
                      max_batch_ops=batch.n_ops) as db:
        db.load_oe(db0)
        for _ in range(times):
            out = db.run("det", batch)
        return out, db.read_oe()


def same(db0, batch, W, cap, out, final, times=1):
    res, reads, stats = out
    ref = db0
    for _ in range(times):
        ref, ref_reads = oracle.oe_serial(ref, W, cap, batch)
    assert stats["committed"] == batch.n_txns and stats["device_error"] == 0, stats
    assert np.array_equal(res["commit_order"], np.arange(batch.n_txns))
    assert np.array_equal(reads, ref_reads)
    for c in wl.OE_COLUMNS:
        assert np.array_equal(ref[c], final[c]), c


# a single transaction, one tile and one more, and past the 2^22 ops of a chunk (about 13 ops each)
@pytest.mark.parametrize("W,n_txns,times", [(1, 1, 2), (1, 39, 1), (3, 512, 2), (1, 1 << 15, 2), (1, 350_000, 1),
                                            (20, 20_000, 1)])
def test_sizes(eng, W, n_txns, times):
    batch = wl.oe_batch(n_txns, W, n_txns, by_name_frac=0.3)
    cap = wl.oe_order_cap([batch] * times, W)
    db0 = wl.oe_initial_db(n_txns, W, cap)
    out, final = run(eng, db0, batch, W, cap, times)
    same(db0, batch, W, cap, out, final, times)


@pytest.mark.parametrize("kind", ["quantity", "order", "remote", "all"])
def test_stock_outside_the_regular_range(eng, kind):
    """Initial quantities below 10, above 100 and negative; order quantities of 0, 91, 92, 2^40 and
    negative ones; remote counts above one: alone and mixed with regular rows, in chains of hundreds."""
    W, n = 1, 6000
    batch = wl.oe_batch(9, W, n)
    cap = wl.oe_order_cap([batch] * 2, W)
    db0 = wl.oe_initial_db(9, W, cap)
    rng = np.random.default_rng(4)
    if kind in ("quantity", "all"):
        hit = rng.random(db0["s_quantity"].size) < 0.3
        db0["s_quantity"][hit] = rng.choice([-5, 0, 9, 101, 1 << 40, -(1 << 40)], size=int(hit.sum()))
        hot = np.bincount(batch.ops["key"][batch.ops["kind"] == wl.OE_S_NEWORDER]).argmax()
        db0["s_quantity"][hot] = 101
    at = np.flatnonzero(batch.ops["kind"] == wl.OE_S_NEWORDER)
    if kind in ("order", "all"):
        odd = at[rng.random(at.size) < 0.1]
        batch.operands[odd, 0] = rng.choice(np.array([0, 91, 92, 1 << 40, -3], dtype=np.int64),
                                            size=odd.size).view(np.uint64)
    if kind in ("remote", "all"):
        odd = at[rng.random(at.size) < 0.05]
        batch.operands[odd, 1] = rng.choice(np.array([1, 2, 1 << 33], dtype=np.uint64), size=odd.size)
    out, final = run(eng, db0, batch, W, cap, 2)
    same(db0, batch, W, cap, out, final, 2)


def test_names_past_the_direct_look_ups(eng):
    """Last-name ids on both sides of 1,024 and the largest an op can name, some shared by many."""
    W, n = 2, 4000
    db0, batch, cap = wl.order_entry(seed=21, W=W, n_txns=n, by_name_frac=1.0)
    names = np.array([0, 1, 1023, 1024, 1025, 40000, 65535])
    rng = np.random.default_rng(2)
    db0["c_last"][:] = rng.choice(names, size=db0["c_last"].size)
    by = batch.ops["kind"] == wl.OE_C_PAY_BY_NAME
    batch.ops["aux"][by] = rng.choice(names, size=int(by.sum()))
    out, final = run(eng, db0, batch, W, cap)
    same(db0, batch, W, cap, out, final)


def test_malformed_and_left_out(eng):
    """A third of the transactions malformed, stray ops between the ranges: the rest run as if alone."""
    W, n = 2, 5000
    db0, full, cap = wl.order_entry(seed=33, W=W, n_txns=n)
    rng = np.random.default_rng(5)
    bad = rng.random(n) < 0.33
    gaps = rng.integers(0, 3, size=n + 1)
    txns = full.txns.copy()
    txns["first_op"] += np.cumsum(gaps)[:n].astype(np.uint32)
    ops = np.zeros(full.n_ops + int(gaps.sum()), dtype=wl.OP_DTYPE)
    opd = np.zeros((ops.size, 2), dtype=np.uint64)
    ops["kind"], opd[:, 0] = wl.OE_W_PAY, 5               # a stray op would pay warehouse 0
    at = np.repeat(txns["first_op"].astype(np.int64) - full.txns["first_op"], txns["n_ops"]) + np.arange(full.n_ops)
    ops[at], opd[at] = full.ops, full.operands
    for t in np.flatnonzero(bad):
        f, k = int(txns["first_op"][t]), int(txns["n_ops"][t])
        how = rng.integers(0, 4)
        if how == 0:
            ops["key"][f] = W
        elif how == 1:
            ops["kind"][f + k - 1] = wl.OE_I_READ
        elif how == 2 and k > 5:
            ops["key"][f + k - 1] = ops["key"][f + 4]      # one stock row twice
        else:
            txns["type"][t] = wl.TXN_KV
    batch = wl.KVBatch(txns=txns, ops=ops, operands=opd)
    (res, reads, stats), final = run(eng, db0, batch, W, cap)
    good = np.flatnonzero(~bad)
    ref, ref_reads = oracle.oe_serial(db0, W, cap, wl.select(full, good))
    assert stats["invalid"] == bad.sum() and stats["committed"] == good.size
    assert np.array_equal(res["commit_order"][good], np.arange(good.size)) and (res["status"][bad] == 3).all()
    pos = np.concatenate([np.arange(f, f + k) for f, k in zip(txns["first_op"][good], txns["n_ops"][good])])
    assert np.array_equal(reads[pos.astype(np.int64)], ref_reads)
    for c in wl.OE_COLUMNS:
        assert np.array_equal(ref[c], final[c]), c
