"""The end of a batch under the schemes that cut backoffs short there (2PL,
2PL wait-die, TicToc, MVCC): contended batches end, and their histories replay.
"""
import numpy as np
import pytest

import oracle
from paper_2406_10158_gb300 import workload as wl

pytestmark = pytest.mark.gpu

SCHEMES = ["2pl", "2pl_wd", "tictoc", "mvcc"]


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_10158_gb300 import engine
    return engine


@pytest.mark.parametrize("n_txns", [48, 1000])
@pytest.mark.parametrize("scheme", SCHEMES)
def test_long_conflicting_transactions_end(eng, scheme, n_txns):
    """60-op transactions on 512 records, nearly every pair in conflict, far
    more aborts than a transaction makes before it joins retry queues: with the
    default policy all commit well before the 20 s deadline."""
    nrec = 512
    table = wl.kv_table_splitmix(31, nrec, 2)
    batch = wl.kv_batch(32, nrec=nrec, nfields=2, n_txns=n_txns, ops_per_txn=60, read_ratio=0.5)
    with eng.Database("kv", n_records=nrec, n_fields=2, field_bytes=8, max_ops_per_txn=60,
                      max_batch_txns=n_txns) as db:
        db.load_kv(table)
        res, reads, stats = db.run(scheme, batch, eng.params(deadline_ns=20_000_000_000))
        final = db.read_kv()
    assert stats["committed"] == n_txns, stats
    rep = oracle.replay_check(table, final, batch, res, reads)
    assert rep["ok"], rep


@pytest.mark.parametrize("scheme", SCHEMES)
def test_small_batches_of_every_launch_shape_end(eng, scheme):
    """Blocks of one lane group up to 32: the look at who is still at work
    counts groups, so every shape is a different count."""
    nrec = 256
    table = wl.kv_table_splitmix(33, nrec, 2)
    batch = wl.kv_batch(34, nrec=nrec, nfields=2, n_txns=333, ops_per_txn=16, read_ratio=0.5, theta=0.9)
    with eng.Database("kv", n_records=nrec, n_fields=2, field_bytes=8, max_ops_per_txn=16,
                      max_batch_txns=333) as db:
        for lanes, warps in ((32, 1), (32, 8), (16, 1), (8, 4), (1, 1), (2, 2)):
            db.load_kv(table)
            res, reads, stats = db.run(scheme, batch, eng.params(
                lanes_per_txn=lanes, warps_per_block=warps, deadline_ns=20_000_000_000))
            assert stats["committed"] == 333, (lanes, warps, stats)
            rep = oracle.replay_check(table, db.read_kv(), batch, res, reads)
            assert rep["ok"], (lanes, warps, rep)


@pytest.mark.parametrize("scheme", SCHEMES)
def test_backoff_the_caller_set_is_kept(eng, scheme):
    """256 transactions on one record, delays of 0, 20 or 40 ms: each delay is
    sat out in full, so the kernel takes at least the 20 ms of the shortest one
    that is not zero (one microsecond per lane group would be 0.26 ms)."""
    table = wl.kv_table_splitmix(35, 16, 1)
    batch = wl.kv_batch_from_lists([[(3, 0, 1, t + 1, 0)] for t in range(256)])
    with eng.Database("kv", n_records=16, n_fields=1, field_bytes=8, max_batch_txns=256) as db:
        db.load_kv(table)
        res, reads, stats = db.run(scheme, batch, eng.params(
            backoff_base_ns=20_000_000, backoff_cap_ns=40_000_000, retry_queue=2))
        final = db.read_kv()
    assert stats["committed"] == 256, stats
    assert oracle.replay_check(table, final, batch, res, reads)["ok"]
    waited = res["attempts"][res["attempts"] > 1].size
    assert waited >= 32, stats                      # all of them draw zero: below 2^-32
    assert stats["kernel_ms"] >= 20.0, stats
