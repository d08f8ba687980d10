"""Commit ranks of batches that draw more timestamps than the rank scratch has bits (32 per transaction of the
largest batch): transactions are listed by the timestamp's high bits.  Forced aborts use the timestamps up."""
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


def params(eng, aborts_ppm):
    return eng.params(immediate_restart=1, inject_abort_ppm=aborts_ppm)


# attempts per transaction from just past the bits to 1,000 (shifts of 5 to 10), sizes around a scan tile, and
# a batch without them before and after on the same database
@pytest.mark.parametrize("scheme", ["to", "mvcc"])
@pytest.mark.parametrize("n,ppm", [(2048, 973_000), (4097, 985_000), (5000, 999_000), (20_000, 975_000)])
def test_ranks_from_lists(eng, scheme, n, ppm):
    nrec = 1 << 14
    table = wl.kv_table_splitmix(1, nrec, 2)
    with eng.Database("kv", n_records=nrec, n_fields=2, max_ops_per_txn=2, max_batch_txns=n) as db:
        db.load_kv(table)
        for i, p in enumerate((None, params(eng, ppm), None, params(eng, ppm))):
            batch = wl.kv_batch(200 + i, nrec=nrec, nfields=2, n_txns=n, ops_per_txn=2)
            res, reads, stats = db.run(scheme, batch, p)
            final = db.read_kv()
            assert stats["committed"] == n and stats["device_error"] == 0, stats
            assert np.array_equal(np.sort(res["commit_order"]), np.arange(n))
            rep = oracle.replay_check(table, final, batch, res, reads)
            assert rep["ok"], (scheme, n, rep)
            table = final
            if p is not None:
                assert stats["aborts"] > 31 * n         # the lists were in use


def test_a_full_batch_is_ranked_in_parallel(eng):
    """2^20 transactions at 50 attempts each: the ranks take well under a millisecond (a radix sort of them 0.14,
    one block working through the timestamps 12)."""
    n, nrec = 1 << 20, 1 << 22
    batch = wl.kv_batch(5, nrec=nrec, nfields=1, n_txns=n, ops_per_txn=1)
    with eng.Database("kv", n_records=nrec, n_fields=1, max_ops_per_txn=1, max_batch_txns=n) as db:
        db.load_kv(wl.kv_table_splitmix(1, nrec, 1))
        for _ in range(2):
            res, _, stats = db.run("to", batch, params(eng, 980_000))
        assert stats["committed"] == n and stats["aborts"] > 40 * n, stats
        assert np.array_equal(np.sort(res["commit_order"]), np.arange(n))
        assert stats["order_ms"] < 1.0, stats
