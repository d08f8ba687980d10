"""Commit ranks of the timestamp schemes: one bit per timestamp, ranked by a scan over the words.  Sizes
around a word, a scan tile (4,096 words) and the smallest scratch, repeated batches on one database, and
batches that use up many more timestamps than the scratch holds (forced aborts)."""
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


def run(eng, scheme, n, times, max_txns=None, **kw):
    nrec = 1 << 14
    table = wl.kv_table_splitmix(1, nrec, 2)
    with eng.Database("kv", n_records=nrec, n_fields=2, max_ops_per_txn=2,
                      max_batch_txns=max_txns or n) as db:
        db.load_kv(table)
        for i in range(times):
            batch = wl.kv_batch(100 + i, nrec=nrec, nfields=2, n_txns=n, ops_per_txn=2)
            res, reads, stats = db.run(scheme, batch, eng.params(**kw) if kw else None)
            final = db.read_kv()
            assert stats["committed"] == n and stats["device_error"] == 0, stats
            assert np.array_equal(np.sort(res["commit_order"]), np.arange(n))
            rep = oracle.replay_check(table, final, batch, res, reads)
            assert rep["ok"], (scheme, n, rep)
            table = final
        return stats


@pytest.mark.parametrize("scheme", ["occ", "to", "mvcc"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 2047, 131071, 131073])
def test_sizes(eng, scheme, n):
    run(eng, scheme, n, 2)


@pytest.mark.parametrize("scheme", ["occ", "to", "mvcc"])
def test_small_batch_of_a_large_database(eng, scheme):
    run(eng, scheme, 100, 3, max_txns=1 << 17)


@pytest.mark.parametrize("scheme", ["to", "mvcc"])
def test_more_timestamps_than_the_scratch_holds(eng, scheme):
    """4,096 transactions whose attempts abort 99 times in 100: about 400,000 timestamps, where the
    scratch of this database holds 131,072; the batch after it is ranked as usual."""
    stats = run(eng, scheme, 4096, 1, immediate_restart=1, inject_abort_ppm=990000)
    assert stats["aborts"] > 200_000
    nrec = 1 << 14
    with eng.Database("kv", n_records=nrec, n_fields=2, max_ops_per_txn=2, max_batch_txns=4096) as db:
        table = wl.kv_table_splitmix(1, nrec, 2)
        db.load_kv(table)
        batch = wl.kv_batch(3, nrec=nrec, nfields=2, n_txns=4096, ops_per_txn=2)
        for p in (eng.params(immediate_restart=1, inject_abort_ppm=990000), None):
            res, reads, stats = db.run(scheme, batch, p)
            final = db.read_kv()
            assert oracle.replay_check(table, final, batch, res, reads)["ok"]
            table = final
