"""2PL's 4-byte control words stand 16 bytes apart for up to 2^22 records and side by side for more.  Contended
batches on the first and last records on both sides of the line, in turn with schemes that use the array in
other ways, and plans whose databases cross it only together."""
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


def ends(seed, nrec, n_txns, fb):
    """Transactions on the first and the last 32 records."""
    b = wl.kv_batch(seed, nrec=64, nfields=1, field_bytes=fb, n_txns=n_txns, ops_per_txn=6, theta=0.6)
    ops = b.ops.copy()
    high = ops["key"] >= 32
    ops["key"][high] = nrec - 1 - (ops["key"][high] - 32)
    return wl.KVBatch(txns=b.txns, ops=ops, operands=b.operands)


@pytest.mark.parametrize("fb", [8, 16])
@pytest.mark.parametrize("nrec", [64, (1 << 22) - 1, 1 << 22, (1 << 22) + 1])
def test_both_layouts(eng, nrec, fb):
    n = 700
    table = wl.kv_table_bytes(3, nrec, 1) if fb == 16 else wl.kv_table_splitmix(3, nrec, 1)
    with eng.Database("kv", n_records=nrec, n_fields=1, field_bytes=fb, max_ops_per_txn=6, max_batch_txns=n) as db:
        db.load_kv(table)
        for i, scheme in enumerate(("2pl", "occ", "2pl_wd", "to", "2pl", "mvcc", "2pl_wd", "tictoc", "2pl")):
            batch = ends(i, nrec, n, fb)
            res, reads, stats = db.run(scheme, batch)
            final = db.read_kv()
            assert stats["committed"] == n, (scheme, stats)
            rep = oracle.replay_check(table, final, batch, res, reads)
            assert rep["ok"], (scheme, rep)
            table = final


@pytest.mark.parametrize("scheme", ["2pl", "2pl_wd"])
@pytest.mark.parametrize("nrecs", [(1 << 21, 1 << 21), (1 << 21, (1 << 21) + 1), ((1 << 22) + 5, 100)])
def test_plans(eng, scheme, nrecs):
    """The plan's layout goes by all its records; a database runs by itself in its own before and after."""
    import torch
    n, fb = 500, 8
    dbs, state, entries = [], [], []
    for i, nrec in enumerate(nrecs):
        db = eng.Database("kv", n_records=nrec, n_fields=1, field_bytes=fb, max_ops_per_txn=6, max_batch_txns=n)
        table = wl.kv_table_splitmix(i, nrec, 1)
        db.load_kv(table)
        b = ends(10 + i, nrec, n, fb)
        dev = [torch.from_numpy(np.ascontiguousarray(x).view(np.uint8).reshape(-1)).cuda()
               for x in (b.txns, b.ops, b.operands)]
        out = [torch.zeros(k * 16, dtype=torch.uint8, device="cuda") for k in (n, b.n_ops)]
        entries.append((db, dev[0], n, dev[1], dev[2], b.n_ops, *out))
        dbs.append((db, b, out))
        state.append(table)

    def alone():
        for i, (db, b, _) in enumerate(dbs):
            res, reads, stats = db.run(scheme, b)
            final = db.read_kv()
            assert stats["committed"] == n and oracle.replay_check(state[i], final, b, res, reads)["ok"]
            state[i] = final

    alone()
    plan = eng.MultiPlan(scheme, entries)
    for graph in (False, True):
        plan.launch(graph)
        torch.cuda.synchronize()
        for i, (db, b, (res, reads)) in enumerate(dbs):
            final = db.read_kv()
            r = res.cpu().numpy().view(wl.RESULT_DTYPE)
            rd = reads.cpu().numpy().view(np.uint64).reshape(-1, 2)
            assert plan.stats(i)["committed"] == n
            assert oracle.replay_check(state[i], final, b, r, rd)["ok"]
            state[i] = final
    alone()
