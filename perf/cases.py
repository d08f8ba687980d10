"""The workloads this engine is measured on: what a program that uses it has it do.

A case is a plain dict; ``prepare`` makes what a program has in hand before the call (a loaded
database and a batch, a plan or a server), ``run`` makes one pass through the public entry points of
``paper_2406_10158_gb300.engine``.  Four forms, as in ``include/gcc_gb300.h``:

* ``kv`` / ``oe``: a device-resident batch through ``Database.execute``;
* ``host``: a batch in host arrays through ``Database.run`` (copied in, executed, copied out);
* ``multi``: many databases' batches in one graph-replayed ``MultiPlan``;
* ``served``: a request trace through ``Server.run_trace``.

What a pass returns.  The deterministic scheme's outcome is fixed by the batch: its results and every
read value come back whole.  The other schemes may commit in any serial order, so commit order,
attempts and the values read under contention differ from run to run; ADDs commute, so every
transaction's status and the final table do not, and those come back (``returns: "table"``).  Where the
keys are uniform over many more slots than the batch touches, the reads agree between runs but for a
few in a thousand, and come back instead of a table far larger than the batch (``returns: "reads"``).
"""
import math

import numpy as np
import torch

from paper_2406_10158_gb300 import engine as eng
from paper_2406_10158_gb300 import workload as wl

DEV = "cuda:0"
CONCURRENT = ("occ", "2pl", "2pl_wd", "to", "tictoc", "mvcc")
_STREAM = None


def listed():
    return [
        # The small key-value store (65,536 records x 8 u64, 4,096 transactions x 16 ops) handed over
        # and taken back in host memory, as a program without device buffers of its own uses it.
        {"name": "host_occ_small", "form": "host", "scheme": "occ", "n_rec": 65536, "fields": 8, "fb": 8,
         "txns": 4096, "ops_lo": 16, "ops_hi": 16, "theta": 0.0, "read": 0.5, "returns": "table"},
        # The same store, device-resident, in id order: the smallest batches, one after another.
        {"name": "det_small", "form": "kv", "scheme": "det", "n_rec": 65536, "fields": 8, "fb": 8,
         "txns": 4096, "ops_lo": 16, "ops_hi": 16, "theta": 0.0, "read": 0.5, "returns": "reads"},
        # The full-size table (2^24 records x 10 fields in 16-byte slots, 2^20 transactions x 16 ops)
        # without contention: OCC and NO_WAIT two-phase locking.
        {"name": "occ_uniform", "form": "kv", "scheme": "occ", "n_rec": 1 << 24, "fields": 10, "fb": 16,
         "txns": 1 << 20, "ops_lo": 16, "ops_hi": 16, "theta": 0.0, "read": 0.5, "returns": "reads"},
        {"name": "2pl_uniform", "form": "kv", "scheme": "2pl", "n_rec": 1 << 24, "fields": 10, "fb": 16,
         "txns": 1 << 20, "ops_lo": 16, "ops_hi": 16, "theta": 0.0, "read": 0.95, "returns": "reads"},
        # The benchmark's default batch: the same table under high contention (Zipf 0.8).
        {"name": "occ_zipf080", "form": "kv", "scheme": "occ", "n_rec": 1 << 24, "fields": 10, "fb": 16,
         "txns": 1 << 20, "ops_lo": 16, "ops_hi": 16, "theta": 0.8, "read": 0.5, "returns": "table"},
        # Read-mostly transactions at medium contention, multi-version.
        {"name": "mvcc_zipf060", "form": "kv", "scheme": "mvcc", "n_rec": 1 << 22, "fields": 10, "fb": 16,
         "txns": 1 << 18, "ops_lo": 16, "ops_hi": 16, "theta": 0.6, "read": 0.95, "returns": "table"},
        # Odd and ragged: a record count that is no power of two, 4 to 64 ops a transaction, u64 slots.
        {"name": "tictoc_ragged", "form": "kv", "scheme": "tictoc", "n_rec": 1000003, "fields": 5, "fb": 8,
         "txns": 50021, "ops_lo": 4, "ops_hi": 64, "theta": 0.6, "read": 0.8, "returns": "table"},
        # The benchmark's batch in id order (the deterministic scheme).
        {"name": "det_zipf080", "form": "kv", "scheme": "det", "n_rec": 1 << 24, "fields": 10, "fb": 16,
         "txns": 1 << 20, "ops_lo": 16, "ops_hi": 16, "theta": 0.8, "read": 0.5, "returns": "reads"},
        # Order entry, half NewOrder and half Payment (`cap`: order slots per district, enough for some
        # hundreds of batches), at both ends of the warehouse range: one
        # warehouse (its row is in every transaction), and 64 with payments by last name.
        {"name": "det_oe_w1", "form": "oe", "scheme": "det", "W": 1, "txns": 1 << 18, "by_name": 0.0,
         "cap": 3 << 22},
        {"name": "det_oe_w64", "form": "oe", "scheme": "det", "W": 64, "txns": 1 << 18, "by_name": 0.6,
         "cap": 3 << 16},
        # 64 independent databases of uneven size in one graph launch.
        {"name": "multi_det", "form": "multi", "scheme": "det", "n_db": 64, "bits_lo": 16, "bits_hi": 22,
         "txns_lo": 1000, "txns_hi": 262144, "ops_lo": 4, "ops_hi": 64, "theta": 0.8, "read": 0.5},
        # The served form saturated: a key-value lane and an order-entry lane, all requests at hand.
        {"name": "served_det", "form": "served", "scheme": "det", "n_rec": 1 << 24, "fields": 8, "W": 8,
         "txns": 1 << 17, "theta": 0.8, "read": 0.8, "max_batch": 1 << 14, "cap": 1 << 17},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(("kv", "kv", "kv", "kv", "kv", "oe", "oe", "multi", "host", "served"))
    if form in ("kv", "host"):
        lo, hi = rng.choice(((16, 16), (16, 16), (4, 16), (4, 64)))
        case = {"form": form, "fields": rng.randint(1, 10), "fb": rng.choice((8, 16)), "ops_lo": lo, "ops_hi": hi,
                "read": rng.choice((0.5, 0.8, 0.95))}
        if rng.random() < 0.5:
            # the deterministic scheme over the whole range of sizes and contention
            case |= {"scheme": "det", "n_rec": _log(rng, 1 << 16, 1 << 24),
                     "txns": _log(rng, 1000, (1 << 20 if form == "kv" else 1 << 16) * 16 // hi),
                     "theta": rng.choice((0.0, 0.6, 0.8, 0.99)), "returns": "reads"}
        else:
            # the others up to medium contention: a few accesses per record at most
            case |= {"scheme": rng.choice(CONCURRENT),
                     "n_rec": _log(rng, 1 << 20, 1 << 24) if form == "kv" else _log(rng, 1 << 16, 1 << 20),
                     "theta": rng.choice((0.0, 0.6)), "returns": "table"}
            case["txns"] = _log(rng, 1000, min(1 << 20 if form == "kv" else 1 << 15, 2 * case["n_rec"] // hi))
        return case
    if form == "oe":
        W = _log(rng, 1, 64)
        return {"form": "oe", "scheme": "det", "W": W, "txns": _log(rng, 1000, 1 << 18),
                "by_name": rng.choice((0.0, 0.6)), "cap": (3 << 22) // W}
    if form == "multi":
        det = rng.random() < 0.5
        return {"form": "multi", "scheme": "det" if det else "occ", "n_db": rng.randint(2, 32), "bits_lo": 16,
                "bits_hi": rng.randint(17, 20), "txns_lo": 1000, "txns_hi": _log(rng, 2000, 1 << 15 if det else 1 << 12),
                "ops_lo": 4, "ops_hi": rng.choice((16, 64)) if det else 16, "theta": rng.choice((0.0, 0.8)) if det else 0.0,
                "read": rng.choice((0.5, 0.8))}
    W = rng.choice((4, 8, 16))
    return {"form": "served", "scheme": "det", "n_rec": _log(rng, 1 << 20, 1 << 24), "fields": 8, "W": W,
            "txns": _log(rng, 1 << 14, 1 << 17), "theta": 0.8, "read": rng.choice((0.5, 0.8)),
            "max_batch": 1 << rng.randint(10, 14), "cap": (1 << 20) // W}


# --- inputs -------------------------------------------------------------------
def _stream():
    """The stream a program issues its batches on."""
    global _STREAM
    if _STREAM is None:
        _STREAM = torch.cuda.Stream(DEV)
    return _STREAM


def _keys(gen, n_rec, theta, rows, width):
    """(rows, width) keys, distinct within a row: uniform, or Zipfian ranks (the closed form of Gray et
    al. that workload.zipf_ranks uses) scattered over the key space by a seeded permutation."""
    if theta == 0.0:
        def some(k):
            return torch.randint(0, n_rec, (k,), generator=gen, device=DEV)
    else:
        zetan = wl._zeta(n_rec, theta)
        alpha, top = 1.0 / (1.0 - theta), 1.0 + 2.0 ** (-theta)
        eta = (1.0 - (2.0 / n_rec) ** (1.0 - theta)) / (1.0 - top / zetan)
        perm = torch.randperm(n_rec, generator=gen, device=DEV)

        def some(k):
            u = torch.rand(k, generator=gen, device=DEV, dtype=torch.float64)
            r = ((u * eta + (1.0 - eta)).pow_(alpha).mul_(n_rec)).long().clamp_(0, n_rec - 1)
            uz = u * zetan
            r = torch.where(uz < 1.0 + 0.5 ** theta, torch.ones_like(r), r)
            return perm[torch.where(uz < 1.0, torch.zeros_like(r), r)]
    a = some(rows * width).view(rows, width)
    while True:
        s, at = a.sort(dim=1, stable=True)
        again = torch.zeros_like(a, dtype=torch.bool)
        again.scatter_(1, at[:, 1:], s[:, 1:] == s[:, :-1])
        k = int(again.sum())
        if k == 0:
            return a
        a[again] = some(k)


def _kv_inputs(gen, n_rec, fields, fb, txns, lo, hi, theta, read):
    """A key-value batch as device tensors in the C ABI's formats (gcc_txn, gcc_op, gcc_operand)."""
    count = lo + torch.randperm(txns, generator=gen, device=DEV) % (hi - lo + 1)
    first = torch.cumsum(count, 0) - count
    keys = _keys(gen, n_rec, theta, txns, hi)
    keys = keys[torch.arange(hi, device=DEV)[None, :] < count[:, None]] if lo < hi else keys.reshape(-1)
    n = keys.numel()
    field = torch.randint(0, fields, (n,), generator=gen, device=DEV)
    add = torch.rand(n, generator=gen, device=DEV) >= read
    operands = torch.zeros(n, 2, dtype=torch.int64, device=DEV)
    if fb == 8:
        operands[:, 0] = torch.randint(-1000, 1001, (n,), generator=gen, device=DEV) * add
    else:
        operands[:, 0] = torch.randint(-(1 << 62), 1 << 62, (n,), generator=gen, device=DEV) * add
        operands[:, 1] = torch.randint(0, 1 << 16, (n,), generator=gen, device=DEV) * add
    ops = keys | (field << 32) | (add.long() << 40)
    return first | (count << 32), ops, operands


def _outputs(n_txns, n_ops):
    """Room for gcc_txn_result (status | attempts << 32, commit order) and the values read."""
    return (torch.zeros(n_txns, 2, dtype=torch.int64, device=DEV),
            torch.zeros(n_ops, 2, dtype=torch.int64, device=DEV))


def _kv_db(n_rec, fields, fb, txns, n_ops, max_ops, seed):
    db = eng.Database("kv", n_records=n_rec, n_fields=fields, field_bytes=fb, max_ops_per_txn=max_ops,
                      max_batch_txns=txns, max_batch_ops=max(1, n_ops))
    db.init_seeded(seed)
    return db


def _oe_db(W, cap, txns, n_ops, seed):
    """An order-entry database whose order tables are still empty (order ids from 1)."""
    db = eng.Database("oe", n_warehouses=W, order_cap=cap, max_ops_per_txn=33, max_batch_txns=txns,
                      max_batch_ops=n_ops)
    rng = np.random.default_rng(seed)
    rows = wl.oe_column_rows(W, cap)
    d_ytd = rng.integers(0, 10_000_001, size=rows["d_ytd"])
    column = {"w_ytd": d_ytd.reshape(W, -1).sum(axis=1), "d_ytd": d_ytd,
              "d_next_o_id": np.ones(rows["d_ytd"], dtype=np.int64)}
    for name, lo, hi in (("w_tax", 0, 2001), ("d_tax", 0, 2001), ("c_balance", -100_000, 100_001),
                         ("c_ytd_payment", 0, 1_000_001), ("c_payment_cnt", 1, 11), ("c_discount", 0, 5001),
                         ("i_price", 100, 10_001), ("s_quantity", 10, 101)):
        column[name] = rng.integers(lo, hi, size=rows[name])
    column.update(wl.oe_customer_names(seed, W))
    for i, name in enumerate(wl.OE_COLUMNS):
        if name in column:
            db.load_table(i, np.ascontiguousarray(column[name], dtype=np.int64))
    return db


def _oe_batch(seed, W, txns, by_name):
    """A mix of fixed composition in random order, dealt like a deck of cards: half Payments, half
    NewOrders with equal shares of 5 to 15 lines."""
    b = wl.oe_batch(seed, W, txns + txns // 4 + 2000, by_name_frac=by_name)
    n_ops = b.txns["n_ops"]
    picked = [np.flatnonzero(n_ops == 3)[:txns - txns // 2]]
    for i in range(11):
        picked.append(np.flatnonzero(n_ops == 3 + 2 * (5 + i))[:(txns // 2 + i) // 11])
    return wl.select(b, np.sort(np.concatenate(picked)))


def _host_batch(txns, ops, operands):
    return wl.KVBatch(txns=txns.cpu().numpy().view(wl.TXN_DTYPE), ops=ops.cpu().numpy().view(wl.OP_DTYPE),
                      operands=operands.cpu().numpy().view(np.uint64))


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    form, s = case["form"], {"form": case["form"], "scheme": case["scheme"], "returns": case.get("returns")}
    if form in ("kv", "host"):
        tx, ops, opd = _kv_inputs(gen, case["n_rec"], case["fields"], case["fb"], case["txns"],
                                  case["ops_lo"], case["ops_hi"], case["theta"], case["read"])
        s["db"] = _kv_db(case["n_rec"], case["fields"], case["fb"], case["txns"], ops.numel(), case["ops_hi"],
                         seed)
        if s["returns"] == "table":
            s["table"] = torch.empty(s["db"].table_bytes(0) // 8, dtype=torch.int64, device=DEV)
        if form == "host":
            s["batch"] = _host_batch(tx, ops, opd)
        else:
            s["in"], s["out"] = (tx, ops, opd), _outputs(tx.numel(), ops.numel())
    elif form == "oe":
        b = _oe_batch(seed, case["W"], case["txns"], case["by_name"])
        s["db"] = _oe_db(case["W"], case["cap"], case["txns"], b.n_ops, seed)
        s["in"] = (torch.from_numpy(b.txns.view(np.int64)).to(DEV), torch.from_numpy(b.ops.view(np.int64)).to(DEV),
                   torch.from_numpy(b.operands.view(np.int64)).to(DEV))
        s["out"] = _outputs(b.n_txns, b.n_ops)
    elif form == "multi":
        s["entries"] = []
        for i, (bits, txns) in enumerate(_multi_sizes(case)):
            tx, ops, opd = _kv_inputs(gen, 1 << bits, 8, 8, txns, case["ops_lo"], case["ops_hi"], case["theta"],
                                      case["read"])
            db = _kv_db(1 << bits, 8, 8, txns, ops.numel(), case["ops_hi"], seed * 64 + i)
            s["entries"].append([db, tx, txns, ops, opd, ops.numel()])
        # every database's outputs side by side in one array
        s["out"] = _outputs(sum(e[2] for e in s["entries"]), sum(e[5] for e in s["entries"]))
        for e, res, reads in zip(s["entries"], s["out"][0].split([e[2] for e in s["entries"]]),
                                 s["out"][1].split([e[5] for e in s["entries"]])):
            e += [res, reads]
        s["plan"] = eng.MultiPlan(case["scheme"], s["entries"])
        if case["scheme"] != "det":
            words = [e[0].table_bytes(0) // 8 for e in s["entries"]]
            s["table"] = torch.empty(sum(words), dtype=torch.int64, device=DEV)
            s["tables"] = s["table"].split(words)
    else:
        half = case["txns"] // 2
        kv = wl.kv_batch(seed, nrec=case["n_rec"], nfields=case["fields"], n_txns=half,
                         ops_per_txn=16, read_ratio=case["read"], theta=case["theta"])
        oe = _oe_batch(seed + 1, case["W"], case["txns"] - half, 0.0)
        s["lane_of"] = (np.random.default_rng(seed).permutation(case["txns"]) >= half).astype(np.uint32)
        s["trace"] = wl.interleave([kv, oe], s["lane_of"])
        s["arrivals"] = np.zeros(case["txns"], dtype=np.uint64)
        mb = case["max_batch"]
        s["dbs"] = [_kv_db(case["n_rec"], case["fields"], 8, mb, mb * 16, 16, seed),
                    _oe_db(case["W"], case["cap"], mb, mb * 33, seed)]
        s["server"] = eng.Server([(db, case["scheme"], mb, 0, 400_000, 4) for db in s["dbs"]])
    torch.cuda.synchronize()
    return s


def _multi_sizes(case):
    """(log2 records, transactions) of every database: the same for every seed, as a program's plan is."""
    rng = np.random.default_rng(case["n_db"] * 1000003 + case["txns_hi"])
    bits = rng.integers(case["bits_lo"], case["bits_hi"] + 1, size=case["n_db"])
    txns = np.exp(rng.uniform(math.log(case["txns_lo"]), math.log(case["txns_hi"]), size=case["n_db"]))
    return [(int(b), int(round(t))) for b, t in zip(bits, txns)]


# --- one pass -------------------------------------------------------------------
def run(state):
    form, scheme = state["form"], state["scheme"]
    if form == "host":
        res, reads, _ = state["db"].run(scheme, state["batch"])
        if state["returns"] == "reads":
            return {"results": res.view(np.int64).reshape(-1, 2), "reads": reads.view(np.int64)}
        return {"status": res["status"], "table": _snapshot(state["db"], state["table"])}
    if form == "served":
        done, reads = state["server"].run_trace(state["lane_of"], state["trace"], state["arrivals"])
        return {"status": done["status"], "reads": reads.view(np.int64)}
    stream = _stream()
    if form == "multi":
        state["plan"].launch(True, stream.cuda_stream)
        res, reads = state["out"]
        if scheme == "det":
            return {"results": res, "reads": reads}
        for e, table in zip(state["entries"], state["tables"]):
            _snapshot(e[0], table)
        return {"status": res.view(torch.int32)[:, 0], "table": state["table"]}
    (tx, ops, opd), (res, reads) = state["in"], state["out"]
    state["db"].execute(scheme, tx, ops, opd, tx.numel(), ops.numel(), res, reads, stream=stream.cuda_stream)
    if scheme == "det":
        return {"results": res, "reads": reads}
    status = res.view(torch.int32)[:, 0]
    if state["returns"] == "reads":
        return {"status": status, "reads": reads}
    return {"status": status, "table": _snapshot(state["db"], state["table"])}


def _snapshot(db, into):
    """The table after the batch (gcc_db_read_table waits for the work before it)."""
    eng.gcc_db_read_table(db.handle, 0, into.data_ptr(), into.numel() * 8, True)
    return into


# --- what a pass cannot do without ------------------------------------------------
def _touched(accesses, n_rec, fields, theta):
    """Expected number of distinct (record, field) slots among `accesses` Zipfian(theta) ones."""
    if theta == 0.0:
        return n_rec * fields * -math.expm1(-accesses / (n_rec * fields))
    edges = np.unique(np.round(np.logspace(0, math.log10(n_rec + 1), 2000)))
    r = np.sqrt(edges[:-1] * edges[1:])
    p = r ** -theta / wl._zeta(n_rec, theta)
    return float(np.sum(np.diff(edges) * fields * -np.expm1(-accesses * p / fields)))


def _kv_bytes(txns, ops_mean, n_rec, fields, fb, theta, read):
    """Descriptor and result of each transaction; per op its descriptor and the value read; an operand
    per ADD; every touched slot read once, every added-to slot written once.  No control words: what a
    scheme keeps beside the data is its own choice."""
    n = txns * ops_mean
    return (24 * txns + n * (8 + 16) + n * (1 - read) * 16
            + fb * (_touched(n, n_rec, fields, theta) + _touched(n * (1 - read), n_rec, fields, theta)))


def _oe_bytes(txns, W):
    """NewOrder of 10 lines and Payment, half each: descriptors, results, operands, values read, the
    columns each op reads and writes (a row counted once where the batch touches it more often), and
    the inserted rows."""
    no = pay = txns / 2
    stock = _touched(no * 10, W * 100_000, 1, 0.0)
    cust = _touched(txns, W * 30_000, 1, 0.0)
    return (24 * txns + no * (23 * 24 + 10 * 16 + 32 + 10 * 32) + pay * 3 * (24 + 16)
            + stock * 64 + cust * 56 + 100_000 * 8)


def work(case):
    form = case["form"]
    if form in ("kv", "host"):
        mean = (case["ops_lo"] + case["ops_hi"]) / 2
        b = _kv_bytes(case["txns"], mean, case["n_rec"], case["fields"], case["fb"], case["theta"], case["read"])
    elif form == "oe":
        b = _oe_bytes(case["txns"], case["W"])
    elif form == "multi":
        mean = (case["ops_lo"] + case["ops_hi"]) / 2
        b = sum(_kv_bytes(t, mean, 1 << k, 8, 8, case["theta"], case["read"]) for k, t in _multi_sizes(case))
    else:
        half = case["txns"] / 2
        b = _kv_bytes(half, 16, case["n_rec"], case["fields"], 8, case["theta"], case["read"]) \
            + _oe_bytes(half, case["W"])
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    """Every output is a whole number, compared bit for bit; there is no rounding to measure."""
    return None
