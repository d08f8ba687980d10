"""What a sort whose bounded wait gave up leaves behind: positions of its output may hold words of an
earlier use of the buffer.  Every kernel that reads sorted pairs skips those that lie outside the array
it indexes, and treats the others as ever.  The pairs here are made by the test."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STRAY = np.array([0xffffffff, 0x7fffffff, 0x80000000, 0x00abcdef], dtype=np.uint32)
GUARD = 64                       # words behind each array that must stay as they were
MARK = 0x5A


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import harness
    torch.zeros(1, device="cuda")
    return harness.load(tmp_path_factory.mktemp("harness"))


def dev(a, guard=0):
    """A device copy of `a`, with `guard` marked elements behind it."""
    import torch
    a = np.ascontiguousarray(a)
    b = a.view(np.uint8).reshape(-1)
    b = np.concatenate([b, np.full(guard * a.itemsize, MARK, np.uint8)])
    return torch.from_numpy(b).cuda()


def host(t, dtype, n):
    """The first n elements; the guard behind them must be untouched."""
    b = t.cpu().numpy()
    size = n * np.dtype(dtype).itemsize
    assert (b[size:] == MARK).all()
    return b[:size].view(dtype)


def p(t):
    import ctypes
    return ctypes.c_void_p(t.data_ptr())


def u32(n):
    import ctypes
    return ctypes.c_uint32(n)


def u64(n):
    import ctypes
    return ctypes.c_uint64(n)


def strays(n, seed):
    """A permutation of 0..n-1 with one value in five replaced by one that is out of range."""
    rng = np.random.default_rng(seed)
    v = rng.permutation(n).astype(np.uint32)
    bad = rng.random(n) < 0.2
    v[bad] = np.append(STRAY, np.uint32(n))[rng.integers(0, 5, bad.sum())]
    return v, bad


COMMITTED = 1
RESULT = np.dtype([("status", "<u4"), ("attempts", "<u4"), ("commit_order", "<u8")])


def committed(n, order=0):
    res = np.zeros(n, dtype=RESULT)
    res["status"] = COMMITTED
    res["commit_order"] = order
    return res


@pytest.mark.parametrize("n", [5, 256, 1000])
def test_single_batch_consumers(lib, n):
    v, bad = strays(n, n)
    good = ~bad
    sv = dev(v, GUARD)
    # ranks
    d_res = dev(committed(n, 77), GUARD)
    assert lib[0].h_dense_rank(p(dev(np.zeros(n, np.uint32))), p(sv), u32(n), p(d_res)) == 0
    want = np.full(n, 77, np.uint64)
    want[v[good]] = np.flatnonzero(good)
    assert np.array_equal(host(d_res, RESULT, n)["commit_order"], want)
    # TicToc's second key, in place over the sorted order
    okey = np.arange(n, dtype=np.uint64) * 3
    keys, vals = dev(np.zeros(n, np.uint32), GUARD), dev(v, GUARD)
    assert lib[0].h_tt_emit(p(dev(committed(n))), p(dev(okey)), p(dev(np.zeros(n, np.uint32))), p(vals), 1,
                            u32(n), p(keys), p(vals)) == 0
    want = np.full(n, 0xffffffff, np.uint32)
    want[good] = v[good] * 3
    assert np.array_equal(host(keys, np.uint32, n), want) and np.array_equal(host(vals, np.uint32, n), v)
    # the deterministic scheme's access table: every op an ADD, keys with strays of their own
    ops = np.full(n, 1 << 40, dtype=np.uint64)
    flags = dev(np.zeros(n, np.uint32), GUARD)
    assert lib[0].h_det_flags(p(dev(ops)), p(sv), u64(n), p(flags)) == 0
    assert np.array_equal(host(flags, np.uint32, n), good.astype(np.uint32))
    k, kbad = strays(n, n + 1)
    need, meta = dev(np.full(n, 9, np.uint32), GUARD), dev(np.full(n, 9, np.uint64), GUARD)
    assert lib[0].h_det_need(p(dev(ops)), p(dev(k)), p(sv), p(dev(np.zeros(n, np.uint32))), u64(n), u32(n), p(need),
                             p(meta)) == 0
    both = good & ~kbad
    want = np.full(n, 9, np.uint32)
    want[v[both]] = np.flatnonzero(both)
    assert np.array_equal(host(need, np.uint32, n), want)
    want = np.full(n, 9, np.uint64)
    want[k[both]] = np.flatnonzero(both).astype(np.uint64) << np.uint64(32)
    assert np.array_equal(host(meta, np.uint64, n), want)
    # group commit's unit links
    link = dev(np.full(n, 9, np.uint32), GUARD)
    none = np.uint32(1 << 20)
    assert lib[1].h_unit_links(p(dev(np.full(n, none, np.uint32))), p(sv), u32(n), u32(4), u32(none), p(link)) == 0
    want = np.full(n, 9, np.uint32)
    want[v[good]] = 0x7fffffff
    assert np.array_equal(host(link, np.uint32, n), want)


@pytest.mark.parametrize("n0,n1", [(3, 2), (100, 300), (256, 0)])
def test_plan_consumers(lib, n0, n1):
    total = n0 + n1
    v, bad = strays(total, total)
    good = ~bad
    res = [dev(committed(n), GUARD) for n in (n0, n1)]
    okey = [dev(np.full(n, (i + 1) << 32, np.uint64)) for i, n in enumerate((n0, n1))]
    seq = [dev(np.zeros(n, np.uint32)) for n in (n0, n1)]
    prefix = np.array([0, n0, total], np.uint32)
    bkeys, tkeys = dev(np.zeros(total, np.uint32), GUARD), dev(np.zeros(total, np.uint32), GUARD)
    vals = dev(v, GUARD)
    assert lib[2].h_multi(p(res[0]), p(res[1]), p(okey[0]), p(okey[1]), p(seq[0]), p(seq[1]), p(dev(prefix)),
                          u64(total), p(bkeys), p(tkeys), p(vals)) == 0
    second = v >= n0
    want = np.where(good, second, 1).astype(np.uint32)
    assert np.array_equal(host(bkeys, np.uint32, total), want)
    want = np.where(good, second + 1, 0xffffffff).astype(np.uint32)
    assert np.array_equal(host(tkeys, np.uint32, total), want)
    assert np.array_equal(host(vals, np.uint32, total), v)
    for i, n in enumerate((n0, n1)):
        order = host(res[i], RESULT, n)["commit_order"]
        at = np.flatnonzero(good & (second == bool(i)))
        want = np.zeros(n, np.uint64)
        want[v[at] - prefix[i]] = (at - int(prefix[i])).astype(np.int64).view(np.uint64)
        assert np.array_equal(order, want)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 200])
def test_order_entry_runs_applied_in_order(lib, n):
    """A stock run whose positions name ops outside the batch: the others' values are stored, nothing else."""
    v, bad = strays(n, n + 7)
    v[bad] |= np.uint32(0x7fffff00)                    # bit 31 is the payment mark, not part of the number
    row, rows = 5, 100_000
    cols = [np.zeros(rows, np.uint64) for _ in range(4)]
    cols[0][row] = 50
    cols = [dev(c) for c in cols]
    opd = np.zeros((n, 2), np.uint64)
    opd[:, 0] = np.arange(n) % 10 + 1
    reads = dev(np.full((n, 2), 9, np.uint64), 2 * GUARD)
    assert lib[3].h_in_order(*[p(c) for c in cols], p(dev(np.full(n, 30011 + row, np.uint32))), p(dev(v)), u32(n),
                             p(dev(opd)), p(reads), u64(n), p(dev(np.array([1], np.uint32))),
                             p(dev(np.array([n - 1], np.uint32)))) == 0
    q, want = 50, np.full((n, 2), 9, np.uint64)
    for at in range(n):
        qty = 0 if bad[at] else int(opd[v[at], 0])
        if not bad[at]:
            want[v[at]] = (q, at)
        q = q - qty if q >= qty + 10 else q - qty + 91
    assert np.array_equal(host(reads, np.uint64, 2 * n).reshape(n, 2), want)
    assert int(cols[0].cpu().numpy().view(np.uint64)[row]) == q


@pytest.mark.parametrize("n", [1, 2, 256])
def test_every_batch_of_a_plan_reports_its_sort(lib, n):
    """The sorts that rank a plan's batches rank them all: a wait that gave up is every batch's error."""
    import ctypes
    out, begun = (ctypes.c_uint * n)(), ctypes.c_uint(7)
    assert lib[2].h_plan_error(u32(n), u32(4), u32(1), out, ctypes.byref(begun)) == 0
    assert begun.value == 0 and list(out) == [5] * n
    assert lib[2].h_plan_error(u32(n), u32(0), u32(1), out, ctypes.byref(begun)) == 0
    assert list(out) == [1] * n
