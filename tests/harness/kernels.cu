// kernels.cu -- entry points for tests into kernels that the library only
// launches itself.  One translation unit of the engine is included per PART, so
// that its internal kernels can be called with buffers of the test's own.
#include <cstring>

#include <cuda_runtime.h>

#if PART == 0
#include "order.cu"
#elif PART == 1
#include "occ_group.cu"
#elif PART == 2
#include "multi.cu"
#elif PART == 3
#include "det_oe.cu"
#include "runtime.cuh"
#elif PART == 4
#include "det_fold.cu"
#include "runtime.cuh"
#endif

namespace {
unsigned grid_of(uint64_t n) { return (unsigned)((n + 255) / 256); }
int done() {
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
}  // namespace

extern "C" {
#if PART == 0
// A stable sort of (key, position) pairs by the passes with 64-bit descriptors, which otherwise only sorts of 2^30
// items and more take.  n above 2^19.
int h_sort_wide(uint32_t* keys, uint32_t n, int bits, int flagged, uint32_t* keys_out, uint32_t* vals_out) {
    if (gcc::sort_items(n) != gcc::SORT_ITEMS_LARGE) return -1;
    gcc::SortScratch s{};
    unsigned* err = nullptr;
    const size_t words = gcc::SORT_DESC + 2 * gcc::sort_tiles(n) * 256 * 2;
    cudaMalloc(&s.k1, n * 4ull);
    cudaMalloc(&s.v0, n * 4ull);
    cudaMalloc(&s.v1, n * 4ull);
    cudaMalloc(&s.work, words * 4);
    cudaMalloc(&err, 4);
    if (!s.k1 || !s.v0 || !s.v1 || !s.work || !err) return -1;
    s.k0 = keys;
    s.err = err;
    cudaMemset(err, 0, 4);
    cudaMemset(s.work, 0, words * 4);
    const gcc::SortPlan plan = gcc::sort_plan(bits);
    gcc::rs_hist<<<100, gcc::RS_BLOCK>>>(keys, n, bits, plan.passes, plan.digit_bits, s.work + gcc::SORT_HIST);
    uint32_t *sk = nullptr, *sv = nullptr;
    cudaError_t e = gcc::rs_passes<uint64_t, gcc::SORT_ITEMS_LARGE>(s, keys, nullptr, n, bits, flagged != 0, &sk, &sv, 0);
    unsigned bad = 1;
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(&bad, err, 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(keys_out, sk, n * 4ull, cudaMemcpyDeviceToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(vals_out, sv, n * 4ull, cudaMemcpyDeviceToDevice);
    cudaFree(s.k1);
    cudaFree(s.v0);
    cudaFree(s.v1);
    cudaFree(s.work);
    cudaFree(err);
    return bad ? -2 : (int)e;
}
int h_dense_rank(const uint32_t* sk, const uint32_t* sv, uint32_t n, gcc_txn_result* res) {
    gcc::dense_rank<<<grid_of(n), 256>>>(sk, sv, n, res);
    return done();
}
int h_tt_emit(const gcc_txn_result* res, const unsigned long long* okey, const uint32_t* seq, const uint32_t* sv,
              int pass, uint32_t n, uint32_t* keys, uint32_t* vals) {
    gcc::tt_emit<<<grid_of(n), 256>>>(res, okey, seq, sv, pass, n, keys, vals);
    return done();
}
int h_det_flags(const uint64_t* ops, const uint32_t* sv, uint64_t n, uint32_t* flags) {
    gcc::det_flags<<<grid_of(n), 256>>>(ops, sv, n, flags);
    return done();
}
int h_det_need(const uint64_t* ops, const uint32_t* sk, const uint32_t* sv, const uint32_t* wpre, uint64_t n,
               uint32_t none, uint32_t* need, uint64_t* meta) {
    gcc::det_need<<<grid_of(n), 256>>>(ops, sk, sv, wpre, n, none, 0, need, meta);
    return done();
}
#elif PART == 1
int h_unit_links(const uint32_t* sk, const uint32_t* sv, uint32_t n, uint32_t U, uint32_t none, uint32_t* link) {
    gcc::unit_links<<<grid_of(n), 256>>>(sk, sv, n, U, none, link);
    return done();
}
#elif PART == 2
// Two databases' results and commit keys; `prefix` on the device.
int h_multi(gcc_txn_result* r0, gcc_txn_result* r1, unsigned long long* o0, unsigned long long* o1, uint32_t* s0,
            uint32_t* s1, const uint32_t* prefix, uint64_t total, uint32_t* batch_keys, uint32_t* tt_keys,
            uint32_t* vals) {
    gcc::ExecArgs a[2]{}, *d = nullptr;
    a[0].results = r0;
    a[1].results = r1;
    a[0].order_key = o0;
    a[1].order_key = o1;
    a[0].seq = s0;
    a[1].seq = s1;
    cudaError_t e = cudaMalloc(&d, sizeof a);
    if (e == cudaSuccess) e = cudaMemcpy(d, a, sizeof a, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return (int)e;
    gcc::multi_batch_keys<<<grid_of(total), 256>>>(prefix, 2, total, batch_keys, vals);
    gcc::multi_tt_keys<<<grid_of(total), 256>>>(d, prefix, 2, total, 2, tt_keys, vals);
    gcc::multi_ranks<<<grid_of(total), 256>>>(d, prefix, 2, total, vals);
    const int r = done();
    cudaFree(d);
    return r;
}
// A plan of n databases that begins, has its sort set `sort_error` and ends; errors[i] as database i reports
// it, which had `own_error` before.  begun: the error word after the beginning.
int h_plan_error(uint32_t n, unsigned sort_error, unsigned own_error, unsigned* errors, unsigned* begun) {
    gcc::ExecArgs* args = nullptr;
    gcc::BatchState* st = nullptr;
    gcc::DbState* dbs = nullptr;
    gcc::DbState** own = nullptr;
    gcc::MultiState* ms = nullptr;
    cudaMallocManaged(&args, n * sizeof *args);
    cudaMallocManaged(&st, n * sizeof *st);
    cudaMallocManaged(&dbs, n * sizeof *dbs);
    cudaMallocManaged(&own, n * sizeof *own);
    cudaMallocManaged(&ms, sizeof *ms);
    if (!args || !st || !dbs || !own || !ms) return -1;
    std::memset(ms, 0xff, sizeof *ms);
    std::memset(dbs, 0, n * sizeof *dbs);
    for (uint32_t i = 0; i < n; ++i) {
        args[i] = gcc::ExecArgs{};
        args[i].st = st + i;
        own[i] = dbs + i;
    }
    gcc::multi_begin<<<1, 256>>>(args, own, n, ms, GCC_OCC);
    int r = done();
    *begun = ms->sort_error;
    ms->sort_error = sort_error;
    for (uint32_t i = 0; i < n; ++i) st[i].error = own_error;
    gcc::multi_end<<<1, 256>>>(args, own, n, ms);
    if (!r) r = done();
    for (uint32_t i = 0; i < n; ++i) errors[i] = st[i].error;
    cudaFree(args);
    cudaFree(st);
    cudaFree(dbs);
    cudaFree(own);
    cudaFree(ms);
    return r;
}
#elif PART == 3
// A run of stock accesses in positions 0..n-1 (one warehouse).
int h_in_order(uint64_t* quantity, uint64_t* ytd, uint64_t* cnt, uint64_t* remote, const uint32_t* sk,
               const uint32_t* sv, uint32_t n, const ulonglong2* operands, ulonglong2* reads, uint64_t n_ops,
               const uint32_t* n_odd, const uint32_t* odd) {
    gcc::ExecArgs a{};
    a.n_warehouses = 1;
    a.n_meta = 130011;
    a.operands = operands;
    a.reads = reads;
    a.n_ops = n_ops;
    gcc::OeTables T{};
    T.c[gcc::oe::S_QUANTITY] = quantity;
    T.c[gcc::oe::S_YTD] = ytd;
    T.c[gcc::oe::S_ORDER_CNT] = cnt;
    T.c[gcc::oe::S_REMOTE_CNT] = remote;
    const gcc::AccessKeys f = gcc::access_keys(a.n_meta, n, gcc::OE_CHUNK_LOG2, gcc::OE_SORT_LOG2, true);
    gcc::oe_in_order<<<1, 256>>>(a, T, f, sk, sv, 0, 0, n, n_odd, odd);
    return done();
}
#endif
#if PART >= 3
// The whole pipeline on a database's own scratch, 2^sort_log2 ops to a sort.
int h_batch_in_parts(gcc_db* db, const gcc_txn* txns, uint32_t n_txns, const uint64_t* ops, const ulonglong2* operands,
                     uint64_t n_ops, gcc_txn_result* results, ulonglong2* reads, int sort_log2) {
    gcc::ExecArgs a{};
    a.txns = txns;
    a.ops = ops;
    a.operands = operands;
    a.n_txns = n_txns;
    a.n_ops = n_ops;
    a.results = results;
    a.reads = reads;
    a.table = db->table;
    a.n_records = db->d.n_records;
    a.n_fields = db->d.n_fields;
    a.n_meta = db->n_meta;
    a.n_warehouses = db->d.n_warehouses;
    a.order_cap = db->d.order_cap;
    a.max_ops = db->d.max_ops_per_txn;
    a.st = db->st;
    a.dbs = db->dbs;
    uint32_t launches = 0;
#if PART == 3
    gcc::OeTables T{};
    for (int c = 0; c < gcc::rt::OE_NCOLS; ++c) T.c[c] = reinterpret_cast<uint64_t*>(db->cols[c]);
    T.names = gcc::NameIndex{db->name_idx, db->name_last, db->name_pick};
    const cudaError_t e = gcc::oe_run(a, T, db->sort, db->fold_seg, db->need, launches, 0, sort_log2);
#else
    const cudaError_t e = db->d.field_bytes == 16
                              ? gcc::fold_run<16>(a, db->sort, db->fold_seg, launches, 0, sort_log2)
                              : gcc::fold_run<8>(a, db->sort, db->fold_seg, launches, 0, sort_log2);
#endif
    return e != cudaSuccess ? (int)e : done();
}
#endif
}
