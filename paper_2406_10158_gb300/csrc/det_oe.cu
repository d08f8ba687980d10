// det_oe.cu -- the deterministic scheme on order-entry batches: every
// record's chain of accesses evaluated by prefix sums over the sorted access
// table.
//
// The deterministic scheme's outcome is serial execution in transaction-id
// order (Sec. II-C, GPUTx).  That outcome decomposes by record: every
// order-entry op computes its record's new columns from that record's old
// columns and its own operand only, so a record's accesses applied in id order
// from its initial state give exactly the values the serial run reads and the
// record it leaves.  Sorted by (record, position), each record's chain is a
// segment, and each class of records sums:
//   warehouse, district, customer: ops add their amount, or one, to columns;
//   stock: s_ytd, s_order_cnt and s_remote_cnt add up.  The quantity rule
//     (q - qty, plus 91 when q < qty + 10) maps 10..100 to itself for every
//     qty in 0..91 and keeps q - qty modulo 91; 10..100 holds each residue
//     once, so the quantity after any number of orders is the value in that
//     range congruent to the initial one less the sum of their quantities.
// So a segmented prefix sum of (amount, count, remote) gives every value read,
// however long the longest chain (a one-warehouse batch has its warehouse row
// in every transaction).  A stock row whose quantity, or an order whose
// quantity or remote flag, lies outside those ranges is applied in order
// instead (oe_in_order).
//
//   begin     batch state, descriptors and histograms zeroed
//   validate  a half-warp per transaction: the execute kernel's checks,
//             payments by last name resolved, item reads answered, every
//             op's access key, the digit histograms of the sort
//   sort      by (chunk, record), as the key-value pipeline (det_fold.cu)
//   fold      per chunk: values read out, final columns in
//   in order  the stock rows that left the regular range
//   commit    NewOrder inserts
//   finish    commit counts; commit order where a transaction was invalid
#include "det_common.cuh"
#include "oe_work.cuh"

namespace gcc {
namespace {

using namespace oe;

constexpr int OF_THREADS = 256;
constexpr int OF_ITEMS = 2;
constexpr int OF_TILE = OF_THREADS * OF_ITEMS;
constexpr int OF_WARPS = OF_THREADS / 32;
// Ops per chunk.  Order-entry tables are small beside a key-value table, so it
// pays to go through them seldom rather than to keep operands and values read in
// L2: 13.6 M ops at 64 warehouses take 1,367 us in chunks of 2^22 ops, 1,426 of
// 2^21 and 1,472 of 2^20; 6.8 M ops 648, 734 and 758; 13.6 M at one warehouse
// 1,157, 1,140 and 1,145.
constexpr int OE_CHUNK_LOG2 = 22;
// Ops per sort: the tile descriptors hold counts of 30 bits.
constexpr int OE_SORT_LOG2 = 29;
constexpr int64_t Q_LO = 10, Q_HI = 100, Q_MOD = 91;

// --- validation and access table ---------------------------------------------
// A half-warp per transaction, lane l holding order line l (its item read and
// its stock op) and, for l < 3, head op l; two transactions per half-warp at
// once.  Bit 31 of a key: the op is a Payment's.  Only stock rows can repeat
// within a well-formed transaction (its head ops are of different tables), so
// one match over the half-warp replaces a comparison of every pair of ops.
// Bound by the transaction's chain of loads and the histogram updates: 61 us for
// 2^18 transactions (a warp per transaction and all pairs: 226 us).
__global__ void __launch_bounds__(256)
oe_validate(const __grid_constant__ ExecArgs a, const __grid_constant__ OeTables T, const AccessKeys f,
            uint32_t* keys, uint32_t* work, uint32_t per_block) {
    constexpr int U = 2, STEP = 16 * U;
    __shared__ DigitHist h[SORT_MAX_PASSES];
    const int lane = threadIdx.x & 31, lig = lane & 15;
    const unsigned gmask = 0xffffu << (lane & 16);
    clear_digits(h);
    after_previous();
    __syncthreads();
    const bool tiled = work[DW_UNTILED] == 0;
    const uint32_t W = a.n_warehouses;
    uint64_t t_end = (uint64_t)(blockIdx.x + 1) * per_block;
    if (t_end > a.n_txns) t_end = a.n_txns;
    unsigned invalid = 0;
    for (uint64_t t0 = (uint64_t)blockIdx.x * per_block; t0 < t_end; t0 += STEP) {
        const uint64_t tb = t0 + (threadIdx.x >> 4) * U;
        uint32_t first[U], nops[U], type[U];
        bool bad[U], inside[U];
        uint64_t head[U], item[U], stock[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            gcc_txn tx{0u, 0, 0};
            if (tb + u < t_end) tx = a.txns[tb + u];
            first[u] = tx.first_op;
            nops[u] = tx.n_ops;
            type[u] = tx.type;
            inside[u] = tb + u < t_end && (uint64_t)tx.first_op + tx.n_ops <= a.n_ops;
            bad[u] = tx.n_ops > a.max_ops || tx.n_ops > 64 || !inside[u] ||
                     !(type[u] == GCC_TXN_PAYMENT ? nops[u] == 3
                                                  : type[u] == GCC_TXN_NEW_ORDER && nops[u] >= 5 &&
                                                        nops[u] <= 3 + 2 * LINES && (nops[u] & 1));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t* op = a.ops + first[u];
            head[u] = !bad[u] && lig < 3 ? op[lig] : 0ull;
            const bool line = !bad[u] && 3 + 2 * lig < nops[u];
            item[u] = line ? op[3 + 2 * lig] : 0ull;
            stock[u] = line ? op[4 + 2 * lig] : 0ull;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool pay = type[u] == GCC_TXN_PAYMENT;
            const bool line = !bad[u] && 3 + 2 * lig < nops[u];
            bool wrong = false;
            uint32_t hrec = f.none;
            if (!bad[u] && lig < 3) {
                uint32_t kind = op_kind(head[u]), row = op_key(head[u]);
                if (pay && lig == 2 && kind == GCC_OE_C_PAY_BY_NAME) {
                    row = T.names.customer(W, row, (uint32_t)(head[u] >> 48));   // ~0u: nobody
                    kind = GCC_OE_C_PAY;
                }
                const uint32_t want = lig == 0   ? (pay ? GCC_OE_W_PAY : GCC_OE_W_READ)
                                      : lig == 1 ? (pay ? GCC_OE_D_PAY : GCC_OE_D_NEWORDER)
                                                 : (pay ? GCC_OE_C_PAY : GCC_OE_C_READ);
                const uint32_t rows = lig == 0 ? W : lig == 1 ? DIST * W : DIST * CUST * W;
                const uint32_t base = lig == 0 ? 0u : lig == 1 ? W : 11u * W;
                wrong = kind != want || row >= rows;
                hrec = base + row;
            }
            if (line)
                wrong = wrong || op_kind(item[u]) != GCC_OE_I_READ || op_key(item[u]) >= ITEMS ||
                        op_kind(stock[u]) != GCC_OE_S_NEWORDER || op_key(stock[u]) >= ITEMS * W;
            const unsigned holders = __ballot_sync(0xffffffffu, line);
            const unsigned peers = __match_any_sync(0xffffffffu, op_key(stock[u]));
            if (line && __popc(peers & holders & gmask) > 1) wrong = true;
            const unsigned any = __ballot_sync(0xffffffffu, wrong);   // by every lane of the warp
            const bool no = bad[u] || (any & gmask);
            const uint64_t op0 = first[u];
            if (!bad[u] && lig < 3) {
                const uint32_t k = f.key(op0 + lig, no ? f.none : hrec, !no && pay);
                put_key(f, h, keys, op0 + lig, k, tiled);
            }
            if (line) {
                const uint64_t op = op0 + 3 + 2 * lig;
                const uint32_t ki = f.key(op, f.none, false);
                const uint32_t ks = f.key(op + 1, no ? f.none : 30011u * W + op_key(stock[u]), false);
                if (!no) a.reads[op] = make_ulonglong2((uint64_t)T.c[I_PRICE][op_key(item[u])], 0ull);
                // the item reads' keys are all one but for the chunk: counted
                // once where the transaction lies in one chunk
                const uint32_t k0 = f.key(op0, f.none, false);
                if (tiled && k0 == f.key(op0 + nops[u] - 1, f.none, false)) {
                    keys[op] = ki;
                    if (lig == 0) count_digits(h, k0, f.bits, f.passes, f.digit_bits, (nops[u] - 3) / 2);
                } else {
                    put_key(f, h, keys, op, ki, tiled);
                }
                put_key(f, h, keys, op + 1, ks, tiled);
            }
            if (inside[u] && bad[u])
                for (uint32_t j = lig; j < nops[u]; j += 16) {
                    const uint32_t k = f.key(op0 + j, f.none, false);
                    put_key(f, h, keys, op0 + j, k, tiled);
                }
            if (lig == 0 && tb + u < t_end) {
                a.results[tb + u] = no ? gcc_txn_result{GCC_TXN_INVALID, 0u, ~0ull}
                                       : gcc_txn_result{GCC_TXN_COMMITTED, 1u, tb + u};
                invalid += no;
            }
        }
    }
    if (invalid) {
        atomicAdd(&a.st->invalid, (unsigned long long)invalid);
        atomicOr(&a.st->error, GCC_DEVERR_INVALID);
    }
    flush_digits(f, h, work, a.n_ops, tiled);
}

// --- fold -------------------------------------------------------------------
// What a run of accesses adds to its record: amount (Payment amounts, order
// quantities), count (orders, payments), remote lines; ODD in `r` marks a
// stock run outside the regular ranges.
constexpr uint32_t ODD = 0x80000000u;
struct Add {
    uint64_t a;
    uint32_t n, r;
    // as a tile descriptor: x the amount, y bits 0..29 the count, 30..59 the
    // remote lines, 60 ODD (and the state)
    __device__ __forceinline__ ulonglong2 pack(uint64_t state) const {
        return make_ulonglong2(a, (uint64_t)n | (uint64_t)(r & ~ODD) << 30 | (r & ODD ? 1ull << 60 : 0ull) | state);
    }
    static __device__ __forceinline__ Add unpack(ulonglong2 w) {
        return Add{w.x, (uint32_t)w.y & 0x3fffffffu,
                   ((uint32_t)(w.y >> 30) & 0x3fffffffu) | (w.y >> 60 & 1 ? ODD : 0u)};
    }
    __device__ __forceinline__ Add of_lane_xor(int o) const {
        return Add{__shfl_xor_sync(0xffffffffu, a, o), __shfl_xor_sync(0xffffffffu, n, o),
                   __shfl_xor_sync(0xffffffffu, r, o)};
    }
};
__device__ __forceinline__ Add operator+(Add x, Add y) {
    return Add{x.a + y.a, x.n + y.n, ((x.r + y.r) & ~ODD) | ((x.r | y.r) & ODD)};
}
__device__ __forceinline__ Add shfl_up(Add s, int o) {
    return Add{__shfl_up_sync(0xffffffffu, s.a, o), __shfl_up_sync(0xffffffffu, s.n, o),
               __shfl_up_sync(0xffffffffu, s.r, o)};
}

enum Class { WAREHOUSE, DISTRICT, CUSTOMER, STOCK };

// An access in sorted order: its record's class and row, the columns it reads.
struct Access {
    uint32_t row;
    int cls;
    uint64_t c0, c1;
};
__device__ __forceinline__ Access access(const OeTables& T, uint32_t W, uint32_t rec, bool pay) {
    Access x{rec, WAREHOUSE, 0ull, 0ull};
    if (rec >= 30011u * W) { x.cls = STOCK; x.row = rec - 30011u * W; }
    else if (rec >= 11u * W) { x.cls = CUSTOMER; x.row = rec - 11u * W; }
    else if (rec >= W) { x.cls = DISTRICT; x.row = rec - W; }
    const int i0 = x.cls == STOCK      ? S_QUANTITY
                   : x.cls == CUSTOMER ? (pay ? C_BALANCE : C_DISCOUNT)
                   : x.cls == DISTRICT ? (pay ? D_YTD : D_NEXT_O_ID)
                                       : (pay ? W_YTD : W_TAX);
    x.c0 = T.c[i0][x.row];
    if (x.cls == STOCK) x.c1 = T.c[S_ORDER_CNT][x.row];
    else if (x.cls == CUSTOMER) x.c1 = T.c[pay ? C_PAYMENT_CNT : C_BALANCE][x.row];
    else if (x.cls == DISTRICT && !pay) x.c1 = T.c[D_TAX][x.row];
    return x;
}
// The regular stock quantity after orders of `sum` in all.
__device__ __forceinline__ uint64_t quantity_after(uint64_t q0, uint64_t sum) {
    uint64_t t = q0 - Q_LO + Q_MOD - sum % Q_MOD;
    if (t >= Q_MOD) t -= Q_MOD;
    return t + Q_LO;
}
// The value the access reads, `b` added to its record before it.
__device__ __forceinline__ ulonglong2 value_read(const Access& x, bool pay, Add b) {
    switch (x.cls) {
        case WAREHOUSE: return make_ulonglong2(pay ? x.c0 + b.a : x.c0, 0ull);
        case DISTRICT: return pay ? make_ulonglong2(x.c0 + b.a, 0ull) : make_ulonglong2(x.c0 + b.n, x.c1);
        case CUSTOMER: return pay ? make_ulonglong2(x.c0 - b.a, x.c1 + b.n) : make_ulonglong2(x.c0, x.c1 - b.a);
        default: return make_ulonglong2(quantity_after(x.c0, b.a), x.c1 + b.n);
    }
}
// The record after its last access, `s` added to it in all.
__device__ __forceinline__ void store_record(const OeTables& T, const Access& x, Add s) {
    const uint32_t r = x.row;
    switch (x.cls) {
        case WAREHOUSE:
            if (s.a) T.c[W_YTD][r] += s.a;
            break;
        case DISTRICT:
            if (s.a) T.c[D_YTD][r] += s.a;
            if (s.n) T.c[D_NEXT_O_ID][r] += s.n;
            break;
        case CUSTOMER:
            if (s.n) {
                T.c[C_BALANCE][r] -= s.a;
                T.c[C_YTD_PAYMENT][r] += s.a;
                T.c[C_PAYMENT_CNT][r] += s.n;
            }
            break;
        default:
            T.c[S_QUANTITY][r] = quantity_after(x.c0, s.a);
            T.c[S_YTD][r] += s.a;
            T.c[S_ORDER_CNT][r] = x.c1 + s.n;
            if (s.r) T.c[S_REMOTE_CNT][r] += s.r;
    }
}

// One tile of sorted accesses, as det_fold.cu's fold_tiles: every value of the
// tile's records is read before the block barrier; a record is stored by the
// tile of its last access, after it has acquired the descriptors of the tiles
// its chain runs through.  Bound by the gathers and scatters (operand, two
// columns, value read) out of L2: 2^18 transactions (3.4 M ops) take 90 us at
// one warehouse and 102 us at 64.  (One warp per record, applying 32 ops at a
// time and a stock row's op by op, took 10.1 ms and 0.67 ms: a one-warehouse
// batch was one warp walking its 262,144 warehouse ops.)  An irregular stock run is not stored but
// listed by its last position for oe_in_order, which also rewrites the values
// its accesses read.
__global__ void __launch_bounds__(OF_THREADS)
oe_fold(const __grid_constant__ ExecArgs a, const __grid_constant__ OeTables T, const AccessKeys f,
        const uint32_t* sk, const uint32_t* sv, uint64_t op0, uint32_t c0,
        uint32_t c1, uint32_t* ticket, ulonglong2* desc, uint32_t* n_odd, uint32_t* odd) {
    __shared__ uint32_t s_tile;
    __shared__ Add s_tot[OF_WARPS];
    __shared__ bool s_begins[OF_WARPS];
    __shared__ Add s_carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    after_previous();
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const uint32_t base = c0 + tile * OF_TILE + threadIdx.x * OF_ITEMS;
    uint32_t k[OF_ITEMS], v[OF_ITEMS];
#pragma unroll
    for (int i = 0; i < OF_ITEMS; ++i) {
        k[i] = base + i < c1 ? sk[base + i] : 0u;
        v[i] = base + i < c1 ? sv[base + i] : 0u;
    }
    uint32_t prev = __shfl_up_sync(0xffffffffu, k[OF_ITEMS - 1], 1);
    uint32_t next = __shfl_down_sync(0xffffffffu, k[0], 1);
    if (lane == 0) prev = base > c0 && base < c1 ? sk[base - 1] : 0u;
    if (lane == 31) next = base + OF_ITEMS < c1 ? sk[base + OF_ITEMS] : 0u;
    uint32_t head = 0, live = 0, seen = 0;     // head, live: a bit per item
    Access x[OF_ITEMS];
    Add d[OF_ITEMS];
#pragma unroll
    for (int i = 0; i < OF_ITEMS; ++i) {
        const bool in = base + i < c1 && f.rec(k[i]) < f.none && f.op(op0, v[i]) < a.n_ops;
        live |= in ? 1u << i : 0u;
        if (!in || (i == 0 ? base == c0 || prev != k[0] : k[i - 1] != k[i])) head |= 1u << i;
        d[i] = Add{0, 0, 0};
        x[i] = Access{0u, WAREHOUSE, 0ull, 0ull};
        if (in) x[i] = access(T, a.n_warehouses, f.rec(k[i]), v[i] >> 31);
    }
#pragma unroll
    for (int i = 0; i < OF_ITEMS; ++i) {
        if (!(live >> i & 1)) continue;
        const bool pay = v[i] >> 31;
        if (pay || x[i].cls == STOCK) {
            const ulonglong2 o = a.operands[f.op(op0, v[i])];
            d[i].a = o.x;
            d[i].n = pay && x[i].cls != CUSTOMER ? 0u : 1u;
            if (!pay) {
                d[i].r = o.y ? 1u : 0u;
                if (o.x > (uint64_t)Q_MOD || o.y > 1 || x[i].c0 - Q_LO > (uint64_t)(Q_HI - Q_LO)) d[i].r |= ODD;
            }
        } else if (x[i].cls == DISTRICT) {
            d[i].n = 1;
        }
        seen ^= (uint32_t)x[i].c0 ^ (uint32_t)x[i].c1;
    }
    Add run{0, 0, 0};
    const bool any = head != 0;
#pragma unroll
    for (int i = 0; i < OF_ITEMS; ++i) run = (head >> i & 1) ? d[i] : run + d[i];
    const unsigned heads = __ballot_sync(0xffffffffu, any);
    const unsigned upto = heads & (0xffffffffu >> (31 - lane));
    const int start = upto ? 31 - __clz(upto) : 0;
    Add inc = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Add y = shfl_up(inc, o);
        if (lane - o >= start) inc = y + inc;
    }
    Add carry = shfl_up(inc, 1);
    if (lane == 0) carry = Add{0, 0, 0};
    if (lane == 31) {
        s_tot[warp] = inc;
        s_begins[warp] = heads != 0;
    }
    // the barrier takes a predicate computed from the columns, so every one of
    // them has arrived before any thread passes it
    __syncthreads_or(seen == 0x9E3779B9u);
    const bool runs_in = !(head & 1);
    if (warp == 0) {
        Add tot{0, 0, 0};
        bool begins = false;
#pragma unroll
        for (int w = 0; w < OF_WARPS; ++w) {
            if (s_begins[w]) { tot = Add{0, 0, 0}; begins = true; }
            tot = tot + s_tot[w];
        }
        const bool whole = begins || tile == 0;
        if (lane == 0) st128_release(desc + tile, tot.pack(whole ? WHOLE : TAIL));
        Add before{0, 0, 0};
        if (__shfl_sync(0xffffffffu, runs_in, 0)) {
            before = look_back<Add>(desc, tile, &a.st->error);
            if (!whole && lane == 0) st128_release(desc + tile, (before + tot).pack(WHOLE));
        }
        if (lane == 0) s_carry = before;
    }
    __syncthreads();
    if (!(heads & (0xffffffffu >> (31 - lane)) & ~(1u << lane))) {   // no lane before begins a record
        bool open = true;
        for (int w = warp - 1; w >= 0 && open; --w) {
            carry = s_tot[w] + carry;
            open = !s_begins[w];
        }
        if (open) carry = s_carry + carry;
    }
#pragma unroll
    for (int i = 0; i < OF_ITEMS; ++i) {
        if (head >> i & 1) carry = Add{0, 0, 0};
        if (!(live >> i & 1)) continue;
        a.reads[f.op(op0, v[i])] = value_read(x[i], v[i] >> 31, carry);
        carry = carry + d[i];
        const bool last = base + i + 1 >= c1 || (i + 1 < OF_ITEMS ? k[(i + 1) % OF_ITEMS] : next) != k[i];
        if (!last) continue;
        if (carry.r & ODD) odd[atomicAdd(n_odd, 1u)] = base + i;
        else store_record(T, x[i], carry);
    }
}

// Stock runs the fold could not sum: a warp per run finds its beginning, then
// lane 0 applies the quantity rule op by op, 32 staged at a time.
// Bound by a run's chain of dependent loads, so two blocks per SM: 2^18
// transactions at 64 warehouses with every order outside the range (1.2 M runs)
// take 846 us, 1,234 with one.
__global__ void __launch_bounds__(256)
oe_in_order(const __grid_constant__ ExecArgs a, const __grid_constant__ OeTables T, const AccessKeys f,
            const uint32_t* sk, const uint32_t* sv, uint64_t op0, uint32_t c0,
            uint32_t c1, const uint32_t* n_odd, const uint32_t* odd) {
    __shared__ ulonglong2 s_o[8][32], s_r[8][32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    after_previous();
    const uint32_t n = *n_odd < c1 - c0 ? *n_odd : c1 - c0;
    for (uint32_t j = blockIdx.x * 8 + wib; j < n; j += gridDim.x * 8) {
        const uint32_t end = odd[j];
        if (end < c0 || end >= c1) continue;
        const uint32_t key = sk[end];
        uint32_t at = end;                     // first position known to be of the run
        for (;;) {
            const bool same = (uint64_t)at >= (uint64_t)c0 + lane + 1 && sk[at - lane - 1] == key;
            const unsigned m = __ballot_sync(0xffffffffu, same);
            const int run = m == 0xffffffffu ? 32 : __ffs(~m) - 1;
            at -= run;
            if (run < 32) break;
        }
        const uint32_t row = f.rec(key) - 30011u * a.n_warehouses;
        uint64_t q = 0, cnt = 0, ytd = 0, rem = 0;
        if (lane == 0) {
            q = T.c[S_QUANTITY][row];
            cnt = T.c[S_ORDER_CNT][row];
            ytd = T.c[S_YTD][row];
            rem = T.c[S_REMOTE_CNT][row];
        }
        // the op of position p + lane and its operand, while lane 0 applies the 32 before
        uint64_t op_next = ~0ull;
        ulonglong2 o_next = make_ulonglong2(0ull, 0ull);
        const auto fetch = [&](uint32_t p) {
            op_next = p + lane <= end ? f.op(op0, sv[p + lane]) : ~0ull;
            o_next = op_next < a.n_ops ? a.operands[op_next] : make_ulonglong2(0ull, 0ull);
        };
        fetch(at);
        for (uint32_t p = at; p < end + 1; p += 32) {
            const uint32_t m = end - p + 1 < 32 ? end - p + 1 : 32;
            const uint64_t op = op_next;
            __syncwarp();
            s_o[wib][lane] = o_next;
            __syncwarp();
            fetch(p + 32);
            if (lane == 0)
                for (uint32_t i = 0; i < m; ++i) {
                    const ulonglong2 o = s_o[wib][i];
                    s_r[wib][i] = make_ulonglong2(q, cnt);
                    const int64_t now = (int64_t)q, qty = (int64_t)o.x;
                    q = (uint64_t)(now >= qty + 10 ? now - qty : now - qty + 91);
                    ytd += o.x;
                    cnt += 1;
                    rem += o.y;
                }
            __syncwarp();
            if (op < a.n_ops) a.reads[op] = s_r[wib][lane];
        }
        if (lane == 0) {
            T.c[S_QUANTITY][row] = q;
            T.c[S_ORDER_CNT][row] = cnt;
            T.c[S_YTD][row] = ytd;
            T.c[S_REMOTE_CNT][row] = rem;
        }
    }
}

// --- commit -----------------------------------------------------------------
// The inserts of the valid NewOrders, a half-warp per transaction (lane l
// order line l), two transactions per half-warp at once: the order id is the
// next order id the transaction read, an id outside the order slots sets the
// insert error.  Bound by the latency of the transaction's loads and the
// scattered row stores: 47 us for 2^18 transactions (a warp per transaction, the
// columns' addresses loaded by every store: 113 us).
__global__ void __launch_bounds__(256)
oe_commit(const __grid_constant__ ExecArgs a, const __grid_constant__ OeTables T) {
    constexpr int U = 2;
    const int lig = threadIdx.x & 15;
    const unsigned gmask = 0xffffu << (threadIdx.x & 16);
    after_previous();
    const uint64_t stride = (uint64_t)gridDim.x * 16 * U;
    // the trip count is the warp's, not the half-warp's: it votes below
    for (uint64_t t0 = (uint64_t)blockIdx.x * 16 * U; t0 < a.n_txns; t0 += stride) {
        const uint64_t tb = t0 + (threadIdx.x >> 4) * U;
        bool go[U];
        uint64_t first[U], dist[U], cust[U], item[U], stock[U], price[U];
        uint32_t lines[U];
        ulonglong2 opd[U];
        int64_t o_id[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            gcc_txn tx{0u, 0, 0};
            go[u] = false;
            if (tb + u < a.n_txns) {
                tx = a.txns[tb + u];
                go[u] = tx.type == GCC_TXN_NEW_ORDER && a.results[tb + u].status == GCC_TXN_COMMITTED;
            }
            first[u] = tx.first_op;
            lines[u] = go[u] ? (tx.n_ops - 3u) / 2 : 0u;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool line = lig < (int)lines[u];
            dist[u] = go[u] ? a.ops[first[u] + 1] : 0ull;
            cust[u] = go[u] ? a.ops[first[u] + 2] : 0ull;
            o_id[u] = go[u] ? (int64_t)a.reads[first[u] + 1].x : 0;
            item[u] = line ? a.ops[first[u] + 3 + 2 * lig] : 0ull;
            stock[u] = line ? a.ops[first[u] + 4 + 2 * lig] : 0ull;
            opd[u] = line ? a.operands[first[u] + 4 + 2 * lig] : make_ulonglong2(0ull, 0ull);
            price[u] = line ? a.reads[first[u] + 3 + 2 * lig].x : 0ull;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned remote_lanes = __ballot_sync(0xffffffffu, opd[u].y != 0);
            const bool remote = remote_lanes & gmask;
            const bool fits = o_id[u] >= 1 && (uint64_t)o_id[u] <= a.order_cap;
            if (go[u] && !fits && lig == 0) atomicOr(&a.st->error, GCC_DEVERR_INSERT);
            if (!go[u] || !fits) continue;
            const uint64_t slot = (uint64_t)op_key(dist[u]) * a.order_cap + (uint64_t)(o_id[u] - 1);
            if (lig < (int)lines[u]) {
                const uint64_t ol = slot * LINES + lig;
                T.c[OL_I_ID][ol] = op_key(item[u]);
                T.c[OL_SUPPLY_W_ID][ol] = op_key(stock[u]) / ITEMS;
                T.c[OL_QUANTITY][ol] = opd[u].x;
                T.c[OL_AMOUNT][ol] = opd[u].x * price[u];
            }
            if (lig == 0) {
                T.c[O_C_ID][slot] = op_key(cust[u]) % CUST;
                T.c[O_OL_CNT][slot] = lines[u];
                T.c[O_ALL_LOCAL][slot] = remote ? 0ull : 1ull;
                T.c[NO_FLAG][slot] = 1ull;
            }
        }
    }
}

// `sort_log2` (OE_CHUNK_LOG2 or more): the ops of one sort.
cudaError_t oe_run(const ExecArgs& a, const OeTables& T, SortScratch& s, void* scratch, uint32_t* list,
                   uint32_t& launches, cudaStream_t st, int sort_log2 = OE_SORT_LOG2) {
    const uint64_t n = a.n_ops;
    const AccessKeys f = access_keys(a.n_meta, n, OE_CHUNK_LOG2, sort_log2, true);
    const DetScratch sc = det_scratch(scratch, n, a.n_txns, OE_CHUNK_LOG2, OF_TILE);
    const bool one_sort = n <= (1ull << sort_log2);
    cudaError_t e = launch_det_begin(a, s, sc, f, one_sort, st);
    launches += 1;
    if (e != cudaSuccess || a.n_txns == 0) return e;
    const uint32_t per_block = (uint32_t)blocks_for(blocks_for(a.n_txns, 32), 152 * 6) * 32;
    e = launch_after(oe_validate, blocks_for(a.n_txns, (int)per_block), 256, st, a, T, f, s.k0, s.work,
                     per_block);
    launches += 1;
    for (uint64_t o0 = 0; o0 < n && e == cudaSuccess; o0 += 1ull << sort_log2) {
        const uint32_t m = (uint32_t)std::min<uint64_t>(n - o0, 1ull << sort_log2);
        uint32_t *sk = nullptr, *sv = nullptr;
        e = radix_sort_positions(s, s.k0 + o0, m, f.bits, true, one_sort, &sk, &sv, st);
        launches += f.passes + (one_sort ? 0 : 1);
        for (uint32_t c0 = 0; c0 < m && e == cudaSuccess;) {
            const uint32_t len = std::min<uint32_t>(m - c0, 1u << f.chunk_log2);
            const uint64_t at = o0 + c0;
            uint32_t* n_odd = sc.lengths + (at >> OE_CHUNK_LOG2);
            e = launch_after(oe_fold, blocks_for(len, OF_TILE), OF_THREADS, st, a, T, f, sk, sv, o0, c0,
                             c0 + len, sc.tickets + (at >> OE_CHUNK_LOG2), sc.tile_desc + at / OF_TILE,
                             n_odd, list);
            if (e == cudaSuccess)
                e = launch_after(oe_in_order, std::min<unsigned>(blocks_for(len, 256), 304u), 256, st, a, T,
                                 f, sk, sv, o0, c0, c0 + len, n_odd, list);
            launches += 2;
            c0 += len;
        }
    }
    if (e != cudaSuccess) return e;
    launches += 2;
    e = launch_after(oe_commit, std::min<unsigned>(blocks_for(a.n_txns, 32), 152u * 16u), 256, st, a, T);
    if (e != cudaSuccess) return e;
    return launch_det_finish(a, s, sc, st);
}

}  // namespace

size_t oe_scratch_bytes(size_t max_ops, size_t max_txns) {
    return det_scratch(nullptr, max_ops, max_txns, OE_CHUNK_LOG2, OF_TILE).n_zero * 16;
}

cudaError_t det_serial_oe(const ExecArgs& a, const OeTables& T, SortScratch& s, void* scratch,
                          uint32_t* list, uint32_t& launches, cudaStream_t st) {
    return oe_run(a, T, s, scratch, list, launches, st);
}

}  // namespace gcc
