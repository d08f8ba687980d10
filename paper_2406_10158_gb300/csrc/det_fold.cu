// det_fold.cu -- the deterministic scheme on key-value batches, by prefix sums.
//
// The deterministic scheme's outcome is the serial execution of the batch in
// transaction-id order (Sec. II-C; Sec. III-E.3 builds the access table the
// same way: (transaction, record) pairs sorted by record).  On a key-value
// batch every op is a READ or an ADD, and ADD is associative and commutative
// (modulo 2^64 on lane 0, modulo 2^16 on bytes 8-9).  So along one slot's
// accesses in transaction-id order, the value an op reads is the slot's
// initial value plus the exclusive prefix sum of the earlier ADD deltas, and
// the final value adds all of them.  This evaluates every record's dependency
// chain with one segmented prefix sum instead of handing the record from op
// to op, which removes the chain latency that dominates under contention.
//
//   begin      batch state, descriptors and histograms zeroed (9 us for 2^24 ops)
//   validate   a lane group per transaction: the same checks as the execute
//              kernel (kinds, keys, fields, distinct keys); every op's access
//              key, and the digit histograms of the sort
//   sort       stable radix sort by (chunk, slot), slot = field * n_records +
//              key: within a chunk, (slot, transaction id) order
//   fold       per chunk, one kernel: segmented prefix sum of the deltas with
//              look-back between tiles, read values out, final values in
//   finish     commit counts; commit order where a transaction was invalid
//
// Chunks.  Serial execution in id order can be cut anywhere: the ops are folded
// in chunks of consecutive positions, each starting from the table the one
// before left.  A chunk's operands are gathered and its read values scattered
// at random (sorted order against op order); cutting keeps the two within L2
// (2^CHUNK_LOG2 ops: 16 MB each), where a batch of 2^24 ops at once would go
// to DRAM sector by sector.  Table accesses pay for it: a chunk touches the
// table more sparsely.  2^24 ops over 2.5 GiB take 1,518 us in chunks of 2^21
// and 1,635 us in chunks of 2^22; 64 databases at once take 6.58 ms in chunks
// of 2^20, 6.85 of 2^21 and 7.17 of 2^22.  The chunk number sorts in the key's
// spare high bits (so few of them may make the chunks larger), and the whole
// batch still takes one sort.
#include "det_common.cuh"

namespace gcc {
namespace {

constexpr int FT_THREADS = 256;
// Accesses per thread of fold_tiles.  16-byte slots hold twice the registers;
// 2 per thread keep 4 blocks on an SM (2^24 ops: 1.52 ms for the batch against
// 1.59 ms with 4), 8-byte slots run 4 (64 databases: 8.1 against 8.3 ms).
template <int FB> constexpr int FT_ITEMS = FB == 16 ? 2 : 4;
template <int FB> constexpr int FT_TILE = FT_THREADS * FT_ITEMS<FB>;
constexpr int FT_WARPS = FT_THREADS / 32;
constexpr int CHUNK_LOG2 = 20;
// One sort handles at most 2^30 ops (30-bit digit counts, 31-bit positions);
// longer batches are sorted and folded in that many at a time.
constexpr int SORT_LOG2 = 30;

__device__ __forceinline__ uint32_t d_key(uint64_t d) { return (uint32_t)d; }
__device__ __forceinline__ uint32_t d_field(uint64_t d) { return (uint32_t)(d >> 32) & 0xffu; }
__device__ __forceinline__ uint32_t d_kind(uint64_t d) { return (uint32_t)(d >> 40) & 0xffu; }

// A running sum in the slot's lane arithmetic.
struct Sum {
    uint64_t lo;
    uint32_t hi;           // modulo 2^16
    // as a tile descriptor: x lane 0, y bits 0..15 bytes 8-9 (and the state)
    __device__ __forceinline__ ulonglong2 pack(uint64_t state) const { return make_ulonglong2(lo, hi | state); }
    static __device__ __forceinline__ Sum unpack(ulonglong2 w) { return Sum{w.x, (uint32_t)w.y & 0xFFFFu}; }
    __device__ __forceinline__ Sum of_lane_xor(int o) const {
        return Sum{__shfl_xor_sync(0xffffffffu, lo, o), __shfl_xor_sync(0xffffffffu, hi, o)};
    }
};
__device__ __forceinline__ Sum operator+(Sum a, Sum b) { return Sum{a.lo + b.lo, (a.hi + b.hi) & 0xFFFFu}; }

// --- validation and access table ---------------------------------------------
// A lane group of G lanes per transaction (G the smallest of 8, 16, 32 that
// holds max_ops; above 32 ops a lane takes two), U consecutive transactions
// per group at once so that their headers and descriptors load together.
// Every block takes one contiguous range of transactions.  Bound by the
// shared-memory histogram updates (one per op and pass): 2^20 transactions of
// 16 ops take about 150 us, of which the stream of descriptors in and keys out would
// take 35; a warp per transaction with every pair of keys compared took 256
// without the histograms, and the sort's own histogram kernels 345 more.
// Equal keys: groups of 8 and 16 lanes compare by rotation (the batch 1,520 ->
// 1,459 us against __match_any_sync, which finds one distinct key at a time);
// for 32 lanes the 16 rotations take too many registers (64 databases of up to
// 64 ops: 6,900 us against 6,573), and 4 blocks on an SM hide the match's
// latency better than 3 (6,573 against 6,795; 5 spill, 6,606).
template <int G>
__global__ void __launch_bounds__(256, G == 32 ? 4 : 1)
fold_validate(const __grid_constant__ ExecArgs a, const AccessKeys f, uint32_t* keys,
              uint32_t* work, uint32_t per_block) {
    constexpr int GROUPS = 256 / G, U = G == 32 ? 2 : 4;
    __shared__ DigitHist h[SORT_MAX_PASSES];
    const int lane = threadIdx.x & 31, lig = lane & (G - 1), gbase = lane & ~(G - 1);
    const uint32_t group = threadIdx.x / G;
    const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << gbase;
    clear_digits(h);
    after_previous();
    __syncthreads();
    const bool tiled = work[DW_UNTILED] == 0;
    uint64_t t_end = (uint64_t)(blockIdx.x + 1) * per_block;
    if (t_end > a.n_txns) t_end = a.n_txns;
    unsigned invalid = 0;
    for (uint64_t t0 = (uint64_t)blockIdx.x * per_block; t0 < t_end; t0 += GROUPS * U) {
        const uint64_t tb = t0 + group * U;
        uint32_t first[U], nops[U];
        uint64_t d[U];
        bool bad[U], inside[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            gcc_txn tx{0u, 0, (uint16_t)GCC_TXN_KV};
            if (tb + u < t_end) tx = a.txns[tb + u];
            first[u] = tx.first_op;
            nops[u] = tx.n_ops;
            inside[u] = tb + u < t_end && (uint64_t)tx.first_op + tx.n_ops <= a.n_ops;
            bad[u] = tx.n_ops > a.max_ops || tx.n_ops > 64 || tx.type != GCC_TXN_KV || !inside[u];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            d[u] = !bad[u] && lig < nops[u] ? a.ops[(uint64_t)first[u] + lig] : 0ull;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool has = !bad[u] && lig < nops[u];
            bool wrong = false;
            if (has)
                wrong = d_key(d[u]) >= a.n_records || d_field(d[u]) >= a.n_fields ||
                        (d_kind(d[u]) != GCC_OP_READ && d_kind(d[u]) != GCC_OP_ADD);
            // equal keys among the group's lanes
            const unsigned holders = __ballot_sync(0xffffffffu, has);
            if constexpr (G <= 16) {
                // every two lanes of the group meet in one of G / 2 rotations
#pragma unroll
                for (int o = 1; o <= G / 2; ++o) {
                    const int other = gbase | ((lig + o) & (G - 1));
                    const uint32_t k = __shfl_sync(0xffffffffu, d_key(d[u]), other);
                    if (has && (holders >> other & 1u) && k == d_key(d[u])) wrong = true;
                }
            } else {
                const unsigned peers = __match_any_sync(0xffffffffu, d_key(d[u]));
                if (has && __popc(peers & holders) > 1) wrong = true;
            }
            uint64_t d2 = 0;
            if constexpr (G == 32) {
                if (!bad[u] && nops[u] > 32) {           // uniform over the warp
                    const bool has2 = lig + 32 < nops[u];
                    if (has2) {
                        d2 = a.ops[(uint64_t)first[u] + 32 + lig];
                        wrong = wrong || d_key(d2) >= a.n_records || d_field(d2) >= a.n_fields ||
                                (d_kind(d2) != GCC_OP_READ && d_kind(d2) != GCC_OP_ADD);
                    }
                    const unsigned h2 = __ballot_sync(0xffffffffu, has2);
                    const unsigned p2 = __match_any_sync(0xffffffffu, d_key(d2));
                    if (has2 && __popc(p2 & h2) > 1) wrong = true;
                    for (int i = 0; i < 32; ++i) {
                        const uint32_t k = __shfl_sync(0xffffffffu, d_key(d[u]), i);
                        if (has2 && k == d_key(d2)) wrong = true;
                    }
                }
            }
            const unsigned any = __ballot_sync(0xffffffffu, wrong);
            const bool no = bad[u] || (any & gmask);
            if (has) {
                const uint64_t op = (uint64_t)first[u] + lig;
                const uint32_t k = f.key(op, no ? f.none : d_field(d[u]) * (uint32_t)a.n_records + d_key(d[u]),
                                         !no && d_kind(d[u]) == GCC_OP_ADD);
                put_key(f, h, keys, op, k, tiled);
            }
            // the ops past the first G of a long or malformed transaction
            if (inside[u] && (bad[u] || nops[u] > G)) {
                for (uint32_t j = (bad[u] ? 0u : (uint32_t)G) + lig; j < nops[u]; j += G) {
                    const uint64_t op = (uint64_t)first[u] + j;
                    const uint32_t k = f.key(op, no ? f.none : d_field(d2) * (uint32_t)a.n_records + d_key(d2),
                                             !no && d_kind(d2) == GCC_OP_ADD);
                    put_key(f, h, keys, op, k, tiled);
                }
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
// A slot's line is not read again soon: 64 of its 128 bytes are fetched (2^24
// ops: 1,542 -> 1,518 us; not keeping it in L1 or marking it to leave L2 first
// were slower, 1,598 us).
template <int FB>
__device__ __forceinline__ ulonglong2 slot_load(const ExecArgs& a, uint32_t slot) {
    const uint8_t* p = a.table + (uint64_t)slot * FB;
    ulonglong2 v = make_ulonglong2(0ull, 0ull);
    if (FB == 16) asm volatile("ld.global.L2::64B.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
    else asm volatile("ld.global.L2::64B.u64 %0, [%1];" : "=l"(v.x) : "l"(p));
    return v;
}
template <int FB>
__device__ __forceinline__ ulonglong2 slot_plus(ulonglong2 v, Sum s) {
    if (FB == 16) return make_ulonglong2(v.x + s.lo, (v.y & ~0xFFFFull) | ((v.y + s.hi) & 0xFFFFull));
    return make_ulonglong2(v.x + s.lo, 0ull);
}

// One tile of sorted accesses: an access reads its slot's initial value
// plus the sum of the deltas before it, the last access of a slot stores the
// final value.  Within the tile every initial value is read before the block
// barrier and stored after it; a slot that runs through several tiles is stored
// by the last of them, after it has acquired the descriptors of the others,
// which they publish (release) behind that barrier.
// Bound by the table's random DRAM accesses (a load and, for a changed slot,
// a write-back each; a kernel that does nothing else makes 39 G a second of
// either): 2^21 ops over 2.5 GiB take 84 us.  One kernel instead of three (tile
// totals, tile scan, apply, and a fourth for slots that cross tiles) removes a
// 16-byte delta per op written and read back; the four took 1.46 ms for 2^24
// ops, the eight launches of this one 0.67 ms.
template <int FB>
__global__ void __launch_bounds__(FT_THREADS, 4)
fold_tiles(const __grid_constant__ ExecArgs a, const AccessKeys f, const uint32_t* sk,
           const uint32_t* sv, uint64_t op0, uint32_t c0, uint32_t c1,
           uint32_t* ticket, ulonglong2* desc) {
    constexpr int ITEMS = FT_ITEMS<FB>;
    __shared__ uint32_t s_tile;
    __shared__ uint64_t s_lo[FT_WARPS];
    __shared__ uint32_t s_hi[FT_WARPS];        // bit 31: the warp begins a slot
    __shared__ Sum s_carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    after_previous();
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const uint32_t base = c0 + tile * FT_TILE<FB> + threadIdx.x * ITEMS;
    uint32_t k[ITEMS], v[ITEMS];
    if (base + ITEMS <= c1) {
        if constexpr (ITEMS == 4) {
            const uint4 x = *reinterpret_cast<const uint4*>(sk + base);
            const uint4 y = *reinterpret_cast<const uint4*>(sv + base);
            k[0] = x.x; k[1] = x.y; k[2] = x.z; k[3] = x.w;
            v[0] = y.x; v[1] = y.y; v[2] = y.z; v[3] = y.w;
        } else {
            const uint2 x = *reinterpret_cast<const uint2*>(sk + base);
            const uint2 y = *reinterpret_cast<const uint2*>(sv + base);
            k[0] = x.x; k[1] = x.y;
            v[0] = y.x; v[1] = y.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            k[i] = base + i < c1 ? sk[base + i] : 0u;
            v[i] = base + i < c1 ? sv[base + i] : 0u;
        }
    }
    // the keys around the thread's own
    uint32_t prev = __shfl_up_sync(0xffffffffu, k[ITEMS - 1], 1);
    uint32_t next = __shfl_down_sync(0xffffffffu, k[0], 1);
    if (lane == 0) prev = base > c0 && base < c1 ? sk[base - 1] : 0u;
    if (lane == 31) next = base + ITEMS < c1 ? sk[base + ITEMS] : 0u;
    uint32_t head = 0, live = 0;               // bit per item
    ulonglong2 init[ITEMS];
    Sum dl[ITEMS];
    uint32_t seen = 0;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const bool in = base + i < c1 && f.rec(k[i]) < f.none && f.op(op0, v[i]) < a.n_ops;
        live |= in ? 1u << i : 0u;
        if (!in || (i == 0 ? base == c0 || prev != k[0] : k[i - 1] != k[i])) head |= 1u << i;
        dl[i] = Sum{0, 0};
        init[i] = make_ulonglong2(0ull, 0ull);
        if (in) init[i] = slot_load<FB>(a, f.rec(k[i]));
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
        if ((live >> i & 1) && (f.flagged ? v[i] >> 31 : d_kind(a.ops[f.op(op0, v[i])]) == GCC_OP_ADD)) {
            const ulonglong2 o = a.operands[f.op(op0, v[i])];
            dl[i] = Sum{o.x, FB == 16 ? (uint32_t)o.y & 0xFFFFu : 0u};
        }
    // within the thread
    Sum run{0, 0};
    const bool any = head != 0;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        if (head >> i & 1) run = Sum{0, 0};
        run = run + dl[i];
        seen ^= (uint32_t)init[i].x;
    }
    // within the warp: inclusive sums since the last lane that begins a slot
    const unsigned heads = __ballot_sync(0xffffffffu, any);
    const unsigned upto = heads & (0xffffffffu >> (31 - lane));
    const int start = upto ? 31 - __clz(upto) : 0;
    Sum inc = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t lo = __shfl_up_sync(0xffffffffu, inc.lo, o);
        const uint32_t hi = FB == 16 ? __shfl_up_sync(0xffffffffu, inc.hi, o) : 0u;
        if (lane - o >= start) inc = inc + Sum{lo, hi};
    }
    Sum carry;                                 // what precedes the thread, in the warp
    carry.lo = __shfl_up_sync(0xffffffffu, inc.lo, 1);
    carry.hi = FB == 16 ? __shfl_up_sync(0xffffffffu, inc.hi, 1) : 0u;
    if (lane == 0) carry = Sum{0, 0};
    if (lane == 31) {
        s_lo[warp] = inc.lo;
        s_hi[warp] = inc.hi | (heads ? 0x80000000u : 0u);
    }
    // the barrier takes a predicate computed from the initial values, so every
    // one of this tile has arrived before any thread passes it
    __syncthreads_or(seen == 0x9E3779B9u);
    const bool runs_in = !(head & 1);          // thread 0: the tile continues a slot
    if (warp == 0) {
        Sum tot{0, 0};
        bool begins = false;
#pragma unroll
        for (int w = 0; w < FT_WARPS; ++w) {
            if (s_hi[w] >> 31) { tot = Sum{0, 0}; begins = true; }
            tot = tot + Sum{s_lo[w], s_hi[w] & 0xFFFFu};
        }
        const bool whole = begins || tile == 0;
        if (lane == 0) st128_release(desc + tile, tot.pack(whole ? WHOLE : TAIL));
        Sum before{0, 0};
        if (__shfl_sync(0xffffffffu, runs_in, 0)) {
            before = look_back<Sum>(desc, tile, &a.st->error);
            if (!whole && lane == 0) st128_release(desc + tile, (before + tot).pack(WHOLE));
        }
        if (lane == 0) s_carry = before;
    }
    __syncthreads();
    if (!(heads & (0xffffffffu >> (31 - lane)) & ~(1u << lane))) {   // no lane before begins a slot
        bool open = true;
        for (int w = warp - 1; w >= 0 && open; --w) {
            carry = carry + Sum{s_lo[w], s_hi[w] & 0xFFFFu};
            open = !(s_hi[w] >> 31);
        }
        if (open) carry = carry + s_carry;
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        if (head >> i & 1) carry = Sum{0, 0};
        if (!(live >> i & 1)) continue;
        a.reads[f.op(op0, v[i])] = slot_plus<FB>(init[i], carry);
        carry = carry + dl[i];
        const bool last = base + i + 1 >= c1 || (i + 1 < ITEMS ? k[(i + 1) % ITEMS] : next) != k[i];
        if (last && (carry.lo | carry.hi)) {                     // unchanged slots are not stored
            const ulonglong2 fin = slot_plus<FB>(init[i], carry);
            uint8_t* dst = a.table + (uint64_t)f.rec(k[i]) * FB;
            if (FB == 16) *reinterpret_cast<ulonglong2*>(dst) = fin;
            else *reinterpret_cast<uint64_t*>(dst) = fin.x;
        }
    }
}

// `sort_log2` (CHUNK_LOG2 or more): the ops of one sort.
template <int FB>
cudaError_t fold_run(const ExecArgs& a, SortScratch& s, void* scratch, uint32_t& launches, cudaStream_t st,
                     int sort_log2 = SORT_LOG2) {
    const uint64_t n = a.n_ops;
    const AccessKeys f = access_keys((uint64_t)a.n_fields * a.n_records, n, CHUNK_LOG2, sort_log2, true);
    const DetScratch sc = det_scratch(scratch, n, a.n_txns, CHUNK_LOG2, FT_TILE<16>);
    const bool one_sort = n <= (1ull << sort_log2);
    cudaError_t e = launch_det_begin(a, s, sc, f, one_sort, st);
    launches += 1;
    if (e != cudaSuccess || a.n_txns == 0) return e;
    const int G = a.max_ops <= 8 ? 8 : a.max_ops <= 16 ? 16 : 32;
    const uint32_t step = G == 8 ? 128 : G == 16 ? 64 : 16;
    const uint32_t steps = blocks_for(a.n_txns, (int)step);
    const uint32_t per_block = (uint32_t)blocks_for(steps, 152 * 6) * step;
    const unsigned grid1 = blocks_for(a.n_txns, (int)per_block);
    auto validate = G == 8 ? fold_validate<8> : G == 16 ? fold_validate<16> : fold_validate<32>;
    e = launch_after(validate, grid1, 256, st, a, f, s.k0, s.work, per_block);
    launches += 1;
    for (uint64_t o0 = 0; o0 < n && e == cudaSuccess; o0 += 1ull << sort_log2) {
        const uint32_t m = (uint32_t)std::min<uint64_t>(n - o0, 1ull << sort_log2);
        uint32_t *sk = nullptr, *sv = nullptr;
        e = radix_sort_positions(s, s.k0 + o0, m, f.bits, f.flagged != 0, one_sort, &sk, &sv, st);
        launches += f.passes + (one_sort ? 0 : 1);
        for (uint32_t c0 = 0; c0 < m && e == cudaSuccess;) {
            const uint32_t len = f.chunk_log2 >= 31 ? m : std::min<uint32_t>(m - c0, 1u << f.chunk_log2);
            const uint64_t at = o0 + c0;
            e = launch_after(fold_tiles<FB>, blocks_for(len, FT_TILE<FB>), FT_THREADS, st, a, f, sk, sv, o0, c0,
                             c0 + len, sc.tickets + (at >> CHUNK_LOG2), sc.tile_desc + at / FT_TILE<FB>);
            launches += 1;
            c0 += len;
        }
    }
    if (e != cudaSuccess) return e;
    launches += 1;
    return launch_det_finish(a, s, sc, st);
}

}  // namespace

// (the version store of an MVCC batch shares this scratch: one 16-byte value per op)
size_t fold_seg_bytes(size_t max_ops, size_t max_txns) {
    return std::max<size_t>(max_ops * 16, det_scratch(nullptr, max_ops, max_txns, CHUNK_LOG2, FT_TILE<16>).n_zero * 16);
}

cudaError_t det_fold_kv(const ExecArgs& a, uint32_t field_bytes, SortScratch& s, void* scratch,
                        uint32_t& launches, cudaStream_t st) {
    return field_bytes == 16 ? fold_run<16>(a, s, scratch, launches, st)
                             : fold_run<8>(a, s, scratch, launches, st);
}

}  // namespace gcc
