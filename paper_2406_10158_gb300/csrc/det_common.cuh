// det_common.cuh -- what the deterministic scheme's passes share for key-value
// (det_fold.cu) and order-entry (det_oe.cu) batches: the kernel that starts a
// batch, the segmented look-back between tiles and the kernel that finishes
// it.
#pragma once

#include <algorithm>

#include "engine.cuh"

namespace gcc {
namespace {

// Words of SortScratch::work between the pass tickets and the histograms.
// The first three are left at zero by the kernel that uses them.
enum { DW_BEGIN_DONE = 8, DW_UNTILED_ACC, DW_FILL_TICKET, DW_UNTILED, DW_FINISH_TICKET };

constexpr uint32_t DET_SPIN_MAX = 1u << 21;

inline unsigned blocks_for(uint64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// The sort keys of a batch's accesses: bits 0..rec_bits-1 the record or slot
// (`none`: the op takes no part), above it the op's chunk, bit 31 (`flagged`)
// one bit of the caller's that the sort hands on in the value.
struct AccessKeys {
    uint32_t none;
    int rec_bits, bits, passes, digit_bits, chunk_log2, sort_log2;
    int flagged;
    __device__ uint32_t key(uint64_t op, uint32_t rec, bool flag) const {
        uint32_t k = rec;
        if (bits > rec_bits) k |= ((uint32_t)(op & ((1ull << sort_log2) - 1)) >> chunk_log2) << rec_bits;
        return k | (flagged && flag ? 0x80000000u : 0u);
    }
    __device__ uint32_t rec(uint32_t k) const { return rec_bits == 32 ? k : k & ((1u << rec_bits) - 1u); }
    // the op of a sorted value, positions counting from op0
    __device__ uint64_t op(uint64_t op0, uint32_t v) const { return op0 + (flagged ? v & 0x7fffffffu : v); }
};

inline AccessKeys access_keys(uint64_t none, uint64_t n_ops, int chunk_log2, int sort_log2, bool flag) {
    AccessKeys f;
    f.none = (uint32_t)none;
    f.rec_bits = 0;
    for (uint64_t v = none; v; v >>= 1) ++f.rec_bits;
    const uint64_t m = std::min<uint64_t>(n_ops, 1ull << sort_log2);
    int want = 0;                            // chunk bits
    while (((uint64_t)1 << (chunk_log2 + want)) < m) ++want;
    f.flagged = flag && f.rec_bits <= 31;
    const int chunk_bits = std::min(want, (f.flagged ? 31 : 32) - f.rec_bits);
    f.chunk_log2 = chunk_log2 + (want - chunk_bits);
    f.sort_log2 = sort_log2;
    f.bits = f.rec_bits + chunk_bits;
    const SortPlan sp = sort_plan(f.bits);
    f.passes = sp.passes;
    f.digit_bits = sp.digit_bits;
    return f;
}

// Scratch of a pass, zeroed by det_begin: a ticket and a list length per chunk,
// one word per tile of transactions (det_finish), one descriptor per tile of ops.
struct DetScratch {
    uint32_t *tickets, *lengths;
    unsigned long long* rank_desc;
    ulonglong2* tile_desc;
    ulonglong2* zero;
    size_t n_zero;
};
constexpr uint32_t RANK_TILE = 1024;
inline DetScratch det_scratch(void* base, uint64_t n_ops, uint64_t n_txns, int chunk_log2, int tile) {
    const auto rounded = [](size_t b) { return (b + 255) & ~size_t(255); };
    char* p = static_cast<char*>(base);
    DetScratch s;
    s.zero = reinterpret_cast<ulonglong2*>(p);
    const size_t chunks = rounded(((size_t)(n_ops >> chunk_log2) + 2) * 4);
    s.tickets = reinterpret_cast<uint32_t*>(p);
    p += chunks;
    s.lengths = reinterpret_cast<uint32_t*>(p);
    p += chunks;
    s.rank_desc = reinterpret_cast<unsigned long long*>(p);
    p += rounded((n_txns / RANK_TILE + 1) * 8);
    s.tile_desc = reinterpret_cast<ulonglong2*>(p);
    p += rounded((n_ops / tile + 2) * 16);
    s.n_zero = (size_t)(p - static_cast<char*>(base)) / 16;
    return s;
}

// A block-wide election: true in every thread of the last block to arrive at
// `counter` (which is left at zero), whose accesses then follow every other
// block's.
__device__ __forceinline__ bool last_block(uint32_t* counter) {
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        fence_acq_rel();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
        if (last) *counter = 0;
        fence_acq_rel();
    }
    __syncthreads();
    return last;
}

// Starts a batch: zeroes the batch state, the sort's tickets, histograms and
// first descriptor area (`zero`, `n_zero` 16-byte words, all of SortScratch::work
// but the words above) and the pass's own descriptors (`zero2`), and checks that
// the transactions' op ranges tile ops[0, n_ops) in id order, which the
// contract asks for.  Where they do not, DW_UNTILED is set and the blocks that
// see it give every op the key of no record, a chunk of ops at a time, so that an
// op outside every range stays out of the access table; the validation pass then
// overwrites the others'.  (2^24 ops, every seventh transaction left out: 1,399 us
// for the batch, 2,840 with the last block filling alone; one transaction left
// out, which one block sees: 2,624 us, 3,169 with chunks of 2^13 ops, whose
// tickets it waits for one after the other.)
constexpr uint32_t FILL_CHUNK = 1u << 16;
__global__ void __launch_bounds__(256)
det_begin(const __grid_constant__ ExecArgs a, uint32_t* work, ulonglong2* zero, size_t n_zero,
          ulonglong2* zero2, size_t n_zero2, uint32_t* keys, const AccessKeys f) {
    after_previous();
    const size_t i0 = (size_t)blockIdx.x * 256 + threadIdx.x, stride = (size_t)gridDim.x * 256;
    if (i0 == 0) {
        BatchState z{};
        z.ticket_base = a.dbs->occ_clock;
        *a.st = z;
        for (int w = 0; w < (int)SORT_HIST; ++w)
            if (w < DW_BEGIN_DONE || w > DW_UNTILED) work[w] = 0;
    }
    const ulonglong2 z2 = make_ulonglong2(0ull, 0ull);
    for (size_t i = i0; i < n_zero; i += stride) zero[i] = z2;
    for (size_t i = i0; i < n_zero2; i += stride) zero2[i] = z2;
    bool untiled = false;
    for (size_t t = i0; t < a.n_txns; t += stride) {
        const gcc_txn x = a.txns[t];
        uint64_t before = 0;
        if (t) {
            const gcc_txn y = a.txns[t - 1];
            before = (uint64_t)y.first_op + y.n_ops;
        }
        if (x.first_op != before) untiled = true;
        if (t + 1 == a.n_txns && (uint64_t)x.first_op + x.n_ops != a.n_ops) untiled = true;
    }
    if (__syncthreads_or(untiled)) {
        __shared__ uint32_t s_chunk;
        const uint64_t chunks = (a.n_ops + FILL_CHUNK - 1) / FILL_CHUNK;
        for (;;) {
            if (threadIdx.x == 0) s_chunk = atomicAdd(work + DW_FILL_TICKET, 1u);
            __syncthreads();
            const uint64_t o0 = (uint64_t)s_chunk * FILL_CHUNK;
            if (s_chunk >= chunks) break;
            const uint32_t k = f.key(o0, f.none, false);       // one for the whole chunk
            const uint32_t m = (uint32_t)(a.n_ops - o0 < FILL_CHUNK ? a.n_ops - o0 : FILL_CHUNK);
            for (uint32_t i = threadIdx.x * 4; i + 4 <= m; i += 1024)
                *reinterpret_cast<uint4*>(keys + o0 + i) = make_uint4(k, k, k, k);
            if (threadIdx.x < m % 4) keys[o0 + m / 4 * 4 + threadIdx.x] = k;
            __syncthreads();
        }
        if (threadIdx.x == 0) atomicOr(work + DW_UNTILED_ACC, 1u);
    }
    if (!last_block(work + DW_BEGIN_DONE)) return;
    const uint32_t bad = *(volatile uint32_t*)(work + DW_UNTILED_ACC);
    __syncthreads();
    if (threadIdx.x == 0) {
        work[DW_UNTILED] = bad;
        work[DW_UNTILED_ACC] = 0;
        work[DW_FILL_TICKET] = 0;
    }
}

// Launches det_begin; with one sort for the whole batch (`one_sort`) it also
// prepares that sort's tickets, histograms and descriptors.
inline cudaError_t launch_det_begin(const ExecArgs& a, SortScratch& s, const DetScratch& sc,
                                    const AccessKeys& f, bool one_sort, cudaStream_t st) {
    const size_t n_zero = one_sort ? (SORT_DESC - SORT_HIST + sort_desc_words(a.n_ops)) / 4 : 0;
    const uint64_t most = std::max<uint64_t>(std::max<uint64_t>(n_zero, sc.n_zero), a.n_txns);
    const unsigned grid = std::min<unsigned>(std::max<unsigned>(blocks_for(most, 256), 1u), 608u);
    return launch_after(det_begin, grid, 256, st, a, s.work,
                        reinterpret_cast<ulonglong2*>(s.work + SORT_HIST), n_zero, sc.zero, sc.n_zero,
                        s.k0, f);
}

// The block's digit histograms: HIST_COPIES copies side by side, a lane adding
// to the copy of its own number, so that lanes of a warp with the same digit
// (the top digits of neighbouring ops often are) rarely meet on one word.
constexpr int HIST_COPIES = 4;
typedef uint32_t DigitHist[256 * HIST_COPIES];
__device__ __forceinline__ void count_digits(DigitHist* h, uint32_t k, int bits, int passes, int digit_bits,
                                             uint32_t times = 1u) {
    const uint32_t copy = threadIdx.x % HIST_COPIES;
#pragma unroll
    for (int p = 0; p < SORT_MAX_PASSES; ++p)
        if (p < passes) {
            const int left = bits - p * digit_bits;
            const uint32_t mask = (1u << (left < digit_bits ? left : digit_bits)) - 1u;
            atomicAdd(&h[p][((k >> (p * digit_bits)) & mask) * HIST_COPIES + copy], times);
        }
}
__device__ __forceinline__ void clear_digits(DigitHist* h) {
#pragma unroll
    for (int p = 0; p < SORT_MAX_PASSES; ++p)
        for (int c = threadIdx.x; c < 256 * HIST_COPIES; c += 256) h[p][c] = 0;
}

// Writes an op's key and counts it.  Where the op ranges do not tile the ops
// (DW_UNTILED) every op holds the key of no record already (det_begin), and may
// be written by more than one transaction: the exchange tells which key the new
// one replaces, so the counts stay those of the keys.
__device__ __forceinline__ void put_key(const AccessKeys& f, DigitHist* h, uint32_t* keys, uint64_t op, uint32_t k,
                                        bool tiled) {
    if (tiled) {
        keys[op] = k;
    } else {
        const uint32_t old = atomicExch(keys + op, k);
        count_digits(h, old, f.bits, f.passes, f.digit_bits, ~0u);
    }
    count_digits(h, k, f.bits, f.passes, f.digit_bits);
}

// The block's histograms into the batch's; where the op ranges do not tile the
// ops, block 0 also counts the keys det_begin wrote.  Every block calls it.
__device__ __forceinline__ void flush_digits(const AccessKeys& f, DigitHist* h, uint32_t* work, uint64_t n,
                                             bool tiled) {
    __syncthreads();
    if (!tiled && blockIdx.x == 0) {
        const uint64_t len = 1ull << f.chunk_log2;
        for (uint64_t o = threadIdx.x * len; o < n; o += 256 * len)
            count_digits(h, f.key(o, f.none, false), f.bits, f.passes, f.digit_bits,
                         (uint32_t)(n - o < len ? n - o : len));
        __syncthreads();
    }
    for (int p = 0; p < f.passes; ++p) {
        uint32_t c = 0;
#pragma unroll
        for (int i = 0; i < HIST_COPIES; ++i) c += h[p][threadIdx.x * HIST_COPIES + i];
        if (c) atomicAdd(work + SORT_HIST + p * 256 + threadIdx.x, c);
    }
}

// --- sums across tiles --------------------------------------------------------
// A tile of sorted accesses publishes one 16-byte descriptor: its sum S and in
// bits 62..63 of the second word its state.  TAIL: no slot's accesses begin in
// the tile, the sum is the whole tile's and what comes before adds to it.
// WHOLE: the sum from the beginning of the slot whose accesses run on past the
// tile.
constexpr uint64_t TAIL = 1ull << 62, WHOLE = 2ull << 62;

// The sum of the accesses before `tile` to the slot that runs into it, by the
// lanes of one warp, 32 predecessors at a time (usually one: nearly every tile
// begins some slot).  Acquire loads: the caller may write that slot only after
// every tile it runs through has read its initial value.  Every lane's acquires
// come before whatever any lane of the warp does next -- lane 0 publishes the
// tile's own WHOLE, which a later tile takes as word of all tiles before --
// and shuffles order no memory, so the warp meets at a barrier at the end.
template <class S>
__device__ __forceinline__ S look_back(const ulonglong2* desc, int64_t tile, unsigned* err) {
    const int lane = threadIdx.x & 31;
    S sum{};
    uint32_t spins = 0;
    for (int64_t p = tile - 1; p >= 0;) {
        ulonglong2 w = make_ulonglong2(0ull, WHOLE);
        if (p - lane >= 0) w = ld128_acquire(desc + (p - lane));
        const unsigned whole = __ballot_sync(0xffffffffu, w.y >= WHOLE);
        const unsigned none = __ballot_sync(0xffffffffu, w.y == 0);
        const int upto = whole ? __ffs(whole) - 1 : 31;             // last lane that counts
        const unsigned need = upto == 31 ? 0xffffffffu : (2u << upto) - 1u;
        if (none & need) {
            if (++spins > DET_SPIN_MAX) {
                if (lane == 0) atomicOr(err, GCC_DEVERR_WAIT_BUDGET);
                break;
            }
            continue;
        }
        S x = lane <= upto ? S::unpack(w) : S{};
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x = x + x.of_lane_xor(o);
        sum = sum + x;
        if (whole) break;
        p -= 32;
    }
    __syncwarp();
    return sum;
}

// Ends a batch: counts the commits.  The validation pass gave every valid
// transaction its id as its commit order, which is right when every
// transaction is valid; otherwise the order is the rank among the valid ones,
// by one scan over tiles of transactions with look-back (rank_desc: one zeroed
// word per tile of 1024).
__global__ void __launch_bounds__(1024)
det_finish(const __grid_constant__ ExecArgs a, uint32_t* work, unsigned long long* rank_desc) {
    __shared__ uint32_t s_tile, s_warp[32], s_before;
    constexpr unsigned long long OWN = 1ull << 62, UP_TO = 2ull << 62, MASK = (1ull << 62) - 1;
    after_previous();
    const unsigned long long invalid = *(volatile unsigned long long*)&a.st->invalid;
    if (invalid == 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            a.st->committed = a.n_txns;
            a.st->max_attempts = a.n_txns ? 1ull : 0ull;
        }
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.st->committed = a.n_txns - invalid;
        a.st->max_attempts = a.n_txns > invalid ? 1ull : 0ull;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_tile = atomicAdd(work + DW_FINISH_TICKET, 1u);
        __syncthreads();
        const uint32_t tile = s_tile;
        const uint64_t t = (uint64_t)tile * RANK_TILE + threadIdx.x;
        if ((uint64_t)tile * RANK_TILE >= a.n_txns) return;
        const bool ok = t < a.n_txns && a.results[t].status == GCC_TXN_COMMITTED;
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        if (lane == 0) s_warp[warp] = __popc(m);
        __syncthreads();
        if (warp == 0) {
            uint32_t x = s_warp[lane], inc = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            s_warp[lane] = inc - x;
            if (lane == 31) {
                unsigned long long* d = rank_desc;
                st_relaxed((uint64_t*)(d + tile), (tile ? OWN : UP_TO) | inc);
                unsigned long long before = 0;
                uint32_t spins = 0;
                for (int64_t p = (int64_t)tile - 1; p >= 0;) {
                    const unsigned long long w = ld_relaxed((const uint64_t*)(d + p));
                    if (w == 0) {
                        if (++spins > DET_SPIN_MAX) {
                            atomicOr(&a.st->error, GCC_DEVERR_WAIT_BUDGET);
                            break;
                        }
                        continue;
                    }
                    before += w & MASK;
                    if (w >= UP_TO) break;
                    --p;
                }
                if (tile) st_relaxed((uint64_t*)(d + tile), UP_TO | (before + inc));
                s_before = (uint32_t)before;
            }
        }
        __syncthreads();
        if (ok) a.results[t].commit_order = s_before + s_warp[warp] + __popc(m & lanemask_lt());
    }
}

inline cudaError_t launch_det_finish(const ExecArgs& a, SortScratch& s, const DetScratch& sc, cudaStream_t st) {
    return launch_after(det_finish, std::min<unsigned>(blocks_for(a.n_txns, RANK_TILE), 152u), 1024, st, a,
                        s.work, sc.rank_desc);
}

}  // namespace
}  // namespace gcc
