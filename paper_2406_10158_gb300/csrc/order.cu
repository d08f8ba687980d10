// order.cu -- ordering kernels: radix sort, prefix sum, the deterministic
// scheme's access table, and dense commit ranks.
//
// The deterministic scheme's preprocessing follows Sec. III-E.3: gather the
// (transaction, record) pairs of the batch into an access table, sort it by
// record, and find each record's boundaries with a prefix sum.  Because the
// ops array is in transaction-id order, a stable sort by record alone yields
// (record, transaction id) order.  Each op then gets a wait threshold:
//   writer at sorted position p     -> all ops before it on the record done
//                                      (record's op counter >= p)
//   reader at sorted position p     -> all writes before it on the record done
//                                      (record's write counter >= W[p], W the
//                                      exclusive prefix count of writes)
// and every record's counter word starts at (first position, W[first]).
// This is the dataflow form of executing the conflict graph rank by rank
// (Sec. II-C): an op runs as soon as its conflicting predecessors have run.
#include "engine.cuh"

namespace gcc {
namespace {

constexpr int RS_BLOCK = SORT_BLOCK;
constexpr int RS_WARPS = RS_BLOCK / 32;

__device__ __forceinline__ unsigned lt_mask() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Exclusive scan of one value per thread over a block of 32*NW threads.
template <int NW>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* warp_sums,
                                                         uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t s = lane < NW ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < NW) warp_sums[lane] = s;
    }
    __syncthreads();
    const uint32_t before = (warp ? warp_sums[warp - 1] : 0) + x - v;
    if (total) *total = warp_sums[NW - 1];
    __syncthreads();
    return before;
}

// --- radix sort --------------------------------------------------------------
// One kernel per pass.  The digit histograms of every pass are taken up front
// in one read of the keys, so a pass knows where each digit's run starts; what
// a tile still needs is the number of each digit's items in the tiles before
// it, which it gets by looking back: every tile publishes its own counts at
// once, sums its predecessors' published words (each either a tile's own
// count or, once that tile has looked back itself, the count of everything up
// to it) and publishes its inclusive count.  Against a histogram kernel, a scan
// kernel and a scatter kernel per pass this reads the keys once per pass instead
// of twice and needs one launch instead of three.
//
// Tiles are numbered by a ticket, so a tile's predecessors are always running
// or done and the wait ends; it is bounded all the same (SPIN_MAX).  A tile
// that gave up sets GCC_DEVERR_WAIT_BUDGET and scatters in bounds, but its
// output positions overlap others': what they leave out holds words of an
// earlier use of the buffer, so whoever reads a sorted pair checks it against
// the array it indexes.
template <class W> struct Count {
    static constexpr int BITS = sizeof(W) * 8 - 2;
    static constexpr W OWN = W(1) << BITS, UP_TO = W(2) << BITS, MASK = (W(1) << BITS) - 1;
};
constexpr uint32_t SPIN_MAX = 1u << 21;

__device__ __forceinline__ uint32_t ld_word(const uint32_t* p) { return ld_relaxed_u32(p); }
__device__ __forceinline__ uint64_t ld_word(const uint64_t* p) { return ld_relaxed(p); }
__device__ __forceinline__ void st_word(uint32_t* p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_word(uint64_t* p, uint64_t v) { st_relaxed(p, v); }

// Items of digit t (this thread's) in the tiles before `tile`.  Four
// predecessors are read at once: in the first wave every tile of the grid
// looks back through unfinished ones, and the reads' latency is what it costs.
template <class W>
__device__ __forceinline__ W look_back(const W* desc, int64_t tile, int t, unsigned* err) {
    constexpr int AHEAD = 4;
    W sum = 0;
    uint32_t spins = 0;
    int64_t p = tile - 1;
    while (p >= 0) {
        W w[AHEAD];
#pragma unroll
        for (int j = 0; j < AHEAD; ++j)
            w[j] = p - j >= 0 ? ld_word(desc + (p - j) * 256 + t) : Count<W>::UP_TO;
        int used = 0;
#pragma unroll
        for (int j = 0; j < AHEAD; ++j) {
            if (used != j || w[j] == 0) continue;          // not published yet: look again
            sum += w[j] & Count<W>::MASK;
            used = w[j] >= Count<W>::UP_TO ? AHEAD + 1 : j + 1;
        }
        if (used > AHEAD) break;
        p -= used;
        if (used == 0 && ++spins > SPIN_MAX) {
            if (err) atomicOr(err, GCC_DEVERR_WAIT_BUDGET);
            break;
        }
    }
    return sum;
}

// Histograms of every pass's digits.
__global__ void __launch_bounds__(RS_BLOCK)
rs_hist(const uint32_t* keys, size_t n, int bits, int passes, int digit_bits,
        uint32_t* hist) {
    __shared__ uint32_t h[SORT_MAX_PASSES][256];
    after_previous();
    for (int p = 0; p < SORT_MAX_PASSES; ++p) h[p][threadIdx.x] = 0;
    __syncthreads();
    const size_t stride = (size_t)gridDim.x * RS_BLOCK * 4;
    for (size_t i = ((size_t)blockIdx.x * RS_BLOCK + threadIdx.x) * 4; i < n; i += stride) {
        uint32_t k[4];
        const int m = n - i < 4 ? (int)(n - i) : 4;
        if (m == 4) {
            const uint4 v = *reinterpret_cast<const uint4*>(keys + i);
            k[0] = v.x; k[1] = v.y; k[2] = v.z; k[3] = v.w;
        } else {
            for (int j = 0; j < m; ++j) k[j] = keys[i + j];
        }
        for (int p = 0; p < passes; ++p) {
            const int left = bits - p * digit_bits;
            const uint32_t mask = (1u << (left < digit_bits ? left : digit_bits)) - 1u;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < m) atomicAdd(&h[p][(k[j] >> (p * digit_bits)) & mask], 1u);
        }
    }
    __syncthreads();
    for (int p = 0; p < passes; ++p)
        if (const uint32_t c = h[p][threadIdx.x]) atomicAdd(&hist[p * 256 + threadIdx.x], c);
}

// One pass over one tile.  Each warp ranks its own contiguous run of ITEMS * 32
// items with warp-private digit counters: the lanes that share a digit are
// found with one ballot per digit bit, no block barrier inside the loop.  One
// digit-major scan over (digit, warp) then gives every item its position in the
// tile staged in digit order -- warp w's items of a digit follow warp w-1's,
// which keeps the sort stable -- and each digit's run goes to its global
// position with consecutive threads on consecutive addresses (coalesced).
// Bound by issue and by the latency of the ranking's shared-memory round trips,
// not by memory (2^24 pairs: 0.14 ms a pass, 1.9 TB/s).  16 items per thread
// took 1.52 ms for a 2^24-op deterministic batch, 8 items 1.61 ms, 12 items
// 1.60 ms; __match_any_sync instead of the ballots 1.69 ms; a minimum of 3 or
// 4 resident blocks (spills) and loading the values behind the ranking were
// slower too.
// `flagged` (first pass of radix_sort_positions): values are positions, bit 31
// of the key moves to bit 31 of the value.
template <class W, int ITEMS>
__global__ void __launch_bounds__(RS_BLOCK)
rs_pass(const uint32_t* kin, const uint32_t* vin,
        uint32_t* kout, uint32_t* vout, size_t n, int shift, int width,
        int flagged, const uint32_t* hist, W* desc, W* desc_next, uint32_t* ticket,
        unsigned* err) {
    constexpr int TILE = RS_BLOCK * ITEMS;
    __shared__ uint32_t gbase[256];            // global start of each digit's run, less dstart
    __shared__ uint32_t wc[RS_WARPS][256];     // per-warp digit counts, then starts in the tile
    __shared__ uint32_t skey[TILE];
    __shared__ uint32_t sval[TILE];
    __shared__ uint32_t warp_sums[32];
    __shared__ uint32_t s_tile;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) wc[w][t] = 0;
    after_previous();
    if (t == 0) s_tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const size_t tile0 = (size_t)tile * TILE;
    const uint32_t tile_n = (uint32_t)(n - tile0 < (size_t)TILE ? n - tile0 : (size_t)TILE);
    const uint32_t base = (uint32_t)warp * (ITEMS * 32) + lane;    // the thread's first item of the tile
    kin += tile0;
    const uint32_t dmask = (1u << width) - 1u;
    uint32_t key[ITEMS], val[ITEMS];
    uint16_t rank[ITEMS];
#pragma unroll
    for (int c = 0; c < ITEMS; ++c) key[c] = base + c * 32 < tile_n ? kin[base + c * 32] : 0u;
    if (vin) {
        vin += tile0;
#pragma unroll
        for (int c = 0; c < ITEMS; ++c) val[c] = base + c * 32 < tile_n ? vin[base + c * 32] : 0u;
    } else {
#pragma unroll
        for (int c = 0; c < ITEMS; ++c) {
            val[c] = (uint32_t)tile0 + base + c * 32;
            if (flagged) {
                val[c] |= key[c] & 0x80000000u;
                key[c] &= 0x7fffffffu;
            }
        }
    }
    desc_next[(size_t)tile * 256 + t] = 0;     // the next pass's descriptors start unpublished
    const uint32_t in_hist = hist[t];
#pragma unroll
    for (int c = 0; c < ITEMS; ++c) {
        const bool valid = base + c * 32 < tile_n;
        const uint32_t dg = (key[c] >> shift) & dmask;
        unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int b = 0; b < 8; ++b) {          // bits from `width` on are zero in every lane
            const int x = (int)(dg << (31 - b)) >> 31;
            const unsigned m = __ballot_sync(0xffffffffu, x);
            peers &= ~(m ^ (unsigned)x);
        }
        const uint32_t prior = valid ? wc[warp][dg] : 0u;
        __syncwarp();
        if (valid && (peers & lt_mask()) == 0) wc[warp][dg] = prior + __popc(peers);
        __syncwarp();
        rank[c] = (uint16_t)(prior + __popc(peers & lt_mask()));
    }
    __syncthreads();
    uint32_t cnt[RS_WARPS], tot = 0;           // thread t owns digit t
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) {
        cnt[w] = tot;
        tot += wc[w][t];
    }
    st_word(desc + (size_t)tile * 256 + t, (tile ? Count<W>::OWN : Count<W>::UP_TO) | (W)tot);
    const uint32_t dstart = block_exclusive_scan<RS_WARPS>(tot, warp_sums, nullptr);
    const uint32_t gstart = block_exclusive_scan<RS_WARPS>(in_hist, warp_sums, nullptr);
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) wc[w][t] = dstart + cnt[w];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < ITEMS; ++c) {
        if (base + c * 32 < tile_n) {
            const uint32_t pos = wc[warp][(key[c] >> shift) & dmask] + rank[c];
            skey[pos] = key[c];
            sval[pos] = val[c];
        }
    }
    if (tile) {
        const W before = look_back<W>(desc, tile, t, err);
        st_word(desc + (size_t)tile * 256 + t, Count<W>::UP_TO | (before + (W)tot));
        gbase[t] = gstart + (uint32_t)before - dstart;
    } else {
        gbase[t] = gstart - dstart;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < ITEMS; ++c) {
        const uint32_t i = (uint32_t)c * RS_BLOCK + t;
        if (i < tile_n) {
            const uint32_t k = skey[i];
            const uint32_t out = gbase[(k >> shift) & dmask] + i;
            if (out < n) {                     // a bounded wait that gave up stays in bounds
                kout[out] = k;
                vout[out] = sval[i];
            }
        }
    }
}

template <class W, int ITEMS>
cudaError_t rs_passes(SortScratch& s, uint32_t* keys, uint32_t* vals, size_t n, int bits, bool flagged,
                      uint32_t** keys_out, uint32_t** vals_out, cudaStream_t st) {
    const SortPlan plan = sort_plan(bits);
    const unsigned tiles = (unsigned)sort_tiles(n);
    uint32_t *ki = keys, *vi = vals, *ko = s.k1, *vo = s.v1;
    W* desc = reinterpret_cast<W*>(s.work + SORT_DESC);
    W* next = desc + (size_t)tiles * 256;
    for (int p = 0; p < plan.passes; ++p) {
        const cudaError_t e = launch_after(
            rs_pass<W, ITEMS>, tiles, RS_BLOCK, st, ki, vi, ko, vo, n, p * plan.digit_bits,
            plan.width(bits, p), flagged && p == 0 ? 1 : 0, s.work + SORT_HIST + p * 256, desc, next,
            s.work + p, s.err);
        if (e != cudaSuccess) return e;
        uint32_t* tk = ki; ki = ko; ko = tk;
        uint32_t* tv = vi ? vi : s.v0; vi = vo; vo = tv;
        W* td = desc; desc = next; next = td;
    }
    *keys_out = ki;
    *vals_out = vi;
    return cudaSuccess;
}

cudaError_t rs_run(SortScratch& s, uint32_t* keys, uint32_t* vals, size_t n, int bits, bool flagged,
                   uint32_t** keys_out, uint32_t** vals_out, cudaStream_t st) {
    if (n <= SORT_SMALL)
        return rs_passes<uint32_t, SORT_ITEMS_SMALL>(s, keys, vals, n, bits, flagged, keys_out, vals_out, st);
    if (n <= SORT_MID)
        return rs_passes<uint32_t, SORT_ITEMS_MID>(s, keys, vals, n, bits, flagged, keys_out, vals_out, st);
    if (n < (size_t(1) << 30))
        return rs_passes<uint32_t, SORT_ITEMS_LARGE>(s, keys, vals, n, bits, flagged, keys_out, vals_out, st);
    return rs_passes<uint64_t, SORT_ITEMS_LARGE>(s, keys, vals, n, bits, flagged, keys_out, vals_out, st);
}

// --- prefix sum -------------------------------------------------------------
constexpr int SC_BLOCK = 1024;
constexpr int SC_ITEMS = 4;
constexpr int SC_TILE = SC_BLOCK * SC_ITEMS;

__global__ void scan_tile_sums(const uint32_t* __restrict__ d, size_t n, uint32_t* __restrict__ sums) {
    __shared__ uint32_t warp_sums[32];
    const size_t base = (size_t)blockIdx.x * SC_TILE + (size_t)threadIdx.x * SC_ITEMS;
    uint32_t s = 0;
    for (int k = 0; k < SC_ITEMS; ++k)
        if (base + k < n) s += d[base + k];
    uint32_t tot;
    block_exclusive_scan<32>(s, warp_sums, &tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void scan_sums(uint32_t* __restrict__ sums, uint32_t ntiles) {
    __shared__ uint32_t warp_sums[32];
    uint32_t carry = 0;
    for (uint32_t base = 0; base < ntiles; base += SC_BLOCK) {
        const uint32_t i = base + threadIdx.x;
        const uint32_t v = i < ntiles ? sums[i] : 0;
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan<32>(v, warp_sums, &tot);
        if (i < ntiles) sums[i] = carry + ex;
        carry += tot;
    }
}

__global__ void scan_apply(uint32_t* __restrict__ d, size_t n, const uint32_t* __restrict__ sums) {
    __shared__ uint32_t warp_sums[32];
    const size_t base = (size_t)blockIdx.x * SC_TILE + (size_t)threadIdx.x * SC_ITEMS;
    uint32_t v[SC_ITEMS];
    uint32_t s = 0;
    for (int k = 0; k < SC_ITEMS; ++k) {
        v[k] = base + k < n ? d[base + k] : 0;
        s += v[k];
    }
    uint32_t run = block_exclusive_scan<32>(s, warp_sums, nullptr) + sums[blockIdx.x];
    for (int k = 0; k < SC_ITEMS; ++k) {
        if (base + k < n) d[base + k] = run;
        run += v[k];
    }
}

// --- deterministic scheme ---------------------------------------------------
__global__ void det_emit(const uint64_t* __restrict__ ops, uint64_t n, int schema, uint32_t W,
                         uint32_t none, uint32_t n_meta, uint32_t* __restrict__ keys,
                         uint32_t* __restrict__ vals) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t r = cc_record(ops[i], schema, W, none);
    if (r >= n_meta) r = none;          // malformed ops are rejected by the kernel
    keys[i] = r;
    vals[i] = (uint32_t)i;
}

__global__ void det_flags(const uint64_t* __restrict__ ops, const uint32_t* __restrict__ sv,
                          uint64_t n, uint32_t* __restrict__ flags) {
    const uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const uint32_t op = sv[p];
    flags[p] = op < n && kind_writes((uint32_t)(ops[op] >> 40) & 0xffu) ? 1u : 0u;
}

// need: a write (or, when every access conflicts, any op) waits for all
// earlier ops on its record, a read for the earlier writes.
__global__ void det_need(const uint64_t* __restrict__ ops, const uint32_t* __restrict__ sk,
                         const uint32_t* __restrict__ sv, const uint32_t* __restrict__ wpre,
                         uint64_t n, uint32_t none, int all_conflict, uint32_t* __restrict__ need,
                         uint64_t* __restrict__ meta) {
    const uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const uint32_t key = sk[p];
    const uint32_t op = sv[p];
    if (key >= none || op >= n) return;
    const bool w = kind_writes((uint32_t)(ops[op] >> 40) & 0xffu);
    need[op] = (w || all_conflict) ? (uint32_t)p : wpre[p];
    if (p == 0 || sk[p - 1] != key) meta[key] = ((uint64_t)p << 32) | wpre[p];
}

// --- dense commit ranks -------------------------------------------------------
// A committed transaction's rank is the number of committed timestamps below
// its own.  The batch drew its timestamps from a counter, so they are small
// offsets from the batch's starting clock: one bit per timestamp marks the
// committed ones, a scan over the words counts the bits before each word, and
// a rank is that count plus the bits below in the word.  The bits and counts
// live in L2 (one bit per attempt), so the three launches cost little more
// than reading the batch's results: they replace a five-kernel radix sort of
// (timestamp, transaction), at 2^20 transactions 80 of OCC's 1,480 us.
// A batch with more timestamps than there are bits (32 per transaction of the
// largest batch) uses the same words as the heads of lists: word i holds the
// transactions whose timestamps share the bits from `shift` on, linked through
// a.seq in no order, the scan counts list lengths, and a rank is the count
// before the list plus the smaller timestamps in it.  A list is short: the
// shift is the smallest that fits the words, so it has one transaction on
// average when the batch is full, and 2^shift at most.  2^20 TO transactions
// at 50 and at 200 attempts each (kernels of 40 and 156 ms) are ranked in 0.06
// ms; one block taking a window of the bits at a time took 12 and 38, the sort
// 0.14.
// Offsets must fit 32 bits; a batch that used more timestamps than that
// reports GCC_DEVERR_TS_OVERFLOW.
__device__ __forceinline__ unsigned long long stamps_used(const ExecArgs& a, int scheme) {
    return scheme == GCC_MVCC ? a.st->ticket
                              : (scheme == GCC_TO ? a.dbs->to_clock : a.dbs->occ_clock) - a.st->ticket_base;
}
// How the batch is ranked: `words` of the scratch in use, 2^shift timestamps a
// word, `bits` one bit each or else a list.  (TO's and MVCC's count from 1.)
struct RankShape {
    uint32_t words;
    int shift;
    bool bits;
};
__device__ __forceinline__ RankShape rank_shape(const ExecArgs& a, const RankScratch& r, int scheme) {
    const unsigned long long n = stamps_used(a, scheme);
    if ((n >> 5) < r.words) return RankShape{(uint32_t)(n >> 5) + 1, 5, true};
    int shift = 5;
    while ((n >> shift) >= r.words) ++shift;
    return RankShape{(uint32_t)(n >> shift) + 1, shift, false};
}
__device__ __forceinline__ unsigned long long stamp(const ExecArgs& a, int scheme, uint32_t t) {
    return a.order_key[t] - (scheme == GCC_MVCC ? 0ull : a.st->ticket_base);
}
__device__ __forceinline__ bool stamp_of(const ExecArgs& a, int scheme, uint32_t t, unsigned long long& d) {
    if (a.results[t].status != GCC_TXN_COMMITTED) return false;
    d = stamp(a, scheme, t);
    return true;
}

__global__ void rank_mark(const __grid_constant__ ExecArgs a, const RankScratch r, int scheme) {
    after_previous();
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long d;
    if (t >= a.n_txns || !stamp_of(a, scheme, t, d)) return;
    if (d >= 0xffffffffull) atomicOr(&a.st->error, GCC_DEVERR_TS_OVERFLOW);
    const RankShape s = rank_shape(a, r, scheme);
    if ((d >> s.shift) >= s.words) return;
    uint32_t* w = r.bits + (d >> s.shift);
    if (s.bits) atomicOr(w, 1u << (d & 31));
    else a.seq[t] = atomicExch(w, t + 1);
}

// Transactions before each word beside the word; leaves `bits` zero.
constexpr int RANK_ITEMS = 4;
__global__ void __launch_bounds__(1024)
rank_scan(const __grid_constant__ ExecArgs a, const RankScratch r, int scheme) {
    __shared__ uint32_t warp_sums[32];
    __shared__ uint32_t s_tile;
    __shared__ unsigned long long s_before;
    after_previous();
    const RankShape s = rank_shape(a, r, scheme);
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_tile = atomicAdd(r.ticket, 1u);
        __syncthreads();
        const uint32_t tile = s_tile;
        const unsigned long long w0 = (unsigned long long)tile * 1024 * RANK_ITEMS + threadIdx.x * RANK_ITEMS;
        if ((unsigned long long)tile * 1024 * RANK_ITEMS >= s.words) return;
        uint32_t b[RANK_ITEMS], m[RANK_ITEMS], n = 0;
#pragma unroll
        for (int i = 0; i < RANK_ITEMS; ++i) {
            b[i] = w0 + i < s.words ? r.bits[w0 + i] : 0u;
            m[i] = 0;
            if (s.bits) m[i] = __popc(b[i]);
            else for (uint32_t u = b[i]; u; u = a.seq[u - 1]) ++m[i];
            n += m[i];
        }
        uint32_t tot;
        uint32_t before = block_exclusive_scan<32>(n, warp_sums, &tot);
        if (threadIdx.x == 0) {
            typedef Count<uint64_t> C;
            st_relaxed(r.desc + tile, (tile ? C::OWN : C::UP_TO) | tot);
            uint64_t sum = 0;
            uint32_t spins = 0;
            for (int64_t p = (int64_t)tile - 1; p >= 0;) {
                const uint64_t w = ld_relaxed(r.desc + p);
                if (w == 0) {
                    if (++spins > SPIN_MAX) { atomicOr(&a.st->error, GCC_DEVERR_WAIT_BUDGET); break; }
                    continue;
                }
                sum += w & C::MASK;
                if (w >= C::UP_TO) break;
                --p;
            }
            if (tile) st_relaxed(r.desc + tile, C::UP_TO | (sum + tot));
            s_before = sum;
        }
        __syncthreads();
        before += (uint32_t)s_before;
#pragma unroll
        for (int i = 0; i < RANK_ITEMS; ++i)
            if (w0 + i < s.words) {
                r.counts[w0 + i] = (uint64_t)before << 32 | b[i];
                if (b[i]) r.bits[w0 + i] = 0u;
                before += m[i];
            }
    }
}

// The ranks, and the scan's words left at zero for the next batch.
__global__ void __launch_bounds__(256)
rank_assign(const __grid_constant__ ExecArgs a, const RankScratch r, int scheme) {
    after_previous();
    const RankShape s = rank_shape(a, r, scheme);
    const uint32_t t = blockIdx.x * 256 + threadIdx.x;
    unsigned long long d;
    if (t < a.n_txns && stamp_of(a, scheme, t, d) && (d >> s.shift) < s.words) {
        const uint64_t count = r.counts[d >> s.shift];
        uint32_t rank = (uint32_t)(count >> 32);
        if (s.bits) rank += __popc((uint32_t)count & ((1u << (d & 31)) - 1u));
        else for (uint32_t u = (uint32_t)count; u; u = a.seq[u - 1]) rank += stamp(a, scheme, u - 1) < d;
        a.results[t].commit_order = rank;
    }
    if (blockIdx.x == 0) {
        for (uint32_t i = threadIdx.x; i < r.words / (1024 * RANK_ITEMS) + 1; i += 256) r.desc[i] = 0;
        if (threadIdx.x == 0) *r.ticket = 0;
    }
}

__global__ void dense_rank(const uint32_t* __restrict__ sk, const uint32_t* __restrict__ sv,
                           uint32_t n, gcc_txn_result* __restrict__ res) {
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n || sk[p] == 0xffffffffu || sv[p] >= n) return;
    res[sv[p]].commit_order = p;
}

// TicToc's serial order, (timestamp, sequence number), by three stable 32-bit
// sorts: sequence number, then the timestamp's low and high words.  Pass 0
// keys each transaction by its sequence number; passes 1 and 2 re-key the
// sorted order by a timestamp word.  Transactions that did not commit carry
// all-ones keys and stay last.
__global__ void tt_emit(const gcc_txn_result* __restrict__ res,
                        const unsigned long long* __restrict__ okey,
                        const uint32_t* __restrict__ seq, const uint32_t* __restrict__ sv,
                        int pass, uint32_t n, uint32_t* __restrict__ keys,
                        uint32_t* __restrict__ vals) {
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const uint32_t t = pass == 0 ? p : sv[p];
    const bool c = t < n && res[t].status == GCC_TXN_COMMITTED;
    uint32_t k = 0xffffffffu;
    if (c) k = pass == 0 ? seq[t] : pass == 1 ? (uint32_t)okey[t] : (uint32_t)(okey[t] >> 32);
    keys[p] = k;
    vals[p] = t;
}

// Deterministic scheme run op by op: every committed transaction's position
// among the committed ones in id order (an invalid transaction takes none).
__global__ void id_rank_emit(const gcc_txn_result* __restrict__ res, uint32_t n,
                             uint32_t* __restrict__ flags) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) flags[t] = res[t].status == GCC_TXN_COMMITTED ? 1u : 0u;
}

__global__ void id_rank_apply(const uint32_t* __restrict__ before, uint32_t n,
                              gcc_txn_result* __restrict__ res) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n && res[t].status == GCC_TXN_COMMITTED) res[t].commit_order = before[t];
}

__global__ void batch_begin_kernel(BatchState* st, DbState* dbs, int scheme) {
    BatchState z{};
    z.ticket_base = scheme == GCC_TO ? dbs->to_clock : dbs->occ_clock;
    *st = z;
}

inline unsigned blocks_for(uint64_t n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

// Zeroed tickets and descriptors, and the histograms of every pass.
static cudaError_t rs_prepare(SortScratch& s, const uint32_t* keys, size_t n, int bits, cudaStream_t st) {
    const SortPlan plan = sort_plan(bits);
    const cudaError_t e = cudaMemsetAsync(s.work, 0, (SORT_DESC + sort_desc_words(n)) * 4, st);
    if (e != cudaSuccess) return e;
    const unsigned grid = blocks_for(n, RS_BLOCK * 4 * 4);
    return launch_after(rs_hist, grid < 608u ? grid : 608u, RS_BLOCK, st, keys, n, bits, plan.passes,
                        plan.digit_bits, s.work + SORT_HIST);
}

cudaError_t radix_sort_pairs(SortScratch& s, size_t n, int bits, uint32_t** keys_out,
                             uint32_t** vals_out, cudaStream_t st) {
    if (n == 0) { *keys_out = s.k0; *vals_out = s.v0; return cudaSuccess; }
    const cudaError_t e = rs_prepare(s, s.k0, n, bits, st);
    if (e != cudaSuccess) return e;
    return rs_run(s, s.k0, s.v0, n, bits, false, keys_out, vals_out, st);
}

int radix_sort_launches(int bits) { return 1 + sort_plan(bits).passes; }

cudaError_t radix_sort_positions(SortScratch& s, uint32_t* keys, size_t n, int bits, bool flagged,
                                 bool prepared, uint32_t** keys_out, uint32_t** vals_out,
                                 cudaStream_t st) {
    if (!prepared) {
        const cudaError_t e = rs_prepare(s, keys, n, bits, st);
        if (e != cudaSuccess) return e;
    }
    return rs_run(s, keys, nullptr, n, bits, flagged, keys_out, vals_out, st);
}

size_t scan_tmp_words(size_t n) { return (n + SC_TILE - 1) / SC_TILE + 1; }

cudaError_t exclusive_scan_u32(uint32_t* d, size_t n, uint32_t* tmp, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const uint32_t ntiles = (uint32_t)((n + SC_TILE - 1) / SC_TILE);
    scan_tile_sums<<<ntiles, SC_BLOCK, 0, st>>>(d, n, tmp);
    scan_sums<<<1, SC_BLOCK, 0, st>>>(tmp, ntiles);
    scan_apply<<<ntiles, SC_BLOCK, 0, st>>>(d, n, tmp);
    return cudaGetLastError();
}

cudaError_t det_prepare(const ExecArgs& a, SortScratch& s, uint32_t* scan_tmp, int key_bits,
                        int schema, cudaStream_t st, bool all_conflict) {
    const uint64_t n = a.n_ops;
    if (n == 0) return cudaSuccess;
    const uint32_t none = (uint32_t)a.n_meta;   // sorts after every real record
    det_emit<<<blocks_for(n, 256), 256, 0, st>>>(a.ops, n, schema, a.n_warehouses, none,
                                                 (uint32_t)a.n_meta, s.k0, s.v0);
    uint32_t *sk, *sv;
    cudaError_t e = radix_sort_pairs(s, n, key_bits, &sk, &sv, st);
    if (e != cudaSuccess) return e;
    uint32_t* flags = (sk == s.k0) ? s.k1 : s.k0;   // the free key buffer
    det_flags<<<blocks_for(n, 256), 256, 0, st>>>(a.ops, sv, n, flags);
    e = exclusive_scan_u32(flags, n, scan_tmp, st);
    if (e != cudaSuccess) return e;
    det_need<<<blocks_for(n, 256), 256, 0, st>>>(a.ops, sk, sv, flags, n, none, all_conflict ? 1 : 0,
                                                 const_cast<uint32_t*>(a.need), a.meta);
    return cudaGetLastError();
}

size_t rank_desc_words(size_t words) { return words / (1024 * RANK_ITEMS) + 1; }

cudaError_t densify_commit_order(const ExecArgs& a, const RankScratch& r, gcc_scheme scheme, cudaStream_t st) {
    const uint32_t n = a.n_txns;
    if (n == 0) return cudaSuccess;
    cudaError_t e = launch_after(rank_mark, blocks_for(n, 256), 256, st, a, r, (int)scheme);
    const unsigned tiles = (unsigned)rank_desc_words(r.words);
    if (e == cudaSuccess)
        e = launch_after(rank_scan, tiles < 152u ? tiles : 152u, 1024, st, a, r, (int)scheme);
    if (e == cudaSuccess) e = launch_after(rank_assign, blocks_for(n, 256), 256, st, a, r, (int)scheme);
    return e;
}

cudaError_t densify_tictoc(const ExecArgs& a, SortScratch& s, cudaStream_t st) {
    const uint32_t n = a.n_txns;
    if (n == 0) return cudaSuccess;
    uint32_t *sk = nullptr, *sv = nullptr;
    for (int pass = 0; pass < 3; ++pass) {
        // the previous pass's sorted values feed the next pass's keys; when the
        // sort left them in (k0, v0), tt_emit rewrites those in place by index
        tt_emit<<<blocks_for(n, 256), 256, 0, st>>>(a.results, a.order_key, a.seq, sv, pass, n,
                                                    s.k0, s.v0);
        cudaError_t e = radix_sort_pairs(s, n, 32, &sk, &sv, st);
        if (e != cudaSuccess) return e;
    }
    dense_rank<<<blocks_for(n, 256), 256, 0, st>>>(sk, sv, n, a.results);
    return cudaGetLastError();
}

cudaError_t densify_in_id_order(const ExecArgs& a, uint32_t* flags, uint32_t* scan_tmp,
                                cudaStream_t st) {
    const uint32_t n = a.n_txns;
    if (n == 0) return cudaSuccess;
    id_rank_emit<<<blocks_for(n, 256), 256, 0, st>>>(a.results, n, flags);
    cudaError_t e = exclusive_scan_u32(flags, n, scan_tmp, st);
    if (e != cudaSuccess) return e;
    id_rank_apply<<<blocks_for(n, 256), 256, 0, st>>>(flags, n, a.results);
    return cudaGetLastError();
}

cudaError_t launch_batch_begin(BatchState* st, DbState* dbs, gcc_scheme scheme, cudaStream_t s) {
    batch_begin_kernel<<<1, 1, 0, s>>>(st, dbs, (int)scheme);
    return cudaGetLastError();
}

}  // namespace gcc
