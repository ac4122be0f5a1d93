// svt_unpack.cu -- stage 1 of the paper's Sec. 2.1 for GB300: the input
// words are parsed and the per-road structures the later stages read are
// built.
//
// The batch is cut into tiles of 1024 words (four warps of 256 words).  A
// prologue maps every tile to the first event that starts in it (one pass over
// the event offsets).  One pass over the tiles then validates every word
// against its left neighbour (rules V2..V7, V9 of include/svt.h's format),
// checks V1 for the events starting in the tile, gives every road header its
// global index (a scan over the tile, plus the road count of the tiles before,
// found by looking back over the counts that earlier tiles publish), records
// where it sits, counts its hits (rule V8, hits per layer) and, for the fused
// path, sizes its work and appends split roads to the work list.  The offsets
// and V10 are checked per event afterwards.
#include "svt_kernels.cuh"

namespace svt {

namespace {

// First index e in [0, n) with off[e] >= v (off assumed non-decreasing),
// searched cooperatively by a warp (every lane gets the result): 32 probes per
// round, so log32(n) dependent loads instead of log2(n).
__device__ __forceinline__ uint64_t warp_lower_bound64(const uint64_t *__restrict__ off,
                                                       uint64_t n, uint64_t v, int lane) {
    uint64_t lo = 0, hi = n;
    while (hi > lo) {
        const uint64_t step = (hi - lo + 31) / 32;
        const uint64_t p = lo + (uint64_t)lane * step;
        const bool lt = p < hi && __ldg(off + p) < v;
        const uint32_t k = __popc(__ballot_sync(0xffffffffu, lt));
        if (k == 0) {
            hi = lo;
        } else {
            const uint64_t pk = lo + (uint64_t)(k - 1) * step;
            hi = min(pk + step, hi);
            lo = pk + 1;
        }
    }
    return lo;
}

// Batch sizes for the launch sequence: the given values, or -- when `sizes`
// is set -- the device-resident pair {n_words, n_events}, which must not
// exceed the capacities the sequence was sized for (else BAD_ARG, empty batch).
// Every block derives the sizes itself; block 0 publishes them.
//
// first_ev[t] = lower_bound(event_off, t * TILE_WORDS) for t = 0..T: event e
// writes the tiles t with event_off[e-1] < t * TILE_WORDS <= event_off[e].
// With increasing offsets every entry is written once; otherwise the offsets
// are reported as BAD_ARG (the smallest key) by the per-event check, and the
// consumers clamp what they read to [0, n_events].
__global__ void k_prologue(Dims *dims, uint64_t n_words, uint64_t n_events,
                           const uint64_t *sizes, const uint64_t *__restrict__ event_off,
                           uint32_t *first_ev, unsigned long long *status, uint64_t *counts,
                           int n_counts, uint64_t *zero, int n_zero,
                           unsigned long long *tile_state, uint32_t *tile_ticket) {
    // first of its sequence: launched in stream order after whatever came
    // before, so only the next kernel is let in early
    allow_next_grid();
    bool bad = false;
    if (sizes) {
        const uint64_t w = sizes[0], e = sizes[1];
        bad = w > n_words || e > n_events;
        n_words = bad ? 0 : w;
        n_events = bad ? 0 : e;
    }
    const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    if (tid == 0) {
        if (dims) {
            dims->n_words = n_words;
            dims->n_events = n_events;
        }
        if (status) *status = bad ? (unsigned long long)SVT_ERR_BAD_ARG : ~0ull;
    }
    if (counts && tid < (uint64_t)n_counts) counts[tid] = 0;
    if (zero && tid < (uint64_t)n_zero) zero[tid] = 0;
    if (!first_ev) return;
    const uint64_t T = n_tiles(n_words);
    // nothing published and no tile taken yet
    if (tile_ticket && tid == 0) *tile_ticket = 0;
    if (tile_state)
        for (uint64_t t = tid; t < T; t += stride) tile_state[t] = 0ull;
    for (uint64_t e = tid; e <= n_events; e += stride) {
        const uint64_t t0 = e > 0 ? min(__ldg(event_off + e - 1), n_words) / TILE_WORDS + 1 : 0;
        const uint64_t t1 = e < n_events ? min(__ldg(event_off + e), n_words) / TILE_WORDS : T;
        for (uint64_t t = t0; t <= min(t1, T); ++t) first_ev[t] = (uint32_t)e;
    }
}

// Events [e_lo, e_hi) that start in tile t, clamped to the batch (fewer than
// 2^31 events).
__device__ __forceinline__ void tile_events(const uint32_t *__restrict__ first_ev, uint32_t t,
                                            uint32_t n_events, uint32_t &e_lo, uint32_t &e_hi) {
    e_lo = min(__ldg(first_ev + t), n_events);
    e_hi = max(e_lo, min(__ldg(first_ev + t + 1), n_events));
}

// ---- road indices across tiles: one pass with look-back --------------------------
// Every tile publishes its road count in tile_state[t] as soon as its block
// has counted (kind TILE_AGGREGATE), and its inclusive prefix -- the roads of
// tiles 0..t -- once it knows the tiles before it (kind TILE_INCLUSIVE; tile 0
// publishes that at once).  Words: kind in bits [63:62], count in [39:0];
// zero means nothing published yet.
constexpr unsigned long long TILE_AGGREGATE = 1, TILE_INCLUSIVE = 2;
constexpr unsigned long long TILE_COUNT_MASK = (1ull << 40) - 1;
constexpr uint32_t LOOK_BACK_SPINS = 1u << 20;   // bounded wait, then SVT_ERR_TIMEOUT

__device__ __forceinline__ void publish_tile(unsigned long long *p, unsigned long long kind,
                                             unsigned long long v) {
    const unsigned long long x = (kind << 62) | (v & TILE_COUNT_MASK);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(x) : "memory");
}
__device__ __forceinline__ unsigned long long peek_tile(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Roads in the tiles before tile t (t >= 1), by one warp: lane k reads tile
// hi - k of a window of 32 tiles, newest first; the sum runs over the window's
// tiles up to the newest one whose inclusive count is out (that one
// included), else over the whole window and on to the next.  A tile that has
// published nothing yet is re-read after a short sleep; it belongs to a block
// that took its tile earlier and is running, so it publishes soon.  After
// LOOK_BACK_SPINS rounds the wait gives up with SVT_ERR_TIMEOUT (the batch's
// status is then an error and its outputs are not used).
__device__ unsigned long long tiles_before(const unsigned long long *state, uint64_t t, int lane,
                                           unsigned long long *status) {
    unsigned long long excl = 0;
    uint32_t spins = 0;
    for (int64_t hi = (int64_t)t - 1; hi >= 0; hi -= 32) {
        const int64_t idx = hi - lane;
        // before tile 0 there is nothing: read as an inclusive count of zero
        unsigned long long v = idx >= 0 ? peek_tile(state + idx) : (TILE_INCLUSIVE << 62);
        for (;;) {
            const uint32_t incl = __ballot_sync(0xffffffffu, (v >> 62) == TILE_INCLUSIVE);
            const uint32_t stop = incl ? (uint32_t)(__ffs(incl) - 1) : 31u;
            const uint32_t need = stop == 31u ? 0xffffffffu : ((2u << stop) - 1u);
            const uint32_t missing = __ballot_sync(0xffffffffu, (v >> 62) == 0) & need;
            if (!missing) {
                unsigned long long x = (uint32_t)lane <= stop ? (v & TILE_COUNT_MASK) : 0ull;
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
                excl += x;
                if (incl) return excl;
                break;
            }
            if (++spins > LOOK_BACK_SPINS) {
                if (lane == 0) report(status, 0, SVT_ERR_TIMEOUT);
                return excl;
            }
            __nanosleep(64);
            if ((missing >> lane) & 1u) v = peek_tile(state + idx);
        }
    }
    return excl;
}

// K2, one tile of 1024 words per block, 256 words per warp: a warp reads its
// words as eight rows of 32, lane l word l, so that what the rules ask of a word
// is a vote over its row and the tile is described by 32-bit masks of its rows
// (hits, road headers, event headers, hits of the same layer as the word
// before).  Between the masks (first barrier) and the outputs (second barrier)
// every warp works by itself:
//  * the masks of all 32 rows, one row per lane, give every warp the index of
//    each road header by one warp scan;
//  * a run of hits of one layer inside a row adds its length to its road's
//    counter of that layer with one shared-memory atomic (the packed
//    5-bits-per-layer word; a field can only overflow with more than 31 hits of
//    one layer, which rule V8 already rejects); hits past the tile's end that
//    continue its last road are read from a back halo (a valid road has at most
//    96 hits, so 100 words cover it);
//  * rule V8: a hit whose 16 predecessors are hits of the same layer is the
//    17th (or later) of a contiguous block.  For the smallest status key this
//    matches counting over the run: the first out-of-order hit of a run is an
//    UNSORTED word that precedes any later, non-contiguous 17th hit.  V8 fires
//    where 16 set bits of the "same layer" mask end;
//  * one thread per road then writes the road's outputs; for the fused path
//    a warp's split roads are appended to the work list at a range that one
//    atomic reserves.
// Bound by issue slots (4900 warp instructions a tile: 2300 in the rows, 700 in
// 56 roads' descriptors; 62 % of the slots taken at 12 tiles per SM) and the
// chain of loads, barriers and look-back of a tile, not by HBM.  Before, a
// thread took eight consecutive words and block scans and barriers (nine a tile)
// joined them.  Alone on the GPU, before and now: cold caches, 1 tile 8.6
// and 6.4 us, 115 tiles 10.4 and 8.6; warm, 1222 tiles 14.2 and 12.7, 3441 29.5
// and 24.5, 7694 47.7 and 43.6.  (Windows of 64 or 128 tiles in the
// look-back gained nothing; the instances differ by the pairing's counts, whose
// code costs 5 % where it is not used.)
template <bool PAIR>
__global__ void __launch_bounds__(TILE_THREADS, 12)
    k_unpack_roads(const uint32_t *__restrict__ words, const uint64_t *__restrict__ event_off,
                   const Dims *__restrict__ dims, const uint32_t *__restrict__ first_ev,
                   unsigned long long *tile_state, uint32_t *tile_ticket, uint64_t *total64,
                   uint64_t road_cap, uint32_t *road_word, uint32_t *road_nhit,
                   uint32_t *event_road, const svt_config cfg, const FusedRoads fr,
                   uint64_t *counts, unsigned long long *status) {
    constexpr int ROWS = TILE_WORDS / 32, WARP_ROWS = ROWS / (TILE_THREADS / 32), BACK = 100;
    constexpr int WARP_WORDS = 32 * WARP_ROWS;
    static_assert(ROWS == 32 && TILE_THREADS == 128 && WARP_ROWS == TILE_PER_THREAD && WARP_ROWS == 8,
                  "a lane per row of the tile, eight rows per warp");
    constexpr uint32_t ALL = 0xffffffffu;
    constexpr uint32_t HIT_END = 1u << 30, EVENT_BEGIN = 3u << 30;   // word types by value
    constexpr uint32_t SENTINEL = EVENT_BEGIN;   // an event-header word: ends every run
    __shared__ __align__(16) uint32_t cnt[TILE_WORDS];   // per road of the tile: 5 bits per layer
    // V11 counts of each road's hit run: layer 4 [9:0], layer 5 [19:10], all
    // hits [31:20].  A field can only overflow in a run of more than 1023 hits,
    // which then also shows more than 96 hits and is not checked.
    __shared__ __align__(16) uint32_t cnt45[PAIR ? TILE_WORDS : 4];
    // each road header: tile position and word (apart for pairing, whose counts
    // would otherwise leave twelve tiles no L1)
    __shared__ uint2 hdr[PAIR ? 1 : TILE_WORDS];
    __shared__ uint32_t hdr_word[PAIR ? TILE_WORDS : 1];
    __shared__ uint16_t hdr_pos[PAIR ? TILE_WORDS : 1];
    __shared__ __align__(16) uint32_t hit_bits[ROWS], road_bits[ROWS];
    __shared__ uint32_t event_bits[ROWS];                // (the reserved type as well)
    __shared__ uint32_t same_bits[1 + ROWS];             // [0]: the 32 words before the tile
    __shared__ uint32_t row_roads[ROWS];                 // road headers before each row
    __shared__ uint32_t last_word[TILE_THREADS / 32];    // the word before each warp's first
    __shared__ int v1_flag;   // a V1 failure in the tile (read after the second barrier)
    __shared__ unsigned long long comb_s;   // evaluated combinations of the block's tiles
    __shared__ uint32_t base_s;             // roads before the tile
    __shared__ uint32_t tile_s;             // the tile this block took
    wait_prior_grid();
    allow_next_grid();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    // tiles are taken in increasing order from a counter, so the tiles before
    // the one a block holds belong to blocks that are already running (the next
    // tile is taken while the block works on one: it is done next)
    if (threadIdx.x == 0) {
        tile_s = atomicAdd(tile_ticket, 1u);
        comb_s = 0;
    }
    const uint32_t n_words = (uint32_t)dims->n_words, n_events = (uint32_t)dims->n_events;
    const uint32_t T = (uint32_t)n_tiles(n_words);
    unsigned long long comb_sum = 0;   // of this thread's roads
    __syncthreads();
    for (;;) {
        const uint32_t t = tile_s;
        if (t >= T) break;
        const uint32_t tile_start = t * TILE_WORDS;
        const uint32_t rest_len = n_words - tile_start;   // words from the tile's first on
        const uint32_t tile_len = min((uint32_t)TILE_WORDS, rest_len);
        const uint32_t first = (uint32_t)(warp * WARP_WORDS + lane);   // this lane's first word
        const uint32_t *__restrict__ mine = words + tile_start + first;
        uint32_t w[WARP_ROWS];
#pragma unroll
        for (int i = 0; i < WARP_ROWS; ++i)
            w[i] = first + 32 * i < rest_len ? __ldg(mine + 32 * i) : SENTINEL;
        // warp 0: the row before the tile; warp 3: the row after it
        uint32_t halo = SENTINEL;
        if (warp == 0) {
            if (t > 0) halo = __ldg(mine - 32);
        } else if (warp == 3) {
            if (first + WARP_WORDS < rest_len) halo = __ldg(mine + WARP_WORDS);
        }
        // the events that start in the tile and this thread's first one
        uint32_t e_lo, e_hi;
        tile_events(first_ev, t, n_events, e_lo, e_hi);
        const uint32_t e_mine = e_lo + ((threadIdx.x + 64) & (TILE_THREADS - 1));   // (warp 2 first)
        // its position in the tile, TILE_WORDS when it does not start in it
        auto event_pos = [&](uint32_t e) {
            const uint64_t d = __ldg(event_off + e) - tile_start;   // (wraps below the tile)
            return d < tile_len ? (uint32_t)d : (uint32_t)TILE_WORDS;
        };
        const uint32_t pos_first = e_mine < e_hi ? event_pos(e_mine) : (uint32_t)TILE_WORDS;
        uint32_t next_tile = 0;
        if (threadIdx.x == 0) {
            next_tile = atomicAdd(tile_ticket, 1u);
            v1_flag = 0;
        }
#pragma unroll
        for (int i = 0; i < TILE_WORDS / 4 / TILE_THREADS; ++i) {
            reinterpret_cast<uint4 *>(cnt)[threadIdx.x + i * TILE_THREADS] = make_uint4(0, 0, 0, 0);
            if (PAIR)
                reinterpret_cast<uint4 *>(cnt45)[threadIdx.x + i * TILE_THREADS] = make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int i = 0; i < WARP_ROWS; ++i) {
            const uint32_t h = __ballot_sync(ALL, w[i] < HIT_END);
            const uint32_t r = __ballot_sync(ALL, (int)w[i] < (int)EVENT_BEGIN);
            if (lane == 0) {
                hit_bits[warp * WARP_ROWS + i] = h;
                road_bits[warp * WARP_ROWS + i] = r;
            }
        }
        if (lane == 31 && warp < 3) last_word[warp + 1] = w[WARP_ROWS - 1];
        if (warp == 0) {
            const uint32_t pw = __shfl_up_sync(ALL, halo, 1);
            const uint32_t h = __ballot_sync(ALL, lane >= 17 && halo < HIT_END && (halo ^ pw) < (1u << 27));
            if (lane == 0) same_bits[0] = h;
            if (lane == 31) last_word[0] = halo;
        }
        __syncthreads();
        // every warp: the road (low half) and event (high half) headers before
        // each row, a lane per row (a word of the reserved type, which breaks
        // V3, counts as an event header: V2 then reports the same key)
        const uint32_t tile_hits = hit_bits[lane], tile_roads = road_bits[lane];
        uint32_t before_row, heads;
        {
            const int in_row = (int)tile_len - 32 * lane;
            const uint32_t ev = ~(tile_hits | tile_roads) &
                                (in_row >= 32 ? ALL : in_row > 0 ? (1u << in_row) - 1u : 0u);
            if (warp == 0) event_bits[lane] = ev;
            const uint32_t own = __popc(tile_roads) | (__popc(ev) << 16);
            uint32_t x = own;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(ALL, x, d);
                if (lane >= d) x += y;
            }
            heads = __shfl_sync(ALL, x, 31);
            before_row = (x - own) & 0xFFFFu;
        }
        const uint32_t n_roads_tile = heads & 0xFFFFu;
        // the tile's road count for the tiles after it, before anything else
        if (threadIdx.x == 0)
            publish_tile(tile_state + t, t == 0 ? TILE_INCLUSIVE : TILE_AGGREGATE, n_roads_tile);
        if (warp == 0) row_roads[lane] = before_row;
        // V1: the events starting in this tile start with an event header; V4:
        // no hit comes right after one (a header elsewhere breaks V2 at the
        // word before)
        for (uint32_t e = e_mine; e < e_hi; e += TILE_THREADS) {
            const uint32_t ps = e == e_mine ? pos_first : event_pos(e);
            if (ps >= TILE_WORDS) continue;
            if (((hit_bits[ps >> 5] | road_bits[ps >> 5]) >> (ps & 31u)) & 1u) {
                report(status, tile_start + ps, SVT_ERR_BAD_TYPE);                      // V1
                v1_flag = 1;
            }
            const uint32_t nx = ps + 1;
            if (nx < TILE_WORDS ? (hit_bits[nx >> 5] >> (nx & 31u)) & 1u
                                : nx < rest_len && __ldg(words + tile_start + nx) < HIT_END)
                report(status, (uint64_t)tile_start + nx, SVT_ERR_BAD_TYPE);            // V4
        }
        // the rows: per-word rules V3 and V5..V7 against the word before (tile 0
        // has none), road headers, hits into their road.
        // A branch-free filter first: a word is suspect when it is a hit with
        // reserved bits, a layer above 5 (the reserved type as well), or a hit
        // of a higher layer before it (as signed values headers are below every
        // hit).  Only warps with a suspect word run the rules one by one (which
        // report the exact status keys).
        {
            uint32_t hit_or = 0;   // the hits' bits; bit 15 also for V7
            int top = 0;           // the largest hit or word of the reserved type
            uint32_t carry = last_word[warp];
            // the latest road header before the row, as an index of the tile
            int r_row = (int)__shfl_sync(ALL, before_row, warp * WARP_ROWS) - 1;
            // pairing counts only hits inside a road's run (a road header and
            // the hits right after it): is the latest earlier non-hit word of
            // the tile a road header?  (Hits before the tile's first header are
            // not counted: the tile before takes them through its back halo.)
            bool in_run = false;
            if (PAIR) {
                const uint32_t rows = __ballot_sync(ALL, ~tile_hits != 0u && lane < warp * WARP_ROWS);
                if (rows) {
                    const int k = 31 - __clz(rows);
                    const uint32_t nh = ~__shfl_sync(ALL, tile_hits, k);
                    in_run = (__shfl_sync(ALL, tile_roads, k) >> (31 - __clz(nh))) & 1u;
                }
            }
            uint4 masks = make_uint4(0, 0, 0, 0);   // road headers of four rows
#pragma unroll
            for (int i = 0; i < WARP_ROWS; ++i) {
                if ((i & 3) == 0)
                    masks = *reinterpret_cast<const uint4 *>(road_bits + warp * WARP_ROWS + i);
                const uint32_t rm = (i & 3) == 0 ? masks.x : (i & 3) == 1 ? masks.y
                                  : (i & 3) == 2 ? masks.z : masks.w;
                const uint32_t x = w[i];
                const uint32_t rot = __shfl_sync(ALL, x, (lane + 31) & 31);
                const uint32_t pw = lane == 0 ? carry : rot;
                carry = rot;
                const bool hit = x < HIT_END;
                top = max(top, (int)x);
                hit_or |= x & ~(uint32_t)((int)x >> 31);
                hit_or |= (uint32_t)(hit & ((int)pw > (int)(x | 0x07FFFFFFu))) << 15;
                const bool same = hit && (x ^ pw) < (1u << 27);
                const uint32_t sm = __ballot_sync(ALL, same);
                if (lane == 0) same_bits[1 + warp * WARP_ROWS + i] = sm;
                const int r = r_row + __popc(rm & lt);   // latest header before this word
                if ((int)x < (int)EVENT_BEGIN) {         // a road header
                    if constexpr (PAIR) {
                        hdr_pos[r + 1] = (uint16_t)(first + 32 * i);
                        hdr_word[r + 1] = x;
                    } else {
                        hdr[r + 1] = make_uint2(first + 32 * i, x);
                    }
                }
                // the first word of a run of hits of one layer (in this row)
                if ((hit & (!same | (lane == 0))) & (r >= 0)) {
                    const uint32_t len = (uint32_t)(__clz((int)__brev(~sm & (0xFFFFFFFEu << lane))) - lane);
                    const uint32_t l = hit_layer(x);
                    atomicAdd(&cnt[r], len << (5 * l));
                    if (PAIR) {
                        const uint32_t nh = ~hit_bits[warp * WARP_ROWS + i] & lt;
                        if (nh ? (rm >> (31 - __clz(nh))) & 1u : (uint32_t)in_run)
                            atomicAdd(&cnt45[r], (len << 20) + (l == 4 ? len : 0u) +
                                                     (l == 5 ? len << 10 : 0u));
                    }
                }
                if (PAIR) {
                    const uint32_t nh = ~hit_bits[warp * WARP_ROWS + i];
                    if (nh) in_run = (rm >> (31 - __clz(nh))) & 1u;
                }
                r_row += __popc(rm);
            }
            if (__any_sync(ALL, (hit_or & 0x07FF8000u) != 0u || top >= (int)(6u << 27))) {
                carry = last_word[warp];
#pragma unroll
                for (int i = 0; i < WARP_ROWS; ++i) {
                    const uint32_t x = w[i];
                    const uint32_t rot = __shfl_sync(ALL, x, (lane + 31) & 31);
                    const uint32_t pw = lane == 0 ? carry : rot;
                    carry = rot;
                    if (first + 32 * i >= rest_len) continue;
                    const uint32_t k = tile_start + first + 32 * i;
                    const uint32_t ty = w_type(x);
                    if (ty == TYPE_BAD) {
                        report(status, k, SVT_ERR_BAD_TYPE);                                    // V3
                    } else if (ty == TYPE_HIT) {
                        // V7 also fires on an event's first word, where V1 already
                        // reports the same word with the smallest code, so the key is unchanged.
                        if (hit_reserved(x) != 0) report(status, k, SVT_ERR_BAD_RESERVED);      // V5
                        if (hit_layer(x) > 5) report(status, k, SVT_ERR_BAD_LAYER);             // V6
                        if (k > 0 && w_type(pw) == TYPE_HIT && hit_layer(pw) > hit_layer(x))
                            report(status, k, SVT_ERR_UNSORTED);                                // V7
                    }
                }
            }
        }
        // hits after the tile that continue the tile's last road: its header is
        // the tile's last word that is no hit
        if (warp == 3 && n_roads_tile > 0) {
            const uint32_t rows = __ballot_sync(ALL, ~tile_hits != 0u);   // (not 0: a road is no hit)
            const int k = 31 - __clz(rows);
            const uint32_t nh = ~__shfl_sync(ALL, tile_hits, k);
            if ((__shfl_sync(ALL, tile_roads, k) >> (31 - __clz(nh))) & 1u) {
                const uint32_t r = n_roads_tile - 1;
                for (int c0 = 0; c0 < BACK; c0 += 32) {
                    if (c0)
                        halo = (uint32_t)(TILE_WORDS + c0 + lane) < rest_len
                                   ? __ldg(words + tile_start + TILE_WORDS + c0 + lane) : SENTINEL;
                    const bool hit = c0 + lane < BACK && halo < HIT_END;
                    const uint32_t miss = ~__ballot_sync(ALL, hit);
                    const uint32_t run = miss ? (uint32_t)__ffs((int)miss) - 1u : 32u;
                    if ((uint32_t)lane < run) {
                        const uint32_t l = hit_layer(halo);
                        atomicAdd(&cnt[r], 1u << (5 * l));
                        if (PAIR)
                            atomicAdd(&cnt45[r], (1u << 20) + (l == 4 ? 1u : 0u) + (l == 5 ? 1u << 10 : 0u));
                    }
                    if (miss) break;
                }
            }
        }
        // the roads of the tiles before this one; then the tile's inclusive
        // count for the tiles after it
        if (warp == 1) {
            const unsigned long long before = t ? tiles_before(tile_state, t, lane, status) : 0ull;
            if (lane == 0) {
                if (t) publish_tile(tile_state + t, TILE_INCLUSIVE, before + n_roads_tile);
                base_s = (uint32_t)before;
                if (t + 1 == T) {   // the last tile: the batch's road count
                    const unsigned long long R = before + n_roads_tile;
                    if (R > 0xFFFFFFFFull) report(status, 0, SVT_ERR_OOM);
                    if (total64) *total64 = R;
                    if (event_road) event_road[n_events] = (uint32_t)R;
                }
            }
        }
        if (threadIdx.x == 0) tile_s = next_tile;   // (every thread has read t)
        __syncthreads();
        const uint32_t tile_base = base_s;   // (fewer roads than words)
        // V2: every event-header word must sit at an event offset.  When the
        // tile holds as many headers as events start in it and all of those
        // start with a header (V1), the headers are exactly those starts;
        // otherwise every header of the tile is looked up.
        if ((heads >> 16) != e_hi - e_lo || v1_flag) {   // (rare: the batch is invalid)
            for (int i = 0; i < WARP_ROWS; ++i) {
                uint32_t bal = event_bits[warp * WARP_ROWS + i];
                for (; bal; bal &= bal - 1) {
                    const uint32_t k = tile_start + (uint32_t)((warp * WARP_ROWS + i) * 32 + __ffs((int)bal) - 1);
                    const uint64_t e = warp_lower_bound64(event_off, n_events, k, lane);
                    if (lane == 0 && !(e < n_events && __ldg(event_off + e) == k))
                        report(status, k, SVT_ERR_BAD_TYPE);
                }
            }
        }
        // V11 where an event starts with a hit: the run of the road before it ends
        // there, and not with the hits (at the offset, V1 decides against the run
        // that the counts below cover).  A run of more than 96 hits breaks another
        // rule at one of its own words.
        if (PAIR && v1_flag) {
            for (uint32_t e = e_mine; e < e_hi; e += TILE_THREADS) {
                const uint32_t ps = event_pos(e), s0 = tile_start + ps;
                if (ps >= TILE_WORDS || !((hit_bits[ps >> 5] >> (ps & 31u)) & 1u)) continue;
                int unpaired = 0;
                for (uint32_t n = 1; n <= min(s0, 97u); ++n) {
                    const uint32_t x = __ldg(words + s0 - n);
                    if (x >= HIT_END) {
                        if (unpaired && (int)x < (int)EVENT_BEGIN)   // the run's road header
                            report(status, (uint64_t)s0 - 1, SVT_ERR_XFT_UNPAIRED);
                        break;
                    }
                    unpaired += (hit_layer(x) == 4 ? 1 : 0) - (hit_layer(x) == 5 ? 1 : 0);
                }
            }
        }
        // V8: a hit whose 16 predecessors are hits of its layer is the 17th (or
        // later) of a run, i.e. 16 consecutive "same" bits end at it.  Lane
        // k - 1 looks at rows k - 2 and k - 1 (mask words k - 1 and k): bit i of
        // X is position 32 (k - 2) + i, and after the four steps bit s of y says
        // bits s .. s + 15 of X are set.
        if (warp == 3) {
            const int k = lane + 1;
            const unsigned long long X =
                (unsigned long long)same_bits[k - 1] | ((unsigned long long)same_bits[k] << 32);
            unsigned long long y = X & (X >> 1);
            y &= y >> 2;
            y &= y >> 4;
            y &= y >> 8;
            const unsigned long long m = y & (0xFFFFFFFFull << 17);   // runs ending in word k
            if (m) {
                const int s_ = __ffsll((long long)m) - 1;
                report(status, (uint64_t)tile_start + (uint64_t)(int64_t)(32 * (k - 2) + s_ + 15),
                       SVT_ERR_TOO_MANY_HITS);
            }
        }
        // first road of every event that starts inside this tile: the number
        // of road headers before the event's first word
        for (uint32_t e = e_mine; e < e_hi; e += TILE_THREADS) {
            const uint32_t ps = e == e_mine ? pos_first : event_pos(e);
            if (ps >= TILE_WORDS) continue;
            event_road[e] = tile_base + row_roads[ps >> 5] +
                            __popc(road_bits[ps >> 5] & ((1u << (ps & 31u)) - 1u));
        }
        // one thread per road of the tile
        for (uint32_t r0 = warp * 32; r0 < n_roads_tile; r0 += TILE_THREADS) {
            const uint32_t rl = r0 + lane;
            const uint32_t r = tile_base + rl;
            uint32_t items = 0;
            if (rl < n_roads_tile) {
                const uint32_t p = tile_start + (PAIR ? hdr_pos[PAIR ? rl : 0] : hdr[PAIR ? 0 : rl].x);
                const uint32_t hw = PAIR ? hdr_word[PAIR ? rl : 0] : hdr[PAIR ? 0 : rl].y;
                const uint32_t packed = cnt[rl];
                if (rd_sector(hw) >= cfg.n_sectors) report(status, p, SVT_ERR_BAD_SECTOR);      // V9
                if (PAIR) {
                    // V11, at the last word of the road's run.  A run of more than 96
                    // hits (or one that goes past the back halo) breaks V6, V7 or V8
                    // at one of its own words, which is then the smaller key.
                    const uint32_t v = cnt45[rl], run = v >> 20;
                    if (run <= 96u && (v & 1023u) != ((v >> 10) & 1023u))
                        report(status, (uint64_t)p + run, SVT_ERR_XFT_UNPAIRED);
                }
                if (r >= road_cap) {
                    report(status, p, SVT_ERR_OOM);
                } else {
                    if (road_word) road_word[r] = p;
                    if (road_nhit) road_nhit[r] = packed;
                    if (fr.desc) {
                        const RoadDesc d = make_road_desc(p, packed, hw, cfg);
                        items = road_big_items(d, fr);
                        fr.desc[r] = d;
                        comb_sum += d.a.w;
                    }
                }
            }
            // the warp's split roads, in order, and their items
            const uint32_t split = __ballot_sync(ALL, items != 0u);
            if (split) {
                unsigned long long x = items;   // inclusive sums
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const unsigned long long y = __shfl_up_sync(ALL, x, d);
                    if (lane >= d) x += y;
                }
                unsigned long long b = 0;
                if (lane == 31) {
                    b = atomicAdd(fr.bl.reserve, (x << 32) | (unsigned long long)__popc(split));
                    if ((b >> 32) + x > 0xFFFFFFFFull)
                        report(status, tile_start, SVT_ERR_OOM);   // item count needs 32 bits
                }
                b = __shfl_sync(ALL, b, 31);
                if (items) {
                    const uint32_t j = (uint32_t)b + __popc(split & lt);   // < R <= road_cap
                    fr.bl.road[j] = r;
                    fr.bl.item_off[j] = (uint32_t)(b >> 32) + (uint32_t)x - items;
                    fr.key[r] = ~0ull;
                    fr.bl.pending[j] = items;
                }
            }
        }
        __syncthreads();   // the tile's shared entries have been read
    }
    if (fr.desc && counts) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) comb_sum += __shfl_xor_sync(ALL, comb_sum, d);
        if (lane == 0 && comb_sum) atomicAdd(&comb_s, comb_sum);
        __syncthreads();
        if (threadIdx.x == 0 && comb_s) atomicAdd((unsigned long long *)(counts + 2), comb_s);
    }
    // an empty batch has no last tile to write the road count of
    if (T == 0 && blockIdx.x == 0 && threadIdx.x == 0 && event_road) event_road[n_events] = 0;
}

__global__ void k_unpack_events(const uint32_t *__restrict__ words,
                                const uint64_t *__restrict__ event_off,
                                const Dims *__restrict__ dims,
                                const uint32_t *__restrict__ event_road,
                                unsigned long long *status) {
    wait_prior_grid();
    allow_next_grid();
    check_events(words, event_off, dims->n_words, dims->n_events, event_road, status,
                 (uint64_t)blockIdx.x * blockDim.x + threadIdx.x,
                 (uint64_t)gridDim.x * blockDim.x);
}

}  // namespace

void launch_prologue(Dims *dims, uint64_t n_words, uint64_t n_events, const uint64_t *sizes,
                     const uint64_t *event_off, uint32_t *first_ev, unsigned long long *status,
                     uint64_t *counts, int n_counts, uint64_t *zero, int n_zero,
                     unsigned long long *tile_state, uint32_t *tile_ticket, int grid,
                     cudaStream_t st) {
    uint64_t g = first_ev ? (n_events + 1 + 255) / 256 : 1;
    const uint64_t gt = tile_state ? (n_tiles(n_words) + 255) / 256 : 1;
    if (gt > g) g = gt;
    if (g > (uint64_t)grid) g = (uint64_t)grid;
    if (g < 1) g = 1;
    k_prologue<<<(int)g, 256, 0, st>>>(dims, n_words, n_events, sizes, event_off, first_ev, status,
                                       counts, n_counts, zero, n_zero, tile_state, tile_ticket);
}

void launch_unpack_roads(const uint32_t *words, const uint64_t *event_off, const Dims *dims,
                         const uint32_t *first_ev, uint64_t max_words,
                         unsigned long long *tile_state, uint32_t *tile_ticket, uint64_t *total64,
                         uint64_t road_cap, uint32_t *road_word, uint32_t *road_nhit,
                         uint32_t *event_road, const svt_config cfg, const FusedRoads fr,
                         uint64_t *counts, unsigned long long *status, int grid,
                         bool max_shared, cudaStream_t st) {
    uint64_t T = n_tiles(max_words);
    int g = (int)(T < (uint64_t)grid ? T : (uint64_t)grid);
    if (g < 1) g = 1;   // an empty batch still writes its road count
    // max_shared (the fit kernel with one road per lane comes next and the words
    // are in device memory): an SM has to run empty to change how its on-chip
    // memory is split, and with this kernel's own choice (164 KB of shared memory)
    // the fit's blocks cannot start beside the last tiles.  3000 events of small
    // roads, whole pass: 41.6 us without, 38.2 with.  Words in mapped host memory
    // want the L1 that the larger split takes: 97 us without, 115 with.  The
    // other forms of the fit gained nothing (3000 events: 206.3 and 206.2) or
    // lost 3 % (512 events of uneven roads).
    launch_chained(max_shared, cfg.xft_pairs ? k_unpack_roads<true> : k_unpack_roads<false>, g,
                   TILE_THREADS, 0, st, words, event_off, dims, first_ev, tile_state, tile_ticket,
                   total64, road_cap, road_word, road_nhit, event_road, cfg, fr, counts, status);
}

void launch_unpack_events(const uint32_t *words, const uint64_t *event_off, const Dims *dims,
                          uint64_t max_events, const uint32_t *event_road,
                          unsigned long long *status, int grid, cudaStream_t st) {
    uint64_t blocks = (max_events + 255) / 256;
    if (blocks < 1) blocks = 1;
    int g = (int)(blocks < (uint64_t)grid ? blocks : (uint64_t)grid);
    launch_after(k_unpack_events, g, 256, 0, st, words, event_off, dims, event_road, status);
}

}  // namespace svt
