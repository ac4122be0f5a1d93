// svt_plain.cu -- the plain per-stage path: combine writes every combination
// of one hit per layer, fit evaluates one combination per thread, select keeps
// the best passing combination per road, format packs the records.  This is
// the structure of the paper's Sec. 2.1 GPU port (one kernel per stage, the
// loops unrolled so that one thread handles one combination), kept here as
// the baseline of the fused path and as the per-stage C ABI.  Its launches are
// chained like the fused path's (launch_after): each kernel waits for the one
// before it on the device, so the gaps between the eight short launches overlap.
#include "svt_kernels.cuh"

namespace svt {

namespace {

__device__ __forceinline__ uint64_t road_count(const uint64_t *n_roads, uint64_t road_cap) {
    uint64_t R = *n_roads;
    return R < road_cap ? R : road_cap;
}

__global__ void k_combine_count(const uint32_t *__restrict__ road_nhit,
                                const uint64_t *__restrict__ n_roads, uint64_t road_cap,
                                const svt_config cfg, uint32_t *road_flags, uint64_t *comb_cnt,
                                const unsigned long long *status) {
    wait_prior_grid();
    allow_next_grid();
    if (!status_ok(status)) return;
    const uint64_t R = road_count(n_roads, road_cap);
    for (uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r < R;
         r += (uint64_t)gridDim.x * blockDim.x) {
        const RoadShape s = road_shape(road_nhit[r], cfg.xft_pairs);
        uint32_t flags = s.total_hits == 0 ? SVT_FLAG_NO_HITS : 0u;
        uint64_t n = 0;
        if (s.n_layers_hit < cfg.min_layers) {
            flags |= SVT_FLAG_BAD_PATTERN;
        } else {
            n = s.C;
            if (s.C > cfg.max_comb) {
                flags |= SVT_FLAG_OVERFLOW;
                n = cfg.max_comb;
            }
        }
        road_flags[r] = flags;
        comb_cnt[r] = n;
    }
}

// ---- exclusive scan of uint64 counts: per-tile sums, one-block scan, apply ----
constexpr int SCAN_THREADS = 256, SCAN_PER = 8, SCAN_TILE = SCAN_THREADS * SCAN_PER;

__global__ void __launch_bounds__(SCAN_THREADS)
    k_scan_u64_reduce(const uint64_t *__restrict__ a, const uint64_t *__restrict__ n_dev,
                      uint64_t cap, uint64_t *tile_sums, const unsigned long long *status) {
    __shared__ unsigned long long red[SCAN_THREADS / 32 + 1];
    wait_prior_grid();
    allow_next_grid();
    if (!status_ok(status)) return;
    const uint64_t n = *n_dev < cap ? *n_dev : cap;
    const uint64_t T = (n + SCAN_TILE - 1) / SCAN_TILE;
    for (uint64_t t = blockIdx.x; t < T; t += gridDim.x) {
        const uint64_t b = t * SCAN_TILE + (uint64_t)threadIdx.x * SCAN_PER;
        unsigned long long s = 0;
#pragma unroll
        for (int j = 0; j < SCAN_PER; ++j) s += (b + j < n) ? a[b + j] : 0ull;
        unsigned long long tot;
        block_exclusive_scan<unsigned long long>(s, red, &tot);
        if (threadIdx.x == 0) tile_sums[t] = tot;
    }
}

__global__ void __launch_bounds__(1024)
    k_scan_u64_tiles(uint64_t *tile_sums, const uint64_t *__restrict__ n_dev, uint64_t cap,
                     const unsigned long long *status) {
    __shared__ unsigned long long sm[33];
    wait_prior_grid();
    allow_next_grid();
    if (!status_ok(status)) return;
    const uint64_t n = *n_dev < cap ? *n_dev : cap;
    const uint64_t T = (n + SCAN_TILE - 1) / SCAN_TILE;
    unsigned long long carry = 0;
    for (uint64_t c0 = 0; c0 < T; c0 += 1024) {
        const uint64_t i = c0 + threadIdx.x;
        unsigned long long v = i < T ? tile_sums[i] : 0ull;
        unsigned long long tot;
        unsigned long long ex = block_exclusive_scan<unsigned long long>(v, sm, &tot);
        if (i < T) tile_sums[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) tile_sums[T] = carry;
}

__global__ void __launch_bounds__(SCAN_THREADS)
    k_scan_u64_apply(uint64_t *a, const uint64_t *__restrict__ n_dev, uint64_t cap,
                     const uint64_t *__restrict__ tile_sums, uint64_t *total,
                     const unsigned long long *status) {
    __shared__ unsigned long long red[SCAN_THREADS / 32 + 1];
    wait_prior_grid();
    allow_next_grid();
    if (!status_ok(status)) return;
    const uint64_t n = *n_dev < cap ? *n_dev : cap;
    const uint64_t T = (n + SCAN_TILE - 1) / SCAN_TILE;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a[n] = tile_sums[T];
        if (total) *total = tile_sums[T];
    }
    for (uint64_t t = blockIdx.x; t < T; t += gridDim.x) {
        const uint64_t b = t * SCAN_TILE + (uint64_t)threadIdx.x * SCAN_PER;
        unsigned long long v[SCAN_PER], s = 0;
#pragma unroll
        for (int j = 0; j < SCAN_PER; ++j) {
            v[j] = (b + j < n) ? a[b + j] : 0ull;
            s += v[j];
        }
        unsigned long long tot;
        unsigned long long run = tile_sums[t] + block_exclusive_scan<unsigned long long>(s, red, &tot);
#pragma unroll
        for (int j = 0; j < SCAN_PER; ++j) {
            if (b + j < n) a[b + j] = run;
            run += v[j];
        }
    }
}

// Per-road metadata of the plain select, read for a group of roads at once
// (one coalesced load per field) instead of road by road.
struct RoadMeta {
    uint64_t off, n;
    uint32_t word;   // road_flags
};

// Every combination of every road, written in order by tiles of WRITE_TILE
// consecutive combinations: thread t of a block takes WRITE_PER consecutive
// ones, finds the road of its first (a search of the tile's offsets, staged in
// shared memory), derives that combination's digits once by
// division and counts them up from there (see the counter below), taking up the next
// road where one ends.  The tiles are equal work whatever the roads' sizes (a
// road per warp, or per block for big ones, left the largest roads running
// alone: 95 us of the scaled workload's 200 events against 26 us), and each
// thread's two runs of 32 bytes leave as 16-byte stores.  The tile's roads are
// found by 32-way searches, three dependent loads where a binary search of the
// 12,800 offsets makes fourteen, and the digits cost about sixteen instructions a
// combination (34 us with binary searches and digits counted one by one).
constexpr int WRITE_THREADS = 256, WRITE_PER = 8, WRITE_TILE = WRITE_THREADS * WRITE_PER;
constexpr uint32_t WRITE_ROADS = 512;   // staged roads of a tile; more are searched in place

// largest r in [lo, hi) with off[r] <= j, given off[lo] <= j: the last of
// several roads at one offset, which is the one that has combinations
__device__ __forceinline__ uint64_t road_of(const uint64_t *off, uint64_t lo, uint64_t hi,
                                            uint64_t j) {
#pragma unroll 1
    while (hi - lo > 1) {
        const uint64_t mid = (lo + hi) >> 1;
        if (off[mid] <= j) lo = mid; else hi = mid;
    }
    return lo;
}
// the same by a warp, 32 offsets a step
__device__ __forceinline__ uint64_t road_of_warp(const uint64_t *__restrict__ off, uint64_t lo,
                                                 uint64_t hi, uint64_t j, uint32_t lane) {
    while (hi - lo > 1) {
        const uint64_t step = (hi - lo + 31) / 32, p = lo + lane * step;
        const uint32_t le = __ballot_sync(0xffffffffu, p < hi && __ldg(off + p) <= j);
        lo += (31u - __clz(le)) * step;   // lane 0's is always set
        hi = min(lo + step, hi);
    }
    return lo;
}

// 16 - n'_l of every layer, layer 5 in the lowest four bits (0 for 16 hits)
__device__ __forceinline__ uint32_t digit_bias(const RoadShape &s) {
    uint32_t b = 0;
#pragma unroll
    for (int l = 0; l < N_LAYERS; ++l) b |= ((16u - s.n[l]) & 15u) << (4 * (N_LAYERS - 1 - l));
    return b;
}

__global__ void __launch_bounds__(WRITE_THREADS)
    k_combine_write(const uint32_t *__restrict__ road_nhit, const uint64_t *__restrict__ n_roads,
                    uint64_t road_cap, const uint64_t *__restrict__ comb_off, uint64_t comb_cap,
                    uint32_t xft_pairs, uint32_t *comb_road, uint32_t *comb_hits,
                    unsigned long long *status) {
    __shared__ uint64_t ends[2];   // roads of the tile's first and last combination
    __shared__ uint64_t off_s[WRITE_ROADS + 1];
    __shared__ uint32_t nhit_s[WRITE_ROADS];
    wait_prior_grid();
    allow_next_grid();
    if (!status_ok(status)) return;
    const uint64_t R = road_count(n_roads, road_cap);
    const uint64_t total = comb_off[R];
    if (total > comb_cap) {   // nothing to write: the status says so
        if (blockIdx.x == 0 && threadIdx.x == 0) report(status, 0, SVT_ERR_OOM);
        return;
    }
    const bool wide = (((uintptr_t)comb_road | (uintptr_t)comb_hits) & 15u) == 0;
    for (uint64_t t0 = (uint64_t)blockIdx.x * WRITE_TILE; t0 < total;
         t0 += (uint64_t)gridDim.x * WRITE_TILE) {
        const uint64_t t1 = min(t0 + (uint64_t)WRITE_TILE, total);
        if (threadIdx.x < 64) {
            const uint64_t r = road_of_warp(comb_off, 0, R, threadIdx.x < 32 ? t0 : t1 - 1,
                                            threadIdx.x & 31u);
            if ((threadIdx.x & 31u) == 0) ends[threadIdx.x >> 5] = r;
        }
        __syncthreads();
        const uint64_t r0 = ends[0], nr = ends[1] - r0 + 1;
        const bool staged = nr <= WRITE_ROADS;
        if (staged) {
            for (uint64_t k = threadIdx.x; k <= nr; k += WRITE_THREADS) {
                off_s[k] = __ldg(comb_off + r0 + k);
                if (k < nr) nhit_s[k] = __ldg(road_nhit + r0 + k);
            }
            __syncthreads();
        }
        // offsets and hits of the tile's roads, by their place from r0
        const uint64_t *off = staged ? off_s : comb_off + r0;
        const uint32_t *nhit = staged ? nhit_s : road_nhit + r0;
        const uint64_t j0 = t0 + (uint64_t)threadIdx.x * WRITE_PER;
        if (j0 < t1) {
            uint64_t r = road_of(off, 0, nr, j0);
            RoadShape s = road_shape(nhit[r], xft_pairs);
            uint64_t end = off[r + 1];
            // The digits as a counter with layer 5 in the lowest four bits, each
            // raised by 16 - n'_l, so that a digit past its layer's last hit carries
            // into the next slower layer by itself and leaves zero, which no raised
            // digit is (unless n'_l = 16, where nothing has to be put back).
            uint32_t rem = (uint32_t)(j0 - off[r]), x = 0, bias = digit_bias(s);
#pragma unroll
            for (int l = N_LAYERS - 1; l >= 0; --l) {
                const uint32_t qd = div_by(rem, s.n[l], kDivMagic[s.n[l]]);
                x |= (rem - qd * s.n[l]) << (4 * (N_LAYERS - 1 - l));
                rem = qd;
            }
            x += bias;
            // combinations up to the road's end (the last of them resets the counter)
            uint32_t left = (uint32_t)min(end - j0, (uint64_t)WRITE_PER + 1);
            uint32_t road[WRITE_PER], hits[WRITE_PER];
#pragma unroll
            for (int i = 0; i < WRITE_PER; ++i) {
                road[i] = (uint32_t)(r0 + r);
                // layer 0 to the lowest bits: the nibbles of each byte and the
                // three bytes change places
                const uint32_t d = x - bias;
                const uint32_t sw = ((d >> 4) & 0x0F0F0Fu) | ((d << 4) & 0xF0F0F0u);
                const uint32_t h = __byte_perm(sw, 0u, 0x4012);
                // with pairs layer 5 (radix 1) takes layer 4's hit
                hits[i] = xft_pairs ? h | (((h >> 16) & 15u) << 20) : h;
                if (--left == 0) {   // the next road that has combinations
                    if (j0 + i + 1 < t1) {
                        // There can be any number of roads without a combination before
                        // it, hence a search (a walk over 190,000 of them took 13 ms;
                        // the whole call now 23 us; doubled steps before the search
                        // cost roads that all have some 2 %).
                        end = off[++r + 1];
                        if (end == j0 + i + 1) {
                            r = road_of(off, r + 1, nr, end);
                            end = off[r + 1];
                        }
                        s = road_shape(nhit[r], xft_pairs);
                        bias = digit_bias(s);
                        left = (uint32_t)min(end - (j0 + i + 1), (uint64_t)WRITE_PER + 1);
                    }
                    x = bias;
                } else {
                    x += 1u;
                    const uint32_t z = ~(x | (x >> 1) | (x >> 2) | (x >> 3)) & 0x111111u;
                    x += bias & (z * 15u);
                }
            }
            if (wide && j0 + WRITE_PER <= t1) {
#pragma unroll
                for (int i = 0; i < WRITE_PER; i += 4) {
                    *reinterpret_cast<uint4 *>(comb_road + j0 + i) =
                        make_uint4(road[i], road[i + 1], road[i + 2], road[i + 3]);
                    *reinterpret_cast<uint4 *>(comb_hits + j0 + i) =
                        make_uint4(hits[i], hits[i + 1], hits[i + 2], hits[i + 3]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < WRITE_PER; ++i)
                    if (j0 + i < t1) {
                        comb_road[j0 + i] = road[i];
                        comb_hits[j0 + i] = hits[i];
                    }
            }
        }
        __syncthreads();   // `ends` is set again for the next tile
    }
}

// A constant row as the fit takes it: F in pairs of 16 bits (F_k,2m low), and
// Q_k = q_k 2^qshift as its low nine bits and the rest (|Q_k| < 2^39).
struct PackedRow {
    int32_t F[18];
    int32_t q_lo[6], q_hi[6];
};
__device__ __forceinline__ int32_t pack_pair(int16_t lo, int16_t hi) {
    return (int32_t)((uint32_t)(uint16_t)lo | ((uint32_t)(uint16_t)hi << 16));
}
__device__ __forceinline__ long long shifted_q(int16_t q, uint32_t qshift) {
    return (long long)((unsigned long long)(long long)q << qshift);
}
// c + a.lo b.byte0 + a.hi b.byte1, and the same with bytes 2 and 3
__device__ __forceinline__ int32_t dot_lo(int32_t a, uint32_t b, int32_t c) {
    int32_t d;
    asm("dp2a.lo.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ int32_t dot_hi(int32_t a, uint32_t b, int32_t c) {
    int32_t d;
    asm("dp2a.hi.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// y_k = floor((Q_k + sum_l F_kl x_l) / 2^oshift) exactly, in 32 bits: with
// x_l = 256 h_l + b_l (x_l < 2^15) the sum is A + 256 B, A and B dot products of
// 16-bit constants and bytes (|A|, |B| < 2^26, two terms an instruction), and
// with Q_k = 512 q_hi + q_lo and oshift >= 9
//   y_k = floor((q_hi + floor((floor((A + q_lo) / 256) + B) / 2)) / 2^(oshift - 9)).
// (Sums of 32-bit products in int64, with rows of half as many constants a word,
// kept the integer pipe 70 % busy: 208 instructions a combination.  7.4 M
// combinations: 56.2 us then, 48.9 now, 26 for the bytes.)  Results: chi2 over
// the three clamped chi rows, p_0..p_2.
__device__ __forceinline__ uint32_t fit_rows(const PackedRow &row, const uint32_t (&x)[N_LAYERS],
                                             uint32_t oshift, int32_t (&p)[3]) {
    const uint32_t x01 = __byte_perm(x[0], x[1], 0x5410), x23 = __byte_perm(x[2], x[3], 0x5410);
    const uint32_t b03 = __byte_perm(x01, x23, 0x6420), h03 = __byte_perm(x01, x23, 0x7531);
    // b_4, b_5, h_4, h_5
    const uint32_t x45 = __byte_perm(x[4], x[5], 0x5140);
    int32_t y[N_LAYERS];
#pragma unroll
    for (int k = 0; k < N_LAYERS; ++k) {
        const int32_t *Fk = row.F + 3 * k;
        int32_t v = dot_lo(Fk[2], x45, dot_hi(Fk[1], b03, dot_lo(Fk[0], b03, row.q_lo[k])));
        v = dot_hi(Fk[2], x45, dot_hi(Fk[1], h03, dot_lo(Fk[0], h03, v >> 8)));
        y[k] = (row.q_hi[k] + (v >> 1)) >> (oshift - 9u);
    }
    uint32_t chi2 = 0;
#pragma unroll
    for (int k = 3; k < N_LAYERS; ++k) {
        const int32_t c = max(min(y[k], 32767), -32767);
        chi2 += (uint32_t)(c * c);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k] = y[k];
    return chi2;
}

// One combination with every input read from global memory (road data, hit
// words, the sector/pattern row of the constants).
__device__ __forceinline__ uint32_t fit_direct(const uint32_t *__restrict__ words,
                                               const uint32_t *__restrict__ road_word,
                                               const uint32_t *__restrict__ road_nhit,
                                               const int16_t *__restrict__ F,
                                               const int16_t *__restrict__ q,
                                               const svt_config &cfg, uint32_t r, uint32_t hits,
                                               int32_t (&p)[3]) {
    const uint32_t rw = __ldg(road_word + r);
    const uint32_t packed = __ldg(road_nhit + r);
    const uint32_t hw = __ldg(words + rw);
    uint32_t mask = 0, hoff = rw + 1;
    uint32_t x[N_LAYERS];
#pragma unroll
    for (int l = 0; l < N_LAYERS; ++l) {
        const uint32_t nl = nhit_of(packed, l);
        x[l] = nl ? hit_coord(__ldg(words + hoff + ((hits >> (4 * l)) & 15u))) : 0u;
        mask |= nl ? (1u << l) : 0u;
        hoff += nl;
    }
    const size_t cs = (size_t)rd_sector(hw) * 64 + mask;
    PackedRow row;
#pragma unroll
    for (int i = 0; i < 18; ++i)
        row.F[i] = pack_pair(__ldg(F + cs * 36 + 2 * i), __ldg(F + cs * 36 + 2 * i + 1));
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const long long Q = shifted_q(__ldg(q + cs * 6 + k), cfg.qshift);
        row.q_lo[k] = (int32_t)(Q & 511);
        row.q_hi[k] = (int32_t)(Q >> 9);
    }
    return fit_rows(row, x, cfg.oshift, p);
}

// A road's row staged in shared memory by the plain fit: its constants and, per
// layer, the index of its first hit in the road's coordinate list (0xFF for a
// layer without hits); the road's hit coordinates sit beside it (at most 96: 6
// layers x 16).
constexpr int FIT_THREADS = 256;
constexpr int FIT_PER_THREAD = 8;
constexpr int FIT_TILE = FIT_THREADS * FIT_PER_THREAD;   // combinations per block tile
constexpr int FIT_STAGE_ROADS = 64;   // tiles over more roads read their inputs directly
struct alignas(16) StagedRow {
    PackedRow row;
    uint8_t first[8];
};
static_assert(sizeof(StagedRow) == 128 && sizeof(PackedRow) == 120, "read as eight 16-byte words");

__device__ __forceinline__ uint32_t fit_staged(const StagedRow &row,
                                               const uint16_t *__restrict__ coord,
                                               uint32_t oshift, uint32_t hits, int32_t (&p)[3]) {
    uint4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = reinterpret_cast<const uint4 *>(&row)[i];
    PackedRow r;
    const uint32_t *const w = reinterpret_cast<const uint32_t *>(v);
#pragma unroll
    for (int i = 0; i < 18; ++i) r.F[i] = (int32_t)w[i];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        r.q_lo[k] = (int32_t)w[18 + k];
        r.q_hi[k] = (int32_t)w[24 + k];
    }
    uint32_t x[N_LAYERS];
#pragma unroll
    for (int l = 0; l < N_LAYERS; ++l) {
        const uint32_t f0 = (w[30 + l / 4] >> (8 * (l & 3))) & 0xFFu;
        x[l] = f0 != 0xFFu ? coord[f0 + ((hits >> (4 * l)) & 15u)] : 0u;
    }
    return fit_rows(r, x, oshift, p);
}

// One thread per combination, over block tiles of FIT_TILE consecutive
// combinations (thread t takes combinations t, t + 256, t + 512, ... of the
// tile and loads their entries first; six blocks per SM, 48.9 us for 7.4 M
// combinations, with five 50.1, with three 54.1).  Combinations are road-major, so a
// tile covers the roads comb_road[first] .. comb_road[last]; when there are
// at most FIT_STAGE_ROADS of them, their rows and hit coordinates are staged
// in shared memory once (coalesced loads) and the combinations of the tile
// need no other global load; otherwise each reads its inputs directly.
__global__ void __launch_bounds__(FIT_THREADS, 6)
    k_fit_plain(const uint32_t *__restrict__ words, const uint32_t *__restrict__ road_word,
                const uint32_t *__restrict__ road_nhit, const uint32_t *__restrict__ comb_road,
                const uint32_t *__restrict__ comb_hits, const uint64_t *__restrict__ n_combs,
                uint64_t comb_cap, const int16_t *__restrict__ F, const int16_t *__restrict__ q,
                const svt_config cfg, uint32_t *fit_chi2, int32_t *fit_par,
                const unsigned long long *status) {
    __shared__ StagedRow rows[FIT_STAGE_ROADS];
    __shared__ uint16_t coords[FIT_STAGE_ROADS][N_LAYERS * MAX_HITS];
    __shared__ uint32_t tile_r0, tile_nr;
    wait_prior_grid();
    allow_next_grid();
    if (!status_ok(status)) return;
    const uint64_t n = *n_combs < comb_cap ? *n_combs : comb_cap;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (uint64_t j0 = (uint64_t)blockIdx.x * FIT_TILE; j0 < n; j0 += (uint64_t)gridDim.x * FIT_TILE) {
        const uint64_t j1 = min(j0 + (uint64_t)FIT_TILE, n);
        uint32_t rr[FIT_PER_THREAD], hh[FIT_PER_THREAD];
#pragma unroll
        for (int i = 0; i < FIT_PER_THREAD; ++i) {
            const uint64_t j = j0 + (uint64_t)(i * FIT_THREADS) + threadIdx.x;
            rr[i] = j < j1 ? __ldg(comb_road + j) : 0u;
            hh[i] = j < j1 ? __ldg(comb_hits + j) : 0u;
        }
        if (threadIdx.x == 0) {
            const uint32_t r0 = __ldg(comb_road + j0), r1 = __ldg(comb_road + j1 - 1);
            tile_r0 = r0;
            tile_nr = r1 - r0 + 1;   // roads are non-decreasing in j
        }
        __syncthreads();
        const uint32_t r0 = tile_r0, nr = tile_nr;
        const bool staged = nr <= (uint32_t)FIT_STAGE_ROADS;
        if (staged) {
            // warp w stages roads w, w + 8, ...: lanes 0..17 the F row, 18..23
            // the q row, 24..29 the layers, and every lane some of the hit
            // coordinates
            for (uint32_t rho = warp; rho < nr; rho += FIT_THREADS / 32) {
                const uint32_t r = r0 + rho;
                const uint32_t rw = __ldg(road_word + r), packed = __ldg(road_nhit + r);
                uint32_t mask = 0, total = 0;
#pragma unroll
                for (int l = 0; l < N_LAYERS; ++l) {
                    mask |= nhit_of(packed, l) ? (1u << l) : 0u;
                    total += nhit_of(packed, l);
                }
                total = min(total, (uint32_t)(N_LAYERS * MAX_HITS));
                const size_t cs = (size_t)rd_sector(__ldg(words + rw)) * 64 + mask;
                StagedRow &row = rows[rho];
                if (lane < 18) {
                    row.row.F[lane] = pack_pair(__ldg(F + cs * 36 + 2 * lane),
                                                __ldg(F + cs * 36 + 2 * lane + 1));
                } else if (lane < 24) {
                    const int k = lane - 18;
                    const long long Q = shifted_q(__ldg(q + cs * 6 + k), cfg.qshift);
                    row.row.q_lo[k] = (int32_t)(Q & 511);
                    row.row.q_hi[k] = (int32_t)(Q >> 9);
                } else if (lane < 24 + N_LAYERS) {
                    const int l = lane - 24;
                    uint32_t before = 0;   // hits on the layers below l
#pragma unroll
                    for (int m = 0; m < N_LAYERS - 1; ++m) before += m < l ? nhit_of(packed, m) : 0u;
                    row.first[l] = nhit_of(packed, l) ? (uint8_t)before : (uint8_t)0xFF;
                }
                for (uint32_t h = lane; h < total; h += 32)
                    coords[rho][h] = (uint16_t)hit_coord(__ldg(words + rw + 1 + h));
            }
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < FIT_PER_THREAD; ++i) {
            const uint64_t j = j0 + (uint64_t)(i * FIT_THREADS) + threadIdx.x;
            if (j < j1) {
                int32_t p[3];
                const uint32_t chi2 =
                    staged ? fit_staged(rows[rr[i] - r0], coords[rr[i] - r0], cfg.oshift, hh[i], p)
                           : fit_direct(words, road_word, road_nhit, F, q, cfg, rr[i], hh[i], p);
                fit_chi2[j] = chi2;
#pragma unroll
                for (int k = 0; k < 3; ++k) fit_par[k * comb_cap + j] = p[k];
            }
        }
        __syncthreads();   // rows are reused by the next tile
    }
}

// Best passing combination of a road from its chi2 values, over the threads
// idx, idx + STEP, ... (a warp, or the block): each visits its combinations in
// increasing c, sixteen loads in flight, so a strict '<' keeps the smallest
// index among equal chi2.  Returns this thread's key (chi2 << 32) | c.
template <uint32_t STEP>
__device__ __forceinline__ unsigned long long scan_chi2(const uint32_t *__restrict__ chi2,
                                                        uint64_t n, uint32_t init_chi,
                                                        uint32_t idx) {
    constexpr int U = 16;
    uint32_t bchi = init_chi, bc = 0;
    for (uint64_t c0 = idx; c0 < n; c0 += (uint64_t)U * STEP) {
        uint32_t v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t c = c0 + (uint64_t)u * STEP;
            v[u] = c < n ? __ldg(chi2 + c) : 0xFFFFFFFFu;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (v[u] < bchi) {
                bchi = v[u];
                bc = (uint32_t)c0 + (uint32_t)u * STEP;
            }
    }
    return bchi != init_chi ? (((unsigned long long)bchi << 32) | bc) : ~0ull;
}

__device__ __forceinline__ unsigned long long warp_min_key(unsigned long long key) {
    const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(key >> 32));
    const uint32_t lo = __reduce_min_sync(
        0xffffffffu, (uint32_t)(key >> 32) == hi ? (uint32_t)key : 0xFFFFFFFFu);
    return ((unsigned long long)hi << 32) | lo;
}

// Chi-square cut and best combination of each road.  A block takes a group of
// consecutive roads at a time: its warps share those of at most SELECT_BIG
// combinations, then the whole block scans each longer one.  Bound at the end by
// the longest road's block, hence the sixteen loads: with eight the scaled
// workload's 200 events (12,800 roads, one of 100 thousand combinations) take
// 33 us instead of 22; blocks of 512 or 1024 threads take 26 to 34, groups of 8 to
// 64 roads 22 to 32.  Where the roads are short on the mean nothing is left to
// wait for, and what counts is the latency of a group: there a group holds as many
// roads as give every block one (at most SELECT_GROUP_MAX).  Roads of at most 64
// combinations take two loads a lane.  In us, one warp per road over the whole
// grid / groups of 16 from a counter in the block / now: 200,000 roads of one
// combination 49 / 89 / 21, 96,000 of 64 27 / 44 / 14, 128,000 of 729 95 / 86 / 67,
// the scaled workload 49 / 16.4 / 14.9 (without the rest of the stages).
constexpr uint32_t SELECT_THREADS = 256, SELECT_GROUP = 16, SELECT_BIG = 1024;
constexpr uint32_t SELECT_GROUP_MAX = 128, SELECT_SMALL_MEAN = 128;
__global__ void __launch_bounds__(SELECT_THREADS)
    k_select(const uint32_t *__restrict__ fit_chi2, const int32_t *__restrict__ fit_par,
             uint64_t comb_cap, const uint64_t *__restrict__ comb_off,
             const uint32_t *__restrict__ road_flags, const uint64_t *__restrict__ n_roads,
             uint64_t road_cap, const svt_config cfg, svt_best *best,
             const unsigned long long *status) {
    __shared__ RoadMeta meta[SELECT_GROUP_MAX];
    __shared__ unsigned long long key_s[SELECT_GROUP_MAX];
    wait_prior_grid();
    allow_next_grid();
    if (!status_ok(status)) return;
    const uint64_t R = road_count(n_roads, road_cap);
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t init_chi = cfg.chi2_cut == 0xFFFFFFFFu ? 0xFFFFFFFFu : cfg.chi2_cut + 1u;
    uint32_t group = SELECT_GROUP;
    if (R && __ldg(comb_off + R) < R * SELECT_SMALL_MEAN)
        group = (uint32_t)max((uint64_t)SELECT_GROUP,
                              min((R + gridDim.x - 1) / gridDim.x, (uint64_t)SELECT_GROUP_MAX));
    for (uint64_t g = (uint64_t)blockIdx.x * group; g < R; g += (uint64_t)gridDim.x * group) {
        const uint32_t n = (uint32_t)min((uint64_t)group, R - g);
        bool big = false;
        if (threadIdx.x < n) {
            RoadMeta m;
            m.off = __ldg(comb_off + g + threadIdx.x);
            m.n = __ldg(comb_off + g + threadIdx.x + 1) - m.off;
            m.word = __ldg(road_flags + g + threadIdx.x);
            if (m.off + m.n > comb_cap) m.n = 0;   // (an error status by now)
            big = m.n > SELECT_BIG;
            meta[threadIdx.x] = m;
            key_s[threadIdx.x] = ~0ull;
        }
        big = __syncthreads_or(big);
        for (uint32_t k = threadIdx.x >> 5; k < n; k += SELECT_THREADS / 32) {
            const RoadMeta m = meta[k];
            if (m.n == 0 || m.n > SELECT_BIG) continue;
            unsigned long long key;
            if (m.n <= 64) {
                const uint32_t *chi2 = fit_chi2 + m.off;
                const uint32_t v0 = lane < m.n ? __ldg(chi2 + lane) : 0xFFFFFFFFu;
                const uint32_t v1 = lane + 32 < m.n ? __ldg(chi2 + lane + 32) : 0xFFFFFFFFu;
                const uint32_t v = min(v0, v1), c = v0 <= v1 ? lane : lane + 32;
                key = v < init_chi ? ((unsigned long long)v << 32) | c : ~0ull;
            } else {
                key = scan_chi2<32>(fit_chi2 + m.off, m.n, init_chi, lane);
            }
            key = warp_min_key(key);
            if (lane == 0) key_s[k] = key;
        }
        for (uint32_t k = 0; big && k < n; ++k) {
            const RoadMeta m = meta[k];
            if (m.n <= SELECT_BIG) continue;   // uniform over the block
            const unsigned long long key = warp_min_key(
                scan_chi2<SELECT_THREADS>(fit_chi2 + m.off, m.n, init_chi, threadIdx.x));
            if (lane == 0) atomicMin(&key_s[k], key);
        }
        __syncthreads();
        if (threadIdx.x < n) {
            const RoadMeta m = meta[threadIdx.x];
            const unsigned long long key = key_s[threadIdx.x];
            svt_best b;
            b.flags = m.word;
            b.comb = 0xFFFFFFFFu;
            b.chi2 = 0;
            b.p[0] = b.p[1] = b.p[2] = 0;
            if (key != ~0ull) {
                const uint32_t c = (uint32_t)key;
                b.flags |= SVT_FLAG_PASS;
                b.comb = c;
                b.chi2 = (uint32_t)(key >> 32);
                b.p[0] = fit_par[m.off + c];
                b.p[1] = fit_par[comb_cap + m.off + c];
                b.p[2] = fit_par[2 * comb_cap + m.off + c];
            }
            best[g + threadIdx.x] = b;
        }
        __syncthreads();   // the group's tables are rebuilt for the next one
    }
}

__global__ void k_format(const svt_best *__restrict__ best, const uint32_t *__restrict__ words,
                         const uint32_t *__restrict__ road_word,
                         const uint64_t *__restrict__ n_roads, uint64_t road_cap, uint32_t *out,
                         const unsigned long long *status) {
    wait_prior_grid();
    allow_next_grid();
    if (!status_ok(status)) return;
    const uint64_t R = road_count(n_roads, road_cap);
    for (uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r < R;
         r += (uint64_t)gridDim.x * blockDim.x) {
        const svt_best b = best[r];
        const uint32_t hw = __ldg(words + road_word[r]);
        uint32_t *o = out + r * 6;
        o[0] = rd_id(hw) | (b.flags << 24);
        o[1] = b.comb;
        o[2] = b.chi2;
        o[3] = (uint32_t)b.p[0];
        o[4] = (uint32_t)b.p[1];
        o[5] = (uint32_t)b.p[2];
    }
}

int grid_for(uint64_t n, int threads, int max_grid) {
    uint64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    return (int)(b < (uint64_t)max_grid ? b : (uint64_t)max_grid);
}

}  // namespace

void launch_combine_count(const uint32_t *road_nhit, const uint64_t *n_roads, uint64_t road_cap,
                          const svt_config cfg, uint32_t *road_flags, uint64_t *comb_cnt,
                          const unsigned long long *status, int grid, cudaStream_t st) {
    launch_after(k_combine_count, grid_for(road_cap, 256, grid), 256, 0, st, road_nhit, n_roads,
                 road_cap, cfg, road_flags, comb_cnt, status);
}

void launch_scan_u64(uint64_t *a, const uint64_t *n_dev, uint64_t cap, uint64_t *tile_sums,
                     uint64_t *total, const unsigned long long *status, int grid, cudaStream_t st) {
    int g = grid_for(cap, SCAN_TILE, grid);
    launch_after(k_scan_u64_reduce, g, SCAN_THREADS, 0, st, (const uint64_t *)a, n_dev, cap,
                 tile_sums, status);
    launch_after(k_scan_u64_tiles, 1, 1024, 0, st, tile_sums, n_dev, cap, status);
    launch_after(k_scan_u64_apply, g, SCAN_THREADS, 0, st, a, n_dev, cap,
                 (const uint64_t *)tile_sums, total, status);
}

size_t scan_u64_tile_count(uint64_t cap) { return (cap + SCAN_TILE - 1) / SCAN_TILE + 1; }

void launch_combine_write(const uint32_t *road_nhit, const uint64_t *n_roads, uint64_t road_cap,
                          const uint64_t *comb_off, uint64_t comb_cap, uint32_t xft_pairs,
                          uint32_t *comb_road, uint32_t *comb_hits, unsigned long long *status,
                          int grid, cudaStream_t st) {
    launch_after(k_combine_write, grid_for((comb_cap + WRITE_PER - 1) / WRITE_PER, WRITE_THREADS, grid),
                 WRITE_THREADS, 0, st, road_nhit, n_roads, road_cap, comb_off, comb_cap, xft_pairs,
                 comb_road, comb_hits, status);
}

void launch_fit_plain(const uint32_t *words, const uint32_t *road_word, const uint32_t *road_nhit,
                      const uint32_t *comb_road, const uint32_t *comb_hits,
                      const uint64_t *n_combs, uint64_t comb_cap, const int16_t *F,
                      const int16_t *q, const svt_config cfg, uint32_t *fit_chi2,
                      int32_t *fit_par, const unsigned long long *status, int grid,
                      cudaStream_t st) {
    launch_after(k_fit_plain,
                 grid_for((comb_cap + FIT_TILE - 1) / FIT_TILE * FIT_THREADS, FIT_THREADS, grid),
                 FIT_THREADS, 0, st, words, road_word, road_nhit, comb_road, comb_hits, n_combs,
                 comb_cap, F, q, cfg, fit_chi2, fit_par, status);
}

void launch_select(const uint32_t *fit_chi2, const int32_t *fit_par, uint64_t comb_cap,
                   const uint64_t *comb_off, const uint32_t *road_flags, const uint64_t *n_roads,
                   uint64_t road_cap, const svt_config cfg, svt_best *best,
                   const unsigned long long *status, int grid, cudaStream_t st) {
    launch_after(k_select, grid_for(road_cap, SELECT_GROUP, grid), SELECT_THREADS, 0, st, fit_chi2,
                 fit_par, comb_cap, comb_off, road_flags, n_roads, road_cap, cfg, best, status);
}

void launch_format(const svt_best *best, const uint32_t *words, const uint32_t *road_word,
                   const uint64_t *n_roads, uint64_t road_cap, uint32_t *out,
                   const unsigned long long *status, int grid, cudaStream_t st) {
    launch_after(k_format, grid_for(road_cap, 256, grid), 256, 0, st, best, words, road_word, n_roads,
                 road_cap, out, status);
}

}  // namespace svt
