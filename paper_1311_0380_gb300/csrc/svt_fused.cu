// svt_fused.cu -- combine + fit + chi-square cut + best-per-road + format of
// the paper's Sec. 2 / Sec. 2.1 in one persistent kernel.
//
// Design (GB300 first; the paper's Kepler port used one thread per
// combination and a separate kernel per stage):
//   * The fit is linear, so with the layers split into a prefix (rows, index
//     a) and a suffix (columns, index b) every accumulator is
//         acc_k(a, b) = A_k(a) + B_k(b),
//     A_k(a) = q_k 2^qshift + sum_{prefix l} F_kl x_l,  B_k(b) = sum_{suffix l} F_kl x_l,
//     exactly in int64.  A warp builds the per-hit terms F_kl x_l and up to 64
//     A rows in shared memory; each lane holds the B of one column in
//     registers.  One combination then costs three 64-bit adds, a 16-bit
//     range test, three multiply-adds and one compare-select (the high word
//     of each sum is y_k + 32768; see eval_rows).  Only the three chi rows are
//     evaluated in the loop; the parameters are formed once for the winning
//     combination.
//   * Work: roads with more than small_max evaluated combinations are split
//     into items of `rows` rows and handled first (items taken from an atomic
//     counter; the road of an item is found by a 32-way warp search of the
//     short list of split roads).  Then warps take chunks of consecutive
//     roads (one coalesced load of their 32-byte descriptors) and fit every
//     remaining road whole, one warp per road; with the grouped instances two
//     consecutive SMALL roads of the same geometry go to the two halves of a
//     warp instead, or four TINY ones to its four quarters, or every TINY road
//     of the chunk to a lane of its own (see lane_fit).
//   * Each lane visits its combinations in increasing c within a column (or
//     within its block of rows of a column), so a strict '<' keeps the
//     smallest index among equal chi2; across columns, row blocks, lanes and
//     items the (chi2, c) pairs are merged as 64-bit keys (warp
//     shuffles; atomicMin on the road's key for split roads, which the warp
//     that retires the road's last item takes over).
//   * A warp lists the roads it has finished with their keys and, 31 or 32
//     at a time, writes their records one road per lane: recovering the hits
//     of the best combination and forming its three parameters is scalar
//     work that would otherwise hold all 32 lanes for every road.
#include <algorithm>
#include <cmath>

#include "svt_kernels.cuh"

namespace svt {

namespace {

constexpr int ROWS_MAX = 64;

// A road's working set in shared memory, for roads with at most MH hits on
// every layer, NS suffix-table entries and NR rows per chunk.  All
// accumulator terms are kept multiplied by 2^(32 - oshift): the high word of a
// 64-bit sum of such terms is then exactly floor(sum / 2^oshift).
template <int MH, int NS, int NR>
struct RoadSmem {
    longlong2 T[N_LAYERS * MH][2];  // chi-row terms F[3+k][l] * x * 2^(32-oshift) of hit i of
                                    // layer l at [l*MH+i]: (k=3, k=4), (k=5, -); 32-byte entries
                                    // so a lookup is one 16-byte and one 8-byte load
    longlong2 S01[NS];              // suffix sums below the top suffix layer, rows 3, 4 [b']
    long long S5[NS];               // ... row 5
    longlong2 A01[NR];              // prefix sums incl. q, rows 3, 4, per row of the chunk
    long long A5[NR];               // ... row 5
    uint32_t x[N_LAYERS * MH];      // hit coordinates [l][i] (x = 0 for an empty layer)
    int32_t F[36];                  // F[s][m][k][l] at k*6+l (chi rows k = 3..5 only)
    int32_t q[6];                   // ... q[s][m][k] (k = 3..5 only)
    uint32_t n[N_LAYERS];           // n'_l = max(n_l, 1)
    uint32_t m[N_LAYERS];           // division magic of n'_l
    uint32_t off[N_LAYERS];         // index of the first hit of layer l in the road
    static constexpr uint32_t kMH = MH, kNR = NR;
};
// one road per warp; or two roads marked SMALL, one per half warp, each in
// half of the same space; or four roads marked TINY, one per quarter warp,
// each in a quarter of it
using WarpSmem = RoadSmem<MAX_HITS, 32, ROWS_MAX>;
using HalfSmem = RoadSmem<8, 16, 16>;
using QuarterSmem = RoadSmem<2, 16, 8>;
static_assert(2 * sizeof(HalfSmem) <= sizeof(WarpSmem), "two half slots fit in a warp slot");
static_assert(4 * sizeof(QuarterSmem) <= sizeof(WarpSmem), "four quarter slots fit in a warp slot");
static_assert(sizeof(HalfSmem) % 16 == 0, "half slots keep 16-byte alignment");
static_assert(sizeof(QuarterSmem) % 16 == 0, "quarter slots keep 16-byte alignment");
static_assert(sizeof(WarpSmem) % 16 == 0, "warp slots keep 16-byte alignment");
static_assert(sizeof(WarpSmem) >= 32 * 6 * sizeof(uint32_t), "a road slot holds 32 records");

// A warp's slot when each lane fits a TINY road alone (lane_fit): the lane's
// column sums B_k(b), at most 8 columns, in column j of the tables.
struct LaneTables {
    longlong2 B01[8][32];   // B_3(b), B_4(b) of lane j at [b][j]
    long long B5[8][32];    // B_5(b)
};
constexpr size_t SLOT_BYTES =
    sizeof(WarpSmem) > sizeof(LaneTables) ? sizeof(WarpSmem) : sizeof(LaneTables);
static_assert(SLOT_BYTES % 16 == 0, "slots keep 16-byte alignment");

// Roads a warp has finished but whose records it has not yet written: when 31
// or 32 are listed (and when the warp runs out of work) each lane writes one
// (write_record), so the per-road tail costs a lane rather than a warp.
struct RecordList {
    unsigned long long key[32];   // best key (UINT64_MAX: none passed)
    uint32_t road[32];
};
constexpr uint32_t GEO_SMALL = 1u << 28, GEO_TINY = 1u << 29;

// The W lanes (the warp, or one half of it) that fit one road.  Every
// warp-synchronous step of the per-road code names only these lanes, so the
// two halves of a warp may run their roads' loops with different trip counts.
template <int W>
struct Lanes {
    uint32_t gl;     // lane within the group
    uint32_t mask;   // the group's lanes
};
template <int W>
__device__ __forceinline__ Lanes<W> lanes_of(int lane) {
    Lanes<W> L;
    L.gl = (uint32_t)lane & (uint32_t)(W - 1);
    L.mask = W == 32 ? 0xffffffffu
                     : (((1u << W) - 1u) << ((uint32_t)lane & (uint32_t)(32 - W)));
    return L;
}

// largest j in [0, n) with off[j] <= it (off non-decreasing, off[0] = 0)
__device__ __forceinline__ uint32_t find_slot(const uint32_t *__restrict__ off, uint32_t n,
                                              uint32_t it, int lane) {
    uint32_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const uint32_t step = (hi - lo + 31) / 32;
        const uint32_t p = lo + (uint32_t)lane * step;
        const bool le = (p < hi) && (__ldg(off + p) <= it);
        const uint32_t bal = __ballot_sync(0xffffffffu, le);
        const uint32_t L = 31 - __clz(bal);
        lo = lo + L * step;
        hi = min(lo + step, hi);
    }
    return lo;
}

// Smallest 64-bit key over the group: the smallest high word, then the
// smallest low word among the lanes that hold it.
template <int W>
__device__ __forceinline__ unsigned long long group_min64(unsigned long long v,
                                                          const Lanes<W> &L) {
    const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
    uint32_t m_hi, m_lo;
    if constexpr (W == 32) {
        m_hi = __reduce_min_sync(0xffffffffu, hi);
        m_lo = __reduce_min_sync(0xffffffffu, hi == m_hi ? lo : 0xFFFFFFFFu);
    } else {
        m_hi = hi;
#pragma unroll
        for (int d = W / 2; d >= 1; d >>= 1) m_hi = min(m_hi, __shfl_xor_sync(L.mask, m_hi, d, W));
        m_lo = hi == m_hi ? lo : 0xFFFFFFFFu;
#pragma unroll
        for (int d = W / 2; d >= 1; d >>= 1) m_lo = min(m_lo, __shfl_xor_sync(L.mask, m_lo, d, W));
    }
    return ((unsigned long long)m_hi << 32) | m_lo;
}

__device__ __forceinline__ int32_t clamp_chi(int32_t y) { return max(min(y, 32767), -32767); }


// Road geometry unpacked from its descriptor (uniform over the road's lanes).
struct Geo {
    uint32_t split, NBp, NB, NA, C_eval, mask, total_hits;
};
__device__ __forceinline__ Geo geo_of(const RoadDesc &D) {
    Geo g;
    const uint32_t w = D.b.x;
    g.split = w & 7u;
    g.NBp = (w >> 3) & 31u;
    g.mask = (w >> 13) & 63u;
    g.total_hits = (w >> 19) & 127u;
    g.NB = D.b.y;
    g.NA = D.b.z;
    g.C_eval = D.a.w;
    return g;
}

// Constants, hit coordinates, per-hit chi terms and the suffix table of road D
// in the group's slot.  Global loads are issued before any shared-memory work.
// A road has at most 96 hits (at most 48 in a half slot: 8 per layer), so
// three passes of W = 32 lanes, or of W = 16 lanes over a SMALL road, hold
// them all.
template <int W, typename SM>
__device__ __forceinline__ void road_setup(SM &sm, const uint32_t *__restrict__ words,
                                           const RoadDesc &D, const Geo &g,
                                           const int16_t *__restrict__ F,
                                           const int16_t *__restrict__ q, uint32_t sh,
                                           uint32_t xft, long long bias, const Lanes<W> &L) {
    constexpr uint32_t MH = SM::kMH;
    // the chi rows k = 3..5 only (18 + 3 constants): the record's parameter
    // rows are read from global memory by the lane that forms it
    constexpr int NFQ = (21 + W - 1) / W;
    const uint32_t rw = D.a.x, packed = D.a.y, gl = L.gl;
    const size_t cs = (size_t)rd_sector(D.a.z) * 64 + g.mask;
    int32_t fv[NFQ];
#pragma unroll
    for (int j = 0; j < NFQ; ++j) {
        const uint32_t e = gl + (uint32_t)W * j;
        fv[j] = e < 18 ? __ldg(F + cs * 36 + 18 + e) : (e < 21 ? __ldg(q + cs * 6 + e - 15) : 0);
    }
    uint32_t hv[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const uint32_t h = gl + (uint32_t)W * j;
        hv[j] = h < g.total_hits ? __ldg(words + rw + 1 + h) : 0u;
    }
#pragma unroll
    for (int j = 0; j < NFQ; ++j) {
        const uint32_t e = gl + (uint32_t)W * j;
        if (e < 18) sm.F[18 + e] = fv[j];
        else if (e < 21) sm.q[e - 15] = fv[j];
    }
    const uint32_t nl = gl < N_LAYERS ? nhit_of(packed, gl) : 0u;
    uint32_t incl = nl;   // inclusive prefix of the layer counts
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) {
        const uint32_t v = __shfl_up_sync(L.mask, incl, d, W);
        if (gl >= (uint32_t)d) incl += v;
    }
    if (gl < N_LAYERS) {
        // with track-trigger pairs layer 5 is no digit of its own (radix 1)
        const uint32_t np = (nl && !(xft && gl == N_LAYERS - 1)) ? nl : 1u;
        sm.n[gl] = np;
        sm.m[gl] = kDivMagic[np];
        sm.off[gl] = incl - nl;
        if (nl == 0) {   // a layer without hits contributes x = 0
            sm.x[gl * MH] = 0;
            sm.T[gl * MH][0] = make_longlong2(0, 0);
            sm.T[gl * MH][1].x = 0;
        }
    }
    __syncwarp(L.mask);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const uint32_t h = gl + (uint32_t)W * j;
        if (h < g.total_hits) {
            const uint32_t l = hit_layer(hv[j]);
            const uint32_t i = h - sm.off[l];   // hits are sorted by layer (validated)
            const uint32_t xc = hit_coord(hv[j]);
            sm.x[l * MH + i] = xc;
            longlong2 *t = sm.T[l * MH + i];
            t[0] = make_longlong2((long long)(sm.F[18 + l] * (int32_t)xc) << sh,
                                  (long long)(sm.F[24 + l] * (int32_t)xc) << sh);
            t[1].x = (long long)(sm.F[30 + l] * (int32_t)xc) << sh;
        }
    }
    __syncwarp(L.mask);
    if (xft) {
        // pair i: layer 4's entry i carries both coordinates of track-trigger
        // track i (equal counts are validated); layer 5 then adds nothing
        const uint32_t n4 = nhit_of(packed, 4);
        if (gl < n4) {
            longlong2 *t4 = sm.T[4 * MH + gl];
            const longlong2 *t5 = sm.T[5 * MH + gl];
            t4[0].x += t5[0].x;
            t4[0].y += t5[0].y;
            t4[1].x += t5[1].x;
        }
        __syncwarp(L.mask);
        if (gl == 0) {
            sm.T[5 * MH][0] = make_longlong2(0, 0);
            sm.T[5 * MH][1].x = 0;
        }
    }
    __syncwarp(L.mask);
    // S[b'] = bias + sum over the suffix layers below the top one, b' < NBp
    // (< 32; <= 16 for a SMALL road)
    // (NBp <= W for whole and half warps; a quarter warp takes two passes)
    for (uint32_t bp = gl; bp < g.NBp; bp += (uint32_t)W) {
        uint32_t rem = bp;
        long long S3 = bias, S4 = bias, S5 = bias;
#pragma unroll
        for (int l = N_LAYERS - 1; l >= 1; --l) {
            if ((uint32_t)l > g.split) {
                const uint32_t nl = sm.n[l];
                const uint32_t qd = div_by(rem, nl, sm.m[l]);
                const uint32_t i = rem - qd * nl;
                rem = qd;
                const longlong2 t01 = sm.T[l * MH + i][0];
                S3 += t01.x;
                S4 += t01.y;
                S5 += sm.T[l * MH + i][1].x;
            }
        }
        sm.S01[bp] = make_longlong2(S3, S4);
        sm.S5[bp] = S5;
    }
    __syncwarp(L.mask);
}

template <typename SM>
__device__ __forceinline__ void build_row(SM &sm, uint32_t split, uint32_t a, uint32_t slot,
                                          uint32_t qsh) {
    constexpr uint32_t MH = SM::kMH;
    uint32_t rem = a;
    long long A3 = (long long)sm.q[3] << qsh;
    long long A4 = (long long)sm.q[4] << qsh;
    long long A5 = (long long)sm.q[5] << qsh;
#pragma unroll
    for (int l = N_LAYERS - 1; l >= 0; --l) {
        if ((uint32_t)l < split) {
            const uint32_t nl = sm.n[l];
            const uint32_t qd = div_by(rem, nl, sm.m[l]);
            const uint32_t i = rem - qd * nl;
            rem = qd;
            const longlong2 t01 = sm.T[l * MH + i][0];
            A3 += t01.x;
            A4 += t01.y;
            A5 += sm.T[l * MH + i][1].x;
        }
    }
    sm.A01[slot] = make_longlong2(A3, A4);
    sm.A5[slot] = A5;
}

__device__ __forceinline__ int32_t hi_word(long long v) {
    return (int32_t)((unsigned long long)v >> 32);
}

// Bias carried by the column terms (in the suffix table): with GUARDED the
// high word of a sum is g_k = y_k + 32768 (mod 2^32) instead of y_k.
template <bool GUARDED>
constexpr long long kColBias = GUARDED ? (32768LL << 32) : 0LL;

// Best key over rows [a_lo, a_hi) of the road, reduced over the group.  The
// key is (chi2 << 32) | (row << 9) | column; since columns < NB < 512 its low
// word orders exactly like the combination index c = row * NB + column.
// Each lane takes one column and runs down the rows of the chunk; in the last
// pass over the columns, when only w < W of them are left, the lanes form
// floor(W / w) groups of w and each group takes one block of the rows.
// GUARDED (valid when chi2_cut < 32767^2): a combination with a chi component
// of magnitude 32767 or more cannot pass, clamped or not.  One range test keeps
// only combinations with -32768 <= y_k <= 32767 for all three components; for
// those the sum of the squares is below 3 * 2^30 < 2^32 and is formed exactly
// in 32 bits, and the clamp changes no square that could still pass.
// Pass/fail, chi2 of passing combinations and the argmin are unchanged.
template <bool GUARDED, int W, typename SM>
__device__ __forceinline__ unsigned long long eval_rows(SM &sm, const Geo &g, uint32_t a_lo,
                                                        uint32_t a_hi, uint32_t qsh,
                                                        uint32_t init_chi, const Lanes<W> &L) {
    constexpr uint32_t MH = SM::kMH, NR = SM::kNR;
    unsigned long long best = ~0ull;
    const uint32_t NB = g.NB, NA = g.NA, C_eval = g.C_eval, NBp = g.NBp, top = g.split;
    const uint32_t mp = kDivMagic[NBp], gl = L.gl;
    for (uint32_t ac = a_lo; ac < a_hi; ac += NR) {
        const uint32_t ae = min(ac + NR, a_hi), rows = ae - ac;
#pragma unroll
        for (uint32_t r0 = 0; r0 < NR; r0 += (uint32_t)W)
            if (r0 + gl < rows) build_row(sm, top, ac + r0 + gl, r0 + gl, qsh);
        __syncwarp(L.mask);
        for (uint32_t b0 = 0; b0 < NB; b0 += (uint32_t)W) {
            uint32_t b = b0 + gl, lo = ac, hi = ae;
            if (NB - b0 < (uint32_t)W) {   // uniform over the group: the last, partial pass
                const uint32_t w = NB - b0, mw = kDivMagic[w];
                const uint32_t grp = div_by(gl, w, mw), n_grp = div_by((uint32_t)W, w, mw);
                const uint32_t len = div_by(rows + n_grp - 1u, n_grp, kDivMagic[n_grp]);
                b -= grp * w;
                lo = min(ac + grp * len, ae);   // groups past the last row get none
                hi = min(lo + len, ae);
            }
            // column b = is * NBp + bp: hit `is` of the top suffix layer and
            // entry bp of the suffix table
            const uint32_t is = div_by(b, NBp, mp), bp = b - is * NBp;
            const longlong2 t01 = sm.T[top * MH + is][0];
            const long long t5 = sm.T[top * MH + is][1].x;
            const longlong2 s01 = sm.S01[bp];
            const long long s5 = sm.S5[bp];
            const long long B3 = t01.x + s01.x, B4 = t01.y + s01.y, B5 = t5 + s5;
            if (hi == NA && lo < hi && (NA - 1) * NB + b >= C_eval) hi -= 1;
            uint32_t bchi = init_chi, ba = 0;
            // whole warps run longer columns: 8 rows per step there took 2-5 %
            // off the fit; half warps (small roads) keep 4
#pragma unroll(W == 32 ? 8 : 4)
            for (uint32_t a = lo; a < hi; ++a) {
                const longlong2 v01 = sm.A01[a - ac];
                const long long v5 = sm.A5[a - ac];
                const int32_t y3 = hi_word(v01.x + B3);
                const int32_t y4 = hi_word(v01.y + B4);
                const int32_t y5 = hi_word(v5 + B5);
                if (GUARDED) {
                    const uint32_t g3 = (uint32_t)y3, g4 = (uint32_t)y4, g5 = (uint32_t)y5;
                    // g_k < 2^16 for all three <=> -32768 <= y_k <= 32767; then
                    // sum (g_k - 32768)^2 = sum g_k^2 - 2^16 sum g_k + 3 * 2^30
                    // holds exactly in 32-bit arithmetic
                    const uint32_t range = g3 | g4 | g5;
                    const uint32_t chi2 = g3 * g3 + g4 * g4 + g5 * g5 + (3u << 30) -
                                          ((g3 + g4 + g5) << 16);
                    if (range < 65536u && chi2 < bchi) {
                        bchi = chi2;
                        ba = a;
                    }
                } else {
                    const int32_t c3 = clamp_chi(y3), c4 = clamp_chi(y4), c5 = clamp_chi(y5);
                    const uint32_t chi2 = (uint32_t)(c3 * c3) + (uint32_t)(c4 * c4) + (uint32_t)(c5 * c5);
                    if (chi2 < bchi) {
                        bchi = chi2;
                        ba = a;
                    }
                }
            }
            if (bchi != init_chi) {
                const unsigned long long key = ((unsigned long long)bchi << 32) | (ba << 9) | b;
                best = key < best ? key : best;
            }
        }
        __syncwarp(L.mask);
    }
    return group_min64<W>(best, L);
}

// Best key of one road fitted whole by a group of W lanes (set-up and all its
// rows), on every lane of the group; UINT64_MAX when no combination passed or
// the road has none to evaluate.
template <bool GUARDED, int W, typename SM>
__device__ __forceinline__ unsigned long long fit_road(SM &sm, const uint32_t *__restrict__ words,
                                                       const RoadDesc &D,
                                                       const int16_t *__restrict__ F,
                                                       const int16_t *__restrict__ q,
                                                       const svt_config &cfg, uint32_t sh,
                                                       uint32_t qsh, uint32_t init_chi,
                                                       const Lanes<W> &L) {
    const Geo g = geo_of(D);
    if (g.C_eval == 0) return ~0ull;
    road_setup<W>(sm, words, D, g, F, q, sh, cfg.xft_pairs, kColBias<GUARDED>, L);
    return eval_rows<GUARDED, W>(sm, g, 0, g.NA, qsh, init_chi, L);
}

// The split of a TINY road for a quarter warp: the shortest suffix of at
// least 8 columns (every layer has one or two hits, so it has exactly 8 when
// the road has 8 or more combinations), one column per lane in a single pass.
// The combination index c = row * NB + column is the same whatever the split,
// so the key is re-expressed in the descriptor's split afterwards (see
// quarter_key).
__device__ __forceinline__ void quarter_geometry(Geo &g, uint32_t packed, uint32_t xft) {
    const RoadShape s = road_shape(packed, xft);
    uint32_t nb = 1, top = 0, NB = (uint32_t)s.C, ntop = s.n[0];
    bool found = false;
#pragma unroll
    for (int l = N_LAYERS - 1; l >= 0; --l) {
        nb *= s.n[l];
        if (!found && nb >= 8u) {
            top = (uint32_t)l;
            NB = nb;
            ntop = s.n[l];
            found = true;
        }
    }
    g.split = top;
    g.NBp = NB / ntop;
    g.NB = NB;
    g.NA = g.C_eval ? (g.C_eval + NB - 1) / NB : 0u;
}

// A key of the quarter split, (chi2, row, column), in the descriptor's split.
__device__ __forceinline__ unsigned long long quarter_key(unsigned long long best,
                                                          uint32_t NB_quarter,
                                                          uint32_t NB_desc) {
    if (best == ~0ull) return best;
    const uint32_t low = (uint32_t)best;
    const uint32_t c = (low >> 9) * NB_quarter + (low & 511u);
    const uint32_t row = c / NB_desc;
    return (best & 0xFFFFFFFF00000000ull) | (row << 9) | (c - row * NB_desc);
}

__device__ __forceinline__ RoadDesc shfl_desc(const uint4 &da, const uint4 &db, uint32_t src) {
    RoadDesc D;
    D.a.x = __shfl_sync(0xffffffffu, da.x, src);
    D.a.y = __shfl_sync(0xffffffffu, da.y, src);
    D.a.z = __shfl_sync(0xffffffffu, da.z, src);
    D.a.w = __shfl_sync(0xffffffffu, da.w, src);
    D.b.x = __shfl_sync(0xffffffffu, db.x, src);
    D.b.y = __shfl_sync(0xffffffffu, db.y, src);
    D.b.z = __shfl_sync(0xffffffffu, db.z, src);
    D.b.w = 0;
    return D;
}

// One TINY road (at most two hits on every layer, so at most 64
// combinations) fitted by one lane, and its record formed there.  The prefix
// layers 0..2 index the rows a and the suffix layers 3..5 the columns b,
// c = a * NB3 + b: the same combination index as in any other split, so the
// lane visits the combinations in increasing c and a strict '<' keeps the
// smallest c among equal chi2.  Every layer has radix 1 or 2, so the digits
// of a row or a column are single bits, and a sum over the layers is the sum
// of the first hits' terms plus, for every digit that is set, the layer's
// difference between its second and its first hit.  The column sums (at most
// 8) go to the lane's column of the slot's tables; each row's sums are formed
// once in registers.  With track-trigger pairs layer 5 has radix 1 and its
// hits' terms are added to those of their layer-4 partners, as in
// road_setup.  With L > 1 lanes to a road (lanes sub = 0..L-1 of a group of
// L consecutive lanes) each lane takes the rows a = sub (mod L) and the group
// merges its (chi2, c) keys; every lane of the group builds the same column
// sums in its own column.  The record is the one form_record writes: flags,
// the best c and its chi2, and the three parameter rows (Eq. 1) of the best
// combination formed in int64 from its hits' coordinates, which the lanes
// still hold.
struct LaneRecord {
    uint32_t w[6];
    bool pass;
};
template <bool GUARDED>
__device__ __forceinline__ LaneRecord lane_fit(LaneTables &tb, const uint32_t *__restrict__ words,
                                               const uint4 &da, const uint4 &db,
                                               const int16_t *__restrict__ F,
                                               const int16_t *__restrict__ q,
                                               const svt_config &cfg, uint32_t sh, uint32_t qsh,
                                               uint32_t init_chi, int lane, uint32_t L,
                                               uint32_t group_mask) {
    const uint32_t C_eval = da.w, packed = da.y, geo = db.x, xft = cfg.xft_pairs;
    const size_t cs = (size_t)rd_sector(da.z) * 64 + ((geo >> 13) & 63u);
    // The chi rows k = 3..5 of F as pairs of int16 (F[k][l], F[k][l+1]) for
    // even l (row k starts at element (cs * 36 + 6 k), an even index, so each
    // pair is 4-byte aligned), the pairs (q_2, q_3), (q_4, q_5); two hit words per
    // layer (the second repeats the first when the layer has one hit; a layer
    // without hits reads the road's header word and takes x = 0).  Every load
    // is issued before any is used.
    const uint32_t *F32 = reinterpret_cast<const uint32_t *>(F + cs * 36);
    const uint32_t *q32 = reinterpret_cast<const uint32_t *>(q + cs * 6);
    uint32_t fp[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) fp[j] = __ldg(F32 + 9 + j);
    const uint32_t q23 = __ldg(q32 + 1), q45 = __ldg(q32 + 2);
    uint32_t hw[N_LAYERS][2];
    {
        uint32_t off = da.x + 1;   // first hit word of layer l (hits are sorted by layer)
#pragma unroll
        for (int l = 0; l < N_LAYERS; ++l) {
            const uint32_t nl = nhit_of(packed, l);
            const uint32_t p0 = nl ? off : da.x;
            hw[l][0] = __ldg(words + p0);
            hw[l][1] = __ldg(words + (nl > 1u ? off + 1u : p0));
            off += nl;
        }
    }
    // the int16 at index j of a run of pairs (little-endian: the even element
    // in the low half)
    auto lo16 = [](uint32_t v) { return (int32_t)(int16_t)(v & 0xFFFFu); };
    auto hi16 = [](uint32_t v) { return (int32_t)v >> 16; };
    auto f_of = [&](int k, int l) -> int32_t {   // F[3 + k][l]
        const uint32_t v = fp[(k * 6 + l) >> 1];
        return (l & 1) ? hi16(v) : lo16(v);
    };
    // Every term is multiplied by P = 2^(32 - oshift) on its way into a 64-bit
    // sum (one wide multiply-add).  A0 and B0 hold the first hits' terms (with
    // q and the column bias); dA and dB the per-layer differences between a
    // layer's second and first hit, F (x1 - x0), which fit in 32 bits.
    const int32_t P = (int32_t)(1u << sh);
    long long A0[3], B0[3];
    int32_t dA[3][3], dB[3][3];
    uint32_t beta[N_LAYERS];   // 1 when the layer's radix is 2
    uint32_t xs[N_LAYERS];     // the layer's two coordinates, x0 | x1 << 16 (0: no hits)
    A0[0] = (long long)hi16(q23) << qsh;
    A0[1] = (long long)lo16(q45) << qsh;
    A0[2] = (long long)hi16(q45) << qsh;
#pragma unroll
    for (int k = 0; k < 3; ++k) B0[k] = kColBias<GUARDED>;
    const uint32_t n5 = nhit_of(packed, N_LAYERS - 1);
#pragma unroll
    for (int l = 0; l < N_LAYERS; ++l) {
        const uint32_t nl = nhit_of(packed, l);
        const bool paired5 = xft && l == N_LAYERS - 1;
        beta[l] = (nl == 2u && !paired5) ? 1u : 0u;
        // with pairs, layer 4's entry i also carries layer 5's hit i
        const bool fold = xft && l == N_LAYERS - 2;
        const int32_t x0 = nl ? (int32_t)hit_coord(hw[l][0]) : 0;
        const int32_t x1 = nl ? (int32_t)hit_coord(hw[l][1]) : 0;
        xs[l] = (uint32_t)x0 | ((uint32_t)x1 << 16);
        const int32_t y0 = (fold && n5) ? (int32_t)hit_coord(hw[N_LAYERS - 1][0]) : 0;
        const int32_t y1 = (fold && n5) ? (int32_t)hit_coord(hw[N_LAYERS - 1][1]) : 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            // |F x| < 2^30: one product, or a pair's two, and their
            // differences fit in 32 bits
            int32_t t0 = 0, d = 0;
            if (!paired5) {
                const int32_t fl = f_of(k, l);
                t0 = fl * x0;
                d = fl * (x1 - x0);
                if (fold) {
                    const int32_t f5 = f_of(k, N_LAYERS - 1);
                    t0 += f5 * y0;
                    d += f5 * (y1 - y0);
                }
            }
            if (l < 3) {
                A0[k] += (long long)t0 * P;
                dA[l][k] = d;
            } else {
                B0[k] += (long long)t0 * P;
                dB[l - 3][k] = d;
            }
        }
    }
    const uint32_t nbB = beta[3] + beta[4] + beta[5], NB3 = 1u << nbB;
    // column sums: column b's digits are bit b5 (layer 5), then layer 4, then layer 3
#pragma unroll
    for (uint32_t b = 0; b < 8u; ++b) {
        if (b < NB3) {
            const uint32_t d5 = b & beta[5], d4 = (b >> beta[5]) & beta[4],
                           d3 = (b >> (beta[5] + beta[4])) & beta[3];
            long long s[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                s[k] = B0[k];
                s[k] += (long long)(d3 ? dB[0][k] : 0) * P;
                s[k] += (long long)(d4 ? dB[1][k] : 0) * P;
                s[k] += (long long)(d5 ? dB[2][k] : 0) * P;
            }
            tb.B01[b][lane] = make_longlong2(s[0], s[1]);
            tb.B5[b][lane] = s[2];
        }
    }
    uint32_t bchi = init_chi, bc = 0;
    const uint32_t NA3 = 1u << (beta[0] + beta[1] + beta[2]), sub = (uint32_t)lane & (L - 1u);
    for (uint32_t a = sub, c0 = sub * NB3; a < NA3 && c0 < C_eval; a += L, c0 += L * NB3) {
        const uint32_t d2 = a & beta[2], d1 = (a >> beta[2]) & beta[1],
                       d0 = (a >> (beta[2] + beta[1])) & beta[0];
        long long A[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            A[k] = A0[k];
            A[k] += (long long)(d0 ? dA[0][k] : 0) * P;
            A[k] += (long long)(d1 ? dA[1][k] : 0) * P;
            A[k] += (long long)(d2 ? dA[2][k] : 0) * P;
        }
        const uint32_t nbr = min(NB3, C_eval - c0);   // columns of this row to evaluate
#pragma unroll
        for (uint32_t b = 0; b < 8u; ++b) {
            if (b < nbr) {
                const longlong2 v01 = tb.B01[b][lane];
                const long long v5 = tb.B5[b][lane];
                const int32_t y3 = hi_word(A[0] + v01.x);
                const int32_t y4 = hi_word(A[1] + v01.y);
                const int32_t y5 = hi_word(A[2] + v5);
                if (GUARDED) {   // as in eval_rows
                    const uint32_t g3 = (uint32_t)y3, g4 = (uint32_t)y4, g5 = (uint32_t)y5;
                    const uint32_t range = g3 | g4 | g5;
                    const uint32_t chi2 = g3 * g3 + g4 * g4 + g5 * g5 + (3u << 30) -
                                          ((g3 + g4 + g5) << 16);
                    if (range < 65536u && chi2 < bchi) {
                        bchi = chi2;
                        bc = c0 + b;
                    }
                } else {
                    const int32_t c3 = clamp_chi(y3), c4 = clamp_chi(y4), c5 = clamp_chi(y5);
                    const uint32_t chi2 =
                        (uint32_t)(c3 * c3) + (uint32_t)(c4 * c4) + (uint32_t)(c5 * c5);
                    if (chi2 < bchi) {
                        bchi = chi2;
                        bc = c0 + b;
                    }
                }
            }
        }
    }
    // the group's best: smallest chi2, then smallest c
    unsigned long long key = bchi != init_chi ? ((unsigned long long)bchi << 32) | bc : ~0ull;
    for (uint32_t d = 1; d < L; d <<= 1) {
        const unsigned long long o = __shfl_xor_sync(group_mask, key, d);
        key = o < key ? o : key;
    }
    bchi = (uint32_t)(key >> 32);
    bc = (uint32_t)key;
    // the record
    LaneRecord rec;
    rec.pass = C_eval > 0 && key != ~0ull;
    uint32_t flags = rec.pass ? SVT_FLAG_PASS : 0u;
    if (((geo >> 19) & 127u) == 0) flags |= SVT_FLAG_NO_HITS;
    if (geo & (1u << 27)) flags |= SVT_FLAG_BAD_PATTERN;
    if (geo & (1u << 26)) flags |= SVT_FLAG_OVERFLOW;
    rec.w[0] = rd_id(da.z) | (flags << 24);
    rec.w[1] = rec.pass ? bc : 0xFFFFFFFFu;
    rec.w[2] = rec.pass ? bchi : 0u;
    rec.w[3] = rec.w[4] = rec.w[5] = 0u;
    if (rec.pass) {
        // the parameter rows k = 0..2 of F and q
#pragma unroll
        for (int j = 0; j < 9; ++j) fp[j] = __ldg(F32 + j);
        const uint32_t q01 = __ldg(q32), q2x = __ldg(q32 + 1);
        // the best combination's digits (with pairs, layer 5 takes layer 4's)
        const uint32_t a = bc >> nbB, b = bc & (NB3 - 1u);
        uint32_t d[N_LAYERS];
        d[5] = b & beta[5];
        d[4] = (b >> beta[5]) & beta[4];
        d[3] = (b >> (beta[5] + beta[4])) & beta[3];
        d[2] = a & beta[2];
        d[1] = (a >> beta[2]) & beta[1];
        d[0] = (a >> (beta[2] + beta[1])) & beta[0];
        if (xft) d[5] = d[4];
        int32_t x[N_LAYERS];
#pragma unroll
        for (int l = 0; l < N_LAYERS; ++l) x[l] = (int32_t)((xs[l] >> (16u * d[l])) & 0xFFFFu);
        const int32_t qv[3] = {lo16(q01), hi16(q01), lo16(q2x)};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            long long acc = (long long)qv[k] * (1ll << cfg.qshift);
#pragma unroll
            for (int l = 0; l < N_LAYERS; ++l) {
                const uint32_t v = fp[(k * 6 + l) >> 1];
                acc += (long long)((l & 1) ? hi16(v) : lo16(v)) * (long long)x[l];
            }
            rec.w[3 + k] = (uint32_t)(int32_t)(acc >> cfg.oshift);   // floor
        }
    }
    return rec;
}

// Record of road r from its best key (six words into w), formed by one lane
// (the warps of the fit kernel hand their finished roads out one per lane,
// see RecordList).
// For a road that passed, the hits of its best combination are the digits of
// c = row * NB + column in the radices n'_l (the column's digits for the
// suffix layers, the row's for the prefix layers), and the parameters
// p_k = floor((q_k 2^qshift + sum_l F_kl x_l) / 2^oshift), k = 0..2, are
// formed from them in int64 (Eq. 1 for the three parameter rows).  Every load
// is issued before any is used, with no branch between them (a layer without
// hits reads the road's header word and discards it).  Returns whether the
// road passed.
__device__ __forceinline__ bool form_record(const uint32_t *__restrict__ words,
                                            const RoadDesc *__restrict__ desc, uint32_t r,
                                            unsigned long long best,
                                            const int16_t *__restrict__ F,
                                            const int16_t *__restrict__ q,
                                            const svt_config &cfg, uint32_t *w) {
    const uint4 da = __ldg(&desc[r].a), db = __ldg(&desc[r].b);
    const uint32_t geo = db.x, packed = da.y, total_hits = (geo >> 19) & 127u;
    const bool pass = best != ~0ull;
    uint32_t flags = 0;
    if (total_hits == 0) flags |= SVT_FLAG_NO_HITS;
    if (geo & (1u << 27)) flags |= SVT_FLAG_BAD_PATTERN;
    if (geo & (1u << 26)) flags |= SVT_FLAG_OVERFLOW;
    uint32_t c = 0xFFFFFFFFu, chi2 = 0;
    int32_t p[3] = {0, 0, 0};
    if (pass) {
        flags |= SVT_FLAG_PASS;
        const uint32_t low = (uint32_t)best, row = low >> 9, col = low & 511u;
        const uint32_t split = geo & 7u;
        c = row * db.y + col;
        chi2 = (uint32_t)(best >> 32);
        uint32_t digit[N_LAYERS];
        uint32_t rem = col;
#pragma unroll
        for (int l = N_LAYERS - 1; l >= 0; --l) {
            if ((uint32_t)l + 1u == split) rem = row;   // the prefix layers take the row
            const uint32_t nl = nhit_of(packed, l);
            const uint32_t np = (nl && !(cfg.xft_pairs && l == N_LAYERS - 1)) ? nl : 1u;
            const uint32_t qd = div_by(rem, np, kDivMagic[np]);
            digit[l] = rem - qd * np;
            rem = qd;
        }
        if (cfg.xft_pairs) digit[N_LAYERS - 1] = digit[N_LAYERS - 2];   // the pair's own index
        const size_t cs = (size_t)rd_sector(da.z) * 64 + ((geo >> 13) & 63u);
        uint32_t hw[N_LAYERS];
        uint32_t off = da.x + 1;   // first hit word of layer l (hits are sorted by layer)
#pragma unroll
        for (int l = 0; l < N_LAYERS; ++l) {
            const uint32_t nl = nhit_of(packed, l);
            hw[l] = __ldg(words + (nl ? off + digit[l] : da.x));
            off += nl;
        }
        int32_t f[3][N_LAYERS], qk[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            qk[k] = __ldg(q + cs * 6 + k);
#pragma unroll
            for (int l = 0; l < N_LAYERS; ++l) f[k][l] = __ldg(F + cs * 36 + k * 6 + l);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            long long acc = (long long)qk[k] * (1ll << cfg.qshift);
#pragma unroll
            for (int l = 0; l < N_LAYERS; ++l) {
                const int32_t x = nhit_of(packed, l) ? (int32_t)hit_coord(hw[l]) : 0;
                acc += (long long)f[k][l] * (long long)x;
            }
            p[k] = (int32_t)(acc >> cfg.oshift);   // floor
        }
    }
    w[0] = rd_id(da.z) | (flags << 24);
    w[1] = c;
    w[2] = chi2;
    w[3] = (uint32_t)p[0];
    w[4] = (uint32_t)p[1];
    w[5] = (uint32_t)p[2];
    return pass;
}

// ---- large roads: screened in single precision ------------------------------------
// Where a batch's roads are large (see SCREEN_MEAN), the exact 64-bit sums and
// squares of every combination are all the work, and nearly every one of them
// is far from the best: so every combination is SCREENED in single precision,
// g_k = A_k(a) + B_k(b) and s = sum_k g_k^2, two rows to a packed fp32
// instruction (about 5.5 warp instructions per 32 combinations instead of 18),
// only the smallest s of each lane is kept, and the few combinations whose s can
// belong to the best one are evaluated in exact 64-bit integers (the bound below
// makes this exact, whatever the constants).
// Screening parameters (host: make_screen).  For a combination let
// v_k = acc_k / 2^oshift (k = 3..5, exact), so y_k = floor(v_k) lies within 1/2
// of v_k - 1/2.  The screen forms g_k = v_k - 1/2 + e_k in single precision,
// |e_k| <= E = 10 u M with u = 2^-24 and M = (6 2^30 + 2^(15+qshift)) / 2^oshift + 1
// the largest magnitude of any partial sum: at most seven additions of terms
// (six terms and q; one more when a track-trigger pair is folded), each
// within u M, and the terms' own roundings, together within 2 u M.  Hence
//     | |y| - |g| | <= delta = sqrt(3) (1/2 + E)      (Euclidean norms),
// and s = fl(|g|^2) is within a factor 1 +- 2^-21 of |g|^2.  So
//   - a combination of chi2 <= X has s <= reach(X, delta),
//   - when some combination has s = m, the best one has
//     s <= reach(m, 2 delta),
// with reach(v, d) = (sqrt(v) (1 + 2^-18) + d)^2 (1 + 2^-18); the factors cover
// every rounding of s, of the square root and of reach itself.  At the usual
// shifts (15, 15) delta is 1.1, in units where a chi component of one
// standard deviation is of the order of 100, so hardly any column but the
// best one is confirmed; for extreme shifts delta grows and more columns are
// confirmed, with the same result.
// Clamping: a combination with |y_k| >= 32767 for some k has chi2 >= 32767^2.
// So below SAT = 32767^2 the clamped and the unclamped chi2 order alike, the
// screen starts at reach(min(cut, SAT), delta), and when nothing below SAT
// turns up while the cut would let larger values pass, every combination of
// the road (or item) is evaluated exactly (see unsure).
struct Screen {
    float f_scale, q_scale;   // 2^-oshift, 2^(qshift - oshift)
    float delta, thr;         // delta; reach(min(cut, SAT), delta)
};
constexpr uint32_t SAT = 32767u * 32767u;

// A road's working set in shared memory.
constexpr uint32_t SCREEN_ROWS = 64;
struct ScreenSmem {
    float4 T[N_LAYERS * MAX_HITS];   // hit i of layer l at [l*16+i]: its terms
                                     // F[3+k][l] x 2^-oshift, k = 0..2, and in .w the bits of
                                     // its coordinate x
    float4 S[32];                    // suffix sums below the top suffix layer [b']
    // rows of the chunk in pairs (a, a + 1) for the packed arithmetic, with one
    // more pair for the last row of a road cut off by max_comb
    float4 A34[SCREEN_ROWS / 2 + 1];   // {A_3(a), A_3(a+1), A_4(a), A_4(a+1)}, incl. q and -1/2
    float2 A5[SCREEN_ROWS / 2 + 2];    // {A_5(a), A_5(a+1)}
    float4 Ff[N_LAYERS];               // F[3+k][l] 2^-oshift, k = 0..2
    int4 Fi[N_LAYERS];                 // F[3+k][l]
    uint2 nm[N_LAYERS];                // n'_l = max(n_l, 1) and its division magic
    uint32_t off[N_LAYERS];            // index of the first hit of layer l in the road
    int32_t q[4];                      // q[3+k]
};

// Listed combinations whose exact chi2 is still to be formed: of every road
// the warp has finished up to LIST_MAX, one after another (one entry with
// combination NONE for a road without any).  When the next road's might not
// fit (and when the warp runs out of work) they are evaluated exactly, one per
// lane, and the roads' records written (flush_records), so that neither the
// exact sums nor the records hold all 32 lanes for every road.
constexpr uint32_t NONE = 0xFFFFFFFFu;
constexpr uint32_t LIST_MAX = 8, CAND = 96;
struct CandList {
    uint2 ent[32];        // road, combination
};
static_assert(sizeof(CandList) <= sizeof(RecordList), "a warp's list holds either form");

// A road's tables and the combinations of it that are within reach, each with
// the bits of its s; flush_records works in the same place between roads: per
// entry six record words, 18 words of F (19: odd, so that the lanes' reads fall
// in different banks), three of q.  The candidates sit in the slot, which is
// larger than the tables, and not beside the list: with 1024 bytes of list a
// warp instead of 384 blocks of four warps fitted seven times on an SM and not
// eight (of two 15 and 16, of one 28 and 30).
union ScreenSlot {
    struct {
        ScreenSmem road;
        uint2 cand[CAND];
    };
    uint32_t flush[32 * (6 + 19 + 3)];
};
static_assert(sizeof(ScreenSlot) <= sizeof(WarpSmem) && alignof(ScreenSlot) <= 16,
              "a road slot holds either form");

// Two packed single-precision operations at once (each half rounded to
// nearest, as the scalar operations are).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 both(float v) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float min2(f32x2 s, float m) {   // the smaller half, and m
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(s));
    return fminf(fminf(a, b), m);
}

// see Screen (the approximate root is within 2^-23 of the root)
__device__ __forceinline__ float reach(float v, float d) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(v));
    r = fmaf(r, 1.f + 0x1p-18f, d);
    return r * r * (1.f + 0x1p-18f);
}

// Constants, hit coordinates and per-hit chi terms of road D in the warp's slot.
// Global loads are issued before any shared-memory work; a road has at most 96
// hits, so three passes of the lanes hold them all.
__device__ __forceinline__ void screen_load(ScreenSmem &sm, const uint32_t *__restrict__ words,
                                          const RoadDesc &D, const Geo &g,
                                          const int16_t *__restrict__ F,
                                          const int16_t *__restrict__ q, const Screen &sc,
                                          uint32_t xft, const Lanes<32> &L) {
    constexpr uint32_t MH = (uint32_t)MAX_HITS;
    // the chi rows k = 3..5 only (18 + 3 constants): the record's parameter
    // rows are read from global memory by the lane that forms it
    const uint32_t rw = D.a.x, packed = D.a.y, gl = L.gl;
    const size_t cs = (size_t)rd_sector(D.a.z) * 64 + g.mask;
    const int32_t fv =
        gl < 18 ? __ldg(F + cs * 36 + 18 + gl) : (gl < 21 ? __ldg(q + cs * 6 + gl - 15) : 0);
    uint32_t hv[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const uint32_t h = gl + 32u * j;
        hv[j] = h < g.total_hits ? __ldg(words + rw + 1 + h) : 0u;
    }
    const uint32_t nl = gl < N_LAYERS ? nhit_of(packed, gl) : 0u;
    uint32_t incl = nl;   // inclusive prefix of the layer counts
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) {
        const uint32_t v = __shfl_up_sync(L.mask, incl, d);
        if (gl >= (uint32_t)d) incl += v;
    }
    if (gl < N_LAYERS) {
        // with track-trigger pairs layer 5 is no digit of its own (radix 1)
        const uint32_t np = (nl && !(xft && gl == N_LAYERS - 1)) ? nl : 1u;
        sm.nm[gl] = make_uint2(np, kDivMagic[np]);
        sm.off[gl] = incl - nl;
        // a layer without hits contributes x = 0
        if (nl == 0) sm.T[gl * MH] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (gl < 18) {
        const uint32_t k = gl / 6, l = gl - 6 * k;
        reinterpret_cast<float *>(&sm.Ff[l])[k] = (float)fv * sc.f_scale;
        reinterpret_cast<int32_t *>(&sm.Fi[l])[k] = fv;
    } else if (gl < 21) {
        sm.q[gl - 18] = fv;
    }
    __syncwarp(L.mask);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const uint32_t h = gl + 32u * j;
        if (h < g.total_hits) {
            const uint32_t l = hit_layer(hv[j]);
            const uint32_t i = h - sm.off[l];   // hits are sorted by layer (validated)
            const uint32_t xc = hit_coord(hv[j]);
            const float x = (float)xc;
            const float4 f = sm.Ff[l];
            sm.T[l * MH + i] = make_float4(f.x * x, f.y * x, f.z * x, __uint_as_float(xc));
        }
    }
    __syncwarp(L.mask);
    if (xft) {
        // pair i: layer 4's entry i carries both coordinates' terms of
        // track-trigger track i (equal counts are validated); layer 5 then
        // adds none (its coordinates stay)
        const uint32_t n4 = nhit_of(packed, 4);
        for (uint32_t i = gl; i < n4; i += 32u) {
            float4 &t4 = sm.T[4 * MH + i], &t5 = sm.T[5 * MH + i];
            const float4 v = t5;
            t4.x += v.x;
            t4.y += v.y;
            t4.z += v.z;
            t5.x = t5.y = t5.z = 0.f;
        }
        __syncwarp(L.mask);
    }
}

// S[b'] = sum over the suffix layers below the top one, b' < NBp (< 32).
__device__ __forceinline__ void screen_suffix(ScreenSmem &sm, const Geo &g, const Lanes<32> &L) {
    constexpr uint32_t MH = (uint32_t)MAX_HITS;
    for (uint32_t bp = L.gl; bp < g.NBp; bp += 32u) {
        uint32_t rem = bp;
        float s3 = 0.f, s4 = 0.f, s5 = 0.f;
#pragma unroll
        for (int l = N_LAYERS - 1; l >= 1; --l) {
            if ((uint32_t)l > g.split) {
                const uint2 nm = sm.nm[l];
                const uint32_t qd = div_by(rem, nm.x, nm.y);
                const float4 t = sm.T[l * MH + rem - qd * nm.x];
                rem = qd;
                s3 += t.x;
                s4 += t.y;
                s5 += t.z;
            }
        }
        sm.S[bp] = make_float4(s3, s4, s5, 0.f);
    }
}

// The sums of row a (q and the -1/2 of the screen included) at index `slot`
// of the chunk's rows.
__device__ __forceinline__ void screen_row(ScreenSmem &sm, uint32_t split, uint32_t a, uint32_t slot,
                                          const Screen &sc) {
    constexpr uint32_t MH = (uint32_t)MAX_HITS;
    uint32_t rem = a;
    float a3 = fmaf((float)sm.q[0], sc.q_scale, -0.5f);
    float a4 = fmaf((float)sm.q[1], sc.q_scale, -0.5f);
    float a5 = fmaf((float)sm.q[2], sc.q_scale, -0.5f);
#pragma unroll
    for (int l = N_LAYERS - 2; l >= 0; --l) {
        if ((uint32_t)l < split) {
            const uint2 nm = sm.nm[l];
            const uint32_t qd = div_by(rem, nm.x, nm.y);
            const float4 t = sm.T[l * MH + rem - qd * nm.x];
            rem = qd;
            a3 += t.x;
            a4 += t.y;
            a5 += t.z;
        }
    }
    float *p34 = reinterpret_cast<float *>(sm.A34 + slot / 2) + (slot & 1u);
    p34[0] = a3;
    p34[2] = a4;
    reinterpret_cast<float *>(sm.A5)[slot] = a5;
}

// chi2 of combination c exactly: the sums in int64 (Eq. 1), the floor, the
// clamp and the squares.
__device__ __forceinline__ uint32_t exact_chi2(const ScreenSmem &sm, uint32_t c, const svt_config &cfg) {
    constexpr uint32_t MH = (uint32_t)MAX_HITS;
    long long acc[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        acc[k] = (long long)((unsigned long long)(long long)sm.q[k] << cfg.qshift);
    uint32_t digit[N_LAYERS], rem = c;
#pragma unroll
    for (int l = N_LAYERS - 1; l >= 0; --l) {
        const uint2 nm = sm.nm[l];
        const uint32_t qd = div_by(rem, nm.x, nm.y);
        digit[l] = rem - qd * nm.x;
        rem = qd;
    }
    if (cfg.xft_pairs) digit[N_LAYERS - 1] = digit[N_LAYERS - 2];   // the pair's own index
#pragma unroll
    for (int l = 0; l < N_LAYERS; ++l) {
        const int32_t x = (int32_t)__float_as_uint(sm.T[l * MH + digit[l]].w);
        const int4 f = sm.Fi[l];
        acc[0] += (long long)f.x * x;
        acc[1] += (long long)f.y * x;
        acc[2] += (long long)f.z * x;
    }
    uint32_t chi2 = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int32_t y = clamp_chi((int32_t)(acc[k] >> cfg.oshift));   // |y| < 2^31
        chi2 += (uint32_t)(y * y);
    }
    return chi2;
}

// Best key over the combinations [c_lo, c_hi), every one evaluated exactly;
// key = (chi2 << 32) | c, UINT64_MAX when none passes the cut.
__device__ __forceinline__ unsigned long long sweep(const ScreenSmem &sm, uint32_t c_lo, uint32_t c_hi,
                                                    const svt_config &cfg, const Lanes<32> &L) {
    unsigned long long best = ~0ull;
    for (uint32_t c = c_lo + L.gl; c < c_hi; c += 32u) {
        const uint32_t chi2 = exact_chi2(sm, c, cfg);
        const unsigned long long key = ((unsigned long long)chi2 << 32) | c;
        if (chi2 <= cfg.chi2_cut && key < best) best = key;
    }
    return group_min64<32>(best, L);
}

// The combinations of rows [a_lo, a_hi) that can be the best one, by a whole
// warp: listed in cand, their number returned (more than CAND: they did not
// fit); thr is the final reach.  Each lane takes one column and runs down the
// rows of the chunk, two per step; in the last pass over the columns, when only
// w < 32 of them are left, the lanes form floor(32 / w) groups of w and each
// group takes one block of the row pairs.  A lane keeps its smallest s, the pass
// it is from and the smallest of its other passes; at the end of the chunk the
// columns that hold combinations within reach are looked at once more, a row
// per lane.
__device__ __forceinline__ uint32_t list_rows(ScreenSmem &sm, uint2 *cand, const Geo &g, uint32_t a_lo,
                                              uint32_t a_hi, const Screen &sc, float &thr,
                                              uint32_t lane) {
    constexpr uint32_t MH = (uint32_t)MAX_HITS, NR = SCREEN_ROWS, ALL = 0xffffffffu;
    constexpr float FAR = 1e18f;   // a row past the last: its s is never the smallest
    uint32_t listed = 0;
    thr = sc.thr;
    const uint32_t NB = g.NB, NA = g.NA, C_eval = g.C_eval, NBp = g.NBp, top = g.split;
    const uint32_t mp = kDivMagic[NBp], n_passes = (NB + 31u) >> 5;
    for (uint32_t ac = a_lo; ac < a_hi; ac += NR) {
        const uint32_t ae = min(ac + NR, a_hi);
        // the road's last row when max_comb cuts it short: kept apart, in the
        // extra pair, for the columns that are left of it
        const bool cut_row = ae == NA && NA * NB > C_eval;
        const uint32_t rows = ae - ac - (cut_row ? 1u : 0u), pairs = (rows + 1u) >> 1;
#pragma unroll
        for (uint32_t r0 = 0; r0 < NR; r0 += 32u) {
            const uint32_t r = r0 + lane;
            if (r < ae - ac) screen_row(sm, top, ac + r, r < rows ? r : NR, sc);
        }
        if (lane == 0 && (rows & 1u)) {
            reinterpret_cast<float *>(sm.A34 + rows / 2)[1] = FAR;
            reinterpret_cast<float *>(sm.A34 + rows / 2)[3] = 0.f;
            reinterpret_cast<float *>(sm.A5)[rows] = 0.f;
        }
        __syncwarp();
        auto screen = [&](uint32_t p, f32x2 b3, f32x2 b4, f32x2 b5) {
            const ulonglong2 v = reinterpret_cast<const ulonglong2 *>(sm.A34)[p];
            const f32x2 g3 = add2(v.x, b3), g4 = add2(v.y, b4),
                        g5 = add2(reinterpret_cast<const f32x2 *>(sm.A5)[p], b5);
            return fma2(g5, g5, fma2(g4, g4, mul2(g3, g3)));
        };
        // lane `ln`'s column in pass cp and its row pairs
        struct Column {
            uint32_t b, lo, hi;
            bool extra;
        };
        auto column = [&](uint32_t cp, uint32_t ln) {
            Column c{cp * 32u + ln, 0u, pairs, cut_row};
            const uint32_t w = NB - cp * 32u;
            if (w < 32u) {   // uniform: the last, partial pass
                const uint32_t mw = kDivMagic[w];
                const uint32_t grp = div_by(ln, w, mw), n_grp = div_by(32u, w, mw);
                const uint32_t len = div_by(pairs + n_grp - 1u, n_grp, kDivMagic[n_grp]);
                c.b -= grp * w;
                c.lo = min(grp * len, pairs);   // groups past the last pair get none
                c.hi = min(c.lo + len, pairs);
                c.extra = cut_row && grp == 0;
            }
            c.extra = c.extra && (NA - 1u) * NB + c.b < C_eval;
            return c;
        };
        // column b = is * NBp + bp: hit `is` of the top suffix layer and entry bp
        // of the suffix table
        auto column_sums = [&](uint32_t b) {
            const uint32_t is = div_by(b, NBp, mp), bp = b - is * NBp;
            const float4 t = sm.T[top * MH + is], u = sm.S[bp];
            return make_float3(t.x + u.x, t.y + u.y, t.z + u.z);
        };
        auto smallest = [&](const Column &c) {
            const float3 B = column_sums(c.b);
            const f32x2 b3 = both(B.x), b4 = both(B.y), b5 = both(B.z);
            float m = 3e38f;
#pragma unroll 4
            for (uint32_t p = c.lo; p < c.hi; ++p) m = min2(screen(p, b3, b4, b5), m);
            if (cut_row && c.extra)
                m = fminf(__uint_as_float((uint32_t)screen(NR / 2, b3, b4, b5)), m);
            return m;
        };
        float m1 = 3e38f, m2 = 3e38f;
        uint32_t cp1 = 0;
        for (uint32_t cp = 0; cp < n_passes; ++cp) {
            const float m = smallest(column(cp, lane));
            m2 = fminf(m2, fmaxf(m, m1));
            cp1 = m < m1 ? cp : cp1;
            m1 = fminf(m, m1);
        }
        // the smallest s so far (s >= 0: its bits order like it)
        const float ms = __uint_as_float(__reduce_min_sync(ALL, __float_as_uint(m1)));
        if (ms <= thr) {   // uniform
            thr = fminf(thr, reach(ms, 2.f * sc.delta));
            // the lanes with something within reach, for the pass their smallest s is
            // from; when one has more in another pass, every pass again
            const bool again = __any_sync(ALL, m2 <= thr);
            for (uint32_t cp = 0; cp < (again ? n_passes : 1u); ++cp) {
                const float m = again ? smallest(column(cp, lane)) : m1;
                uint32_t todo = __ballot_sync(ALL, m <= thr);
                while (todo) {
                    const uint32_t src = (uint32_t)__ffs(todo) - 1u;
                    todo &= todo - 1u;
                    const Column c = column(again ? cp : __shfl_sync(ALL, cp1, src), src);
                    const float3 B = column_sums(c.b);
                    const uint32_t r_lo = 2u * c.lo, r_hi = min(2u * c.hi, rows);
                    const uint32_t n_r = r_hi > r_lo ? r_hi - r_lo : 0u;
                    const uint32_t n_x = n_r + (c.extra ? 1u : 0u);
                    for (uint32_t i0 = 0; i0 < n_x; i0 += 32u) {
                        const uint32_t i = i0 + lane, sl = i < n_r ? r_lo + i : NR;   // row slot
                        const float *p =
                            reinterpret_cast<const float *>(sm.A34 + sl / 2) + (sl & 1u);
                        const float g3 = __fadd_rn(p[0], B.x), g4 = __fadd_rn(p[2], B.y),
                                    g5 = __fadd_rn(reinterpret_cast<const float *>(sm.A5)[sl], B.z);
                        const float s = __fmaf_rn(g5, g5, __fmaf_rn(g4, g4, __fmul_rn(g3, g3)));
                        const bool hit = i < n_x && s <= thr;
                        const uint32_t hits = __ballot_sync(ALL, hit);
                        const uint32_t k = listed + __popc(hits & ((1u << lane) - 1u));
                        if (hit && k < CAND)
                            cand[k] = make_uint2((i < n_r ? ac + r_lo + i : NA - 1u) * NB + c.b,
                                                 __float_as_uint(s));
                        listed += __popc(hits);
                    }
                    if (listed > CAND) return listed;   // (uniform)
                }
            }
        }
        __syncwarp();
        // what later columns and rows have put out of reach leaves the list
        if (listed > 1u && listed <= CAND) {   // uniform
            uint32_t kept = 0;
            for (uint32_t k0 = 0; k0 < listed; k0 += 32u) {
                const uint2 e = k0 + lane < listed ? cand[k0 + lane] : make_uint2(0u, ~0u);
                const bool keep = k0 + lane < listed && __uint_as_float(e.y) <= thr;
                const uint32_t kb = __ballot_sync(ALL, keep);
                if (keep) cand[kept + __popc(kb & ((1u << lane) - 1u))] = e;
                kept += __popc(kb);
                __syncwarp();
            }
            listed = kept;
        }
    }
    return listed;
}

// Whether the list of rows [a_lo, a_hi) does not decide: it did not hold all that
// is within reach, or nothing is sure to lie below SAT (see Screen).
__device__ __forceinline__ bool unsure(uint32_t listed, float thr, const svt_config &cfg) {
    return listed > CAND || (cfg.chi2_cut >= SAT && !(thr < (float)SAT));
}

// Best key of the listed combinations, evaluated exactly by a whole warp.
__device__ __forceinline__ unsigned long long best_of_list(const ScreenSmem &sm, const uint2 *cand,
                                                           uint32_t listed, const svt_config &cfg,
                                                           const Lanes<32> &L) {
    unsigned long long best = ~0ull;
    for (uint32_t k = L.gl; k < listed; k += 32u) {
        const uint32_t c = cand[k].x, chi2 = exact_chi2(sm, c, cfg);
        const unsigned long long key = ((unsigned long long)chi2 << 32) | c;
        if (chi2 <= cfg.chi2_cut && key < best) best = key;
    }
    return group_min64<32>(best, L);
}

// A road of at most DIRECT passes of a group's lanes over its combinations is
// evaluated exactly at once, without the tables.
constexpr uint32_t DIRECT = 2;

// One road fitted whole by the warp: its candidates in cand, their number
// returned (at most LIST_MAX, or UNSURE).
constexpr uint32_t UNSURE = 0xFFFFFFFFu;
__device__ __forceinline__ uint32_t screen_road(ScreenSmem &sm, uint2 *cand,
                                              const uint32_t *__restrict__ words,
                                              const RoadDesc &D, const int16_t *__restrict__ F,
                                              const int16_t *__restrict__ q,
                                              const svt_config &cfg, const Screen &sc,
                                              const Lanes<32> &L) {
    const Geo g = geo_of(D);
    if (g.C_eval == 0) return 0;
    screen_load(sm, words, D, g, F, q, sc, cfg.xft_pairs, L);
    unsigned long long best;
    if (g.C_eval <= DIRECT * 32u) {
        best = sweep(sm, 0, g.C_eval, cfg, L);
    } else {
        screen_suffix(sm, g, L);
        float thr;
        const uint32_t n = list_rows(sm, cand, g, 0, g.NA, sc, thr, L.gl);
        if (unsure(n, thr, cfg)) return UNSURE;
        if (n <= LIST_MAX) return n;
        best = best_of_list(sm, cand, n, cfg, L);
    }
    __syncwarp();
    if (L.gl == 0) cand[0].x = (uint32_t)best;   // (UINT64_MAX reads as NONE)
    return 1;
}

// The coordinates of combination c's hits in the road with descriptor words da
// (svt_roads.cuh), by one lane: the hits are the digits of c in the radices
// n'_l.  Every load is issued before any is used (a layer without hits reads
// the road's header word and discards it: x = 0).
__device__ __forceinline__ void comb_coords(const uint32_t *__restrict__ words,
                                            const svt_config &cfg, const uint4 &da, uint32_t c,
                                            int32_t (&x)[N_LAYERS]) {
    const uint32_t packed = da.y;
    uint32_t digit[N_LAYERS], rem = c;
#pragma unroll
    for (int l = N_LAYERS - 1; l >= 0; --l) {
        const uint32_t nl = nhit_of(packed, l);
        const uint32_t np = (nl && !(cfg.xft_pairs && l == N_LAYERS - 1)) ? nl : 1u;
        const uint32_t qd = div_by(rem, np, kDivMagic[np]);
        digit[l] = rem - qd * np;
        rem = qd;
    }
    if (cfg.xft_pairs) digit[N_LAYERS - 1] = digit[N_LAYERS - 2];   // the pair's own index
    uint32_t hw[N_LAYERS];
    uint32_t off = da.x + 1;   // first hit word of layer l (hits are sorted by layer)
#pragma unroll
    for (int l = 0; l < N_LAYERS; ++l) {
        const uint32_t nl = nhit_of(packed, l);
        hw[l] = __ldg(words + (nl ? off + digit[l] : da.x));
        off += nl;
    }
#pragma unroll
    for (int l = 0; l < N_LAYERS; ++l) x[l] = nhit_of(packed, l) ? (int32_t)hit_coord(hw[l]) : 0;
}

// y_k = floor((q_k 2^qshift + sum_l F_kl x_l) / 2^oshift) (Eq. 1), in int64
template <typename GetF>
__device__ __forceinline__ int32_t exact_y(const svt_config &cfg, int32_t qk, GetF F,
                                           const int32_t (&x)[N_LAYERS]) {
    long long acc = (long long)qk * (1ll << cfg.qshift);
#pragma unroll
    for (int l = 0; l < N_LAYERS; ++l) acc += (long long)F(l) * (long long)x[l];
    return (int32_t)(acc >> cfg.oshift);   // |y| < 2^31
}

__device__ __forceinline__ uint32_t chi_square(int32_t y3, int32_t y4, int32_t y5) {
    const int32_t a = clamp_chi(y3), b = clamp_chi(y4), c = clamp_chi(y5);
    return (uint32_t)(a * a) + (uint32_t)(b * b) + (uint32_t)(c * c);
}

// Records of the n_rec listed combinations: each lane forms one, the first
// lane of every road picks the road's best one, and the warp stores the records
// with consecutive lanes on consecutive words.  The entries' rows of constants
// (84 bytes each, scattered over the table) are fetched by the whole warp, word
// after word, and read back by the entry's lane: lane by lane every one of 42
// loads touched 32 cache lines, 18 us of the paper's shape at 3000 events.
// Returns the passing roads this lane picked for.
__device__ __forceinline__ uint32_t flush_records(const uint32_t *__restrict__ words,
                                                  const RoadDesc *__restrict__ desc,
                                                  const int16_t *__restrict__ F,
                                                  const int16_t *__restrict__ q,
                                                  const svt_config &cfg, uint32_t *out,
                                                  CandList &rl, uint32_t *stage,
                                                  uint32_t n_rec) {
    const uint32_t lane = threadIdx.x & 31u;
    __syncwarp();
    uint32_t *Fs = stage + 32 * 6, *qs = Fs + 32 * 19;
    const uint2 e = rl.ent[lane];
    const bool on = lane < n_rec;
    const bool head = on && (lane == 0 || rl.ent[lane - 1].x != e.x);
    uint4 da = make_uint4(0, 0, 0, 0);
    uint32_t geo = 0;
    if (on) {
        da = __ldg(&desc[e.x].a);
        geo = __ldg(&desc[e.x].b.x);
    }
    const uint32_t cs = rd_sector(da.z) * 64u + ((geo >> 13) & 63u);
    if ((((uintptr_t)F | (uintptr_t)q) & 3u) == 0) {
        const uint32_t *F32 = reinterpret_cast<const uint32_t *>(F);
        const uint32_t *q32 = reinterpret_cast<const uint32_t *>(q);
#pragma unroll 4
        for (uint32_t j = 0; j * 32u < n_rec * 21u; ++j) {
            const uint32_t i = j * 32u + lane, k = i / 21u, w = i - k * 21u;
            const uint32_t c = __shfl_sync(0xffffffffu, cs, k);
            if (k < n_rec) {
                if (w < 18u)
                    Fs[k * 19u + w] = __ldg(F32 + c * 18u + w);
                else
                    qs[k * 3u + w - 18u] = __ldg(q32 + c * 3u + w - 18u);
            }
        }
    } else {
        uint16_t *Fh = reinterpret_cast<uint16_t *>(Fs), *qh = reinterpret_cast<uint16_t *>(qs);
        for (uint32_t j = 0; j * 32u < n_rec * 42u; ++j) {
            const uint32_t i = j * 32u + lane, k = i / 42u, w = i - k * 42u;
            const uint32_t c = __shfl_sync(0xffffffffu, cs, k);
            if (k < n_rec) {
                if (w < 36u)
                    Fh[k * 38u + w] = (uint16_t)__ldg(F + c * 36u + w);
                else
                    qh[k * 6u + w - 36u] = (uint16_t)__ldg(q + c * 6u + w - 36u);
            }
        }
    }
    int32_t x[N_LAYERS] = {0, 0, 0, 0, 0, 0};
    if (on && e.y != NONE) comb_coords(words, cfg, da, e.y, x);
    __syncwarp();
    uint32_t *mine = stage + lane * 6;
    if (on) {
        // 16-bit entry i of a row of pairs (little-endian: even ones in the low half)
        auto at16 = [](const uint32_t *w, int i) {
            return (i & 1) ? (int32_t)w[i >> 1] >> 16 : (int32_t)(int16_t)(w[i >> 1] & 0xFFFFu);
        };
        int32_t y[6];
#pragma unroll
        for (int k = 0; k < 6; ++k)
            y[k] = exact_y(cfg, at16(qs + lane * 3, k),
                           [&](int l) { return at16(Fs + lane * 19, k * 6 + l); }, x);
        const uint32_t chi2 = chi_square(y[3], y[4], y[5]);
        const bool pass = e.y != NONE && chi2 <= cfg.chi2_cut;
        uint32_t flags = pass ? SVT_FLAG_PASS : 0u;
        if (((geo >> 19) & 127u) == 0) flags |= SVT_FLAG_NO_HITS;
        if (geo & (1u << 27)) flags |= SVT_FLAG_BAD_PATTERN;
        if (geo & (1u << 26)) flags |= SVT_FLAG_OVERFLOW;
        mine[0] = rd_id(da.z) | (flags << 24);
        mine[1] = pass ? e.y : NONE;
        mine[2] = pass ? chi2 : 0u;
#pragma unroll
        for (int k = 0; k < 3; ++k) mine[3 + k] = pass ? (uint32_t)y[k] : 0u;
    }
    __syncwarp();
    uint32_t pick = lane, n_pass = 0;
    if (head) {
        bool ok = mine[1] != NONE;
        for (uint32_t t = lane + 1; t < n_rec && rl.ent[t].x == e.x; ++t) {
            const uint32_t *a = stage + t * 6, *b = stage + pick * 6;
            if (a[1] != NONE && (!ok || a[2] < b[2] || (a[2] == b[2] && a[1] < b[1]))) {
                pick = t;
                ok = true;
            }
        }
        n_pass = ok ? 1u : 0u;
    }
    const uint32_t heads = __ballot_sync(0xffffffffu, head), n_out = __popc(heads) * 6u;
    if (head) rl.ent[__popc(heads & ((1u << lane) - 1u))] = make_uint2(e.x, pick);
    __syncwarp();
    for (uint32_t i = lane; i < n_out; i += 32) {
        const uint32_t k = i / 6;
        const uint2 o = rl.ent[k];
        out[(size_t)o.x * 6 + (i - k * 6)] = stage[o.y * 6 + (i - k * 6)];
    }
    __syncwarp();
    return n_pass;
}

// Chunks of consecutive roads that the warps claim (GROUP 1): roads_per_chunk
// roads each, but single roads for the last GUIDED_TAIL roads per warp, so that
// the warps finish together and a batch of few roads spreads over all of them,
// while a large batch does not queue on the counter (0.7 ns a claim).  Whole
// passes with chunks of 4 throughout and like this: scaled shape, 100 events
// 37.2 and 30.9 us, 3000 events 205.2 and 204.6; 1000 paired events 75.6 and
// 74.0; with single roads throughout 29.9, 211.8 and 80.7.  A tail of 1 road per
// warp leaves 100 events at 34.8, one of 4 costs 3 % for 32,000 short roads.
// (First claims handed out without the counter, or one counter for items and
// chunks, are 2 us faster for 100 events and 1-15 % slower for large batches.)
constexpr uint32_t GUIDED_TAIL = 2;
__device__ __forceinline__ uint32_t full_chunks(uint32_t R, uint32_t per, uint32_t warps) {
    return (R - min(R, GUIDED_TAIL * warps)) / per;
}
// the first road of chunk k (R or more: there is no such chunk)
__device__ __forceinline__ uint32_t chunk_first(uint32_t k, uint32_t n_full, uint32_t per,
                                                uint32_t R) {
    return k < n_full ? k * per : n_full * per + min(k - n_full, R);
}

// The fit of a whole batch by screening: items of split roads, then chunks of
// consecutive roads, each road by one warp.  Returns the passing roads whose
// records this lane wrote.
// A road or item whose list does not decide (many equal hits, shifts that leave
// few bits of chi2, every component saturated) is fitted by the exact form in the
// same slot; after such an item the warp screens one in 2, 4, 8, then 16 of the
// items that follow until one is decided.  Batches of such roads only, kernel and
// extraction, in us, the exact form for every road / this / every combination
// with digits of its own, which it did before: roads of 4096 combinations with
// equal hits, 256 of them 47 / 31 / 90, 25,600 131 / 168 / 730; of 15,625
// combinations (split) 33 / 39 / 116 and 441 / 487 / 3704; chi2 above SAT and no
// cut, 25,600 roads 132 / 111 / 299 and 441 / 471 / 976.  (Leaving the screen out
// for roads as well takes 168 to 149, but 1.5 % more for every other batch.)
template <bool GUARDED>
__device__ __forceinline__ uint32_t screen_path(
    ScreenSlot &slot, CandList &rl, const uint32_t *__restrict__ words,
    const RoadDesc *__restrict__ desc, const int16_t *__restrict__ F,
    const int16_t *__restrict__ q, const svt_config &cfg, const Screen &sc, const FusedRoads &fr,
    uint32_t n_big, uint32_t n_items, uint32_t R, uint32_t roads_per_chunk, uint32_t *out) {
    ScreenSmem &sm = slot.road;
    const BigList &bl = fr.bl;
    const int lane = threadIdx.x & 31;
    const Lanes<32> LW = lanes_of<32>(lane);
    uint32_t n_rec = 0, n_pass = 0;   // entries of rl (uniform over the warp)
    auto flush = [&]() {
        n_pass += flush_records(words, desc, F, q, cfg, out, rl, slot.flush, n_rec);
        n_rec = 0;
    };
    uint32_t skip = 0;   // the screen is left out where this mask hits the item's number
    // best (chi2 << 32) | c of rows [a_lo, a_hi), every combination exactly
    auto exact = [&](const RoadDesc &D, const Geo &g, uint32_t a_lo, uint32_t a_hi) {
        const uint32_t sh = 32u - cfg.oshift;
        const uint32_t init_chi = cfg.chi2_cut == 0xFFFFFFFFu ? 0xFFFFFFFFu : cfg.chi2_cut + 1u;
        WarpSmem &ws = reinterpret_cast<WarpSmem &>(slot);
        __syncwarp();
        road_setup<32>(ws, words, D, g, F, q, sh, cfg.xft_pairs, kColBias<GUARDED>, LW);
        const unsigned long long k =
            eval_rows<GUARDED, 32>(ws, g, a_lo, a_hi, cfg.qshift + sh, init_chi, LW);
        const uint32_t low = (uint32_t)k;
        __syncwarp();
        return k == ~0ull ? k : (k & 0xFFFFFFFF00000000ull) | ((low >> 9) * g.NB + (low & 511u));
    };
    while (n_items) {   // (no items: no claim, 3.5 us of queueing for a grid's warps)
        uint32_t it = 0;
        if (lane == 0) it = atomicAdd(bl.counters + 0, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= n_items) break;
        const uint32_t j = find_slot(bl.item_off, n_big, it, lane);
        const uint32_t r = __ldg(bl.road + j);
        const uint32_t k = it - __ldg(bl.item_off + j);
        RoadDesc D;
        D.a = __ldg(&desc[r].a);
        D.b = __ldg(&desc[r].b);
        const Geo g = geo_of(D);
        const uint32_t a_lo = k * fr.rows;
        const uint32_t a_hi = min(a_lo + fr.rows, g.NA);
        uint32_t n_c = UNSURE;
        if ((it & skip) == 0) {
            screen_load(sm, words, D, g, F, q, sc, cfg.xft_pairs, LW);
            screen_suffix(sm, g, LW);
            float thr;
            n_c = list_rows(sm, slot.cand, g, a_lo, a_hi, sc, thr, (uint32_t)lane);
            if (unsure(n_c, thr, cfg)) n_c = UNSURE;
            skip = n_c == UNSURE ? (2u * skip + 1u) & 15u : 0u;
        }
        const unsigned long long best = n_c == UNSURE ? exact(D, g, a_lo, a_hi)
                                                      : best_of_list(sm, slot.cand, n_c, cfg, LW);
        uint32_t last = 0;
        if (lane == 0) {
            if (best != ~0ull) atomicMin(fr.key + r, best);
            __threadfence();
            last = (atomicSub(bl.pending + j, 1u) == 1u) ? 1u : 0u;
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last) {   // every item of road r is done: list it with its final key
            if (n_rec == 32) flush();
            if (lane == 0) {
                __threadfence();
                // (the low word of these keys is the combination index itself)
                rl.ent[n_rec] = make_uint2(r, (uint32_t)__ldcg(fr.key + r));   // (or NONE)
            }
            n_rec += 1;
        }
        __syncwarp();
    }
    const uint32_t n_full = full_chunks(R, roads_per_chunk, gridDim.x * (blockDim.x >> 5));
    for (;;) {
        uint32_t k = 0;
        if (lane == 0) k = atomicAdd(bl.counters + 1, 1u);
        k = __shfl_sync(0xffffffffu, k, 0);
        const uint32_t c0 = chunk_first(k, n_full, roads_per_chunk, R);
        if (c0 >= R) break;
        const uint32_t n = k < n_full ? roads_per_chunk : 1u;
        uint4 da = make_uint4(0, 0, 0, 0), db = make_uint4(0, 0, 0, 0);
        if ((uint32_t)lane < n) {
            da = __ldg(&desc[c0 + lane].a);
            db = __ldg(&desc[c0 + lane].b);
        }
        for (uint32_t jj = 0; jj < n; ++jj) {
            const RoadDesc D = shfl_desc(da, db, jj);
            if (D.a.w > fr.small_max) continue;   // split road: done above
            if (n_rec > 32u - LIST_MAX) flush();
            uint32_t n_c = screen_road(sm, slot.cand, words, D, F, q, cfg, sc, LW);
            if (n_c == UNSURE) {
                // (read again: kept over the screen it spills)
                const RoadDesc E{__ldg(&desc[c0 + jj].a), __ldg(&desc[c0 + jj].b)};
                const Geo g = geo_of(E);
                const unsigned long long best = exact(E, g, 0, g.NA);
                if (lane == 0) slot.cand[0].x = (uint32_t)best;   // (UINT64_MAX reads as NONE)
                n_c = 1;
            }
            __syncwarp();
            const uint32_t n_e = max(n_c, 1u);   // at most LIST_MAX
            if ((uint32_t)lane < n_e)
                rl.ent[n_rec + lane] = make_uint2(c0 + jj, n_c ? slot.cand[lane].x : NONE);
            n_rec += n_e;
            __syncwarp();
        }
    }
    if (n_rec) flush();
    return n_pass;
}

// Mean evaluated combinations of a batch's roads from which on the batch is
// fitted by screening (one road per warp, GROUP 1; one form per launch, so that
// the warps keep to one path of code).  Its set-up, listing and exact step cost
// about 250 warp instructions a road more than the exact form's, its loop 13 less
// per 32 combinations: fit kernel, exact / screened, in us, 1500 events of 64
// roads: mean 244 combinations 80 / 92, 582: 119 / 123, 731: 121 / 121, 994: 143 /
// 142, 1337: 201 / 199, 1837: 207 / 178, 2927 (256-row items): 267 / 190, 3981: 338
// / 227, 4096: 287 / 190; at 100 events the line lies at the same place.
// The line was measured on batches whose roads are all alike.  In a mixed batch
// the mean decides for all roads, so that large ones among many small are fitted
// exactly though screening each of them alone would take less: in the scaled
// workload (mean 581) the 12 % of the roads above 1024 combinations hold 70 % of
// the combinations.
// (Screening every batch, with tables for several small roads at once, a lane
// to a small road or size classes of 4 to 32 lanes a road, took fewer
// instructions at small means but kept fewer warps busy: 1.1 to 1.7 times the
// exact form's time on the scaled workload.)
constexpr uint64_t SCREEN_MEAN = 1024;

// K4: persistent fit / cut / select / format.  GROUP 2: two consecutive SMALL
// roads of one chunk with the same geometry go to the two halves of the warp;
// GROUP 4: four consecutive TINY roads of the same geometry go to its four
// quarters (else two SMALL roads to its halves, as with GROUP 2); GROUP 32:
// every TINY road of the chunk goes to a lane of its own (lane k: the chunk's
// road k), then the warp fits the chunk's other roads one at a time.  Each is
// a separate instance, so that warps never switch between the code paths
// unless grouping was asked for.
// (GROUP 32 keeps every load of a lane's road in flight at once with up to 85
// registers a thread, blocks of at most 12 warps: 80 are used, three blocks of
// 8 warps per SM; with 64, loads were serialised or spilled and with 128 only
// 16 warps per SM were resident.  The others fit in 64, for two blocks of
// 512 threads.)
template <bool GUARDED, int GROUP>
__global__ void __launch_bounds__(GROUP == 32 ? 384 : 512, 2)
    k_fit_persistent(const uint32_t *__restrict__ words, const uint64_t *__restrict__ event_off,
                     const Dims *__restrict__ dims, const uint32_t *__restrict__ event_road,
                     const RoadDesc *__restrict__ desc, uint64_t *counts, uint64_t road_cap,
                     const int16_t *__restrict__ F, const int16_t *__restrict__ q,
                     const svt_config cfg, const Screen sc, const FusedRoads fr,
                     uint32_t roads_per_chunk, uint32_t *out, unsigned long long *status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WarpSmem &sm = *reinterpret_cast<WarpSmem *>(smem_raw + SLOT_BYTES * (threadIdx.x >> 5));
    unsigned char *list = smem_raw + SLOT_BYTES * (blockDim.x >> 5) +
                          sizeof(RecordList) * (threadIdx.x >> 5);
    RecordList &rl = *reinterpret_cast<RecordList *>(list);
    const int lane = threadIdx.x & 31;
    const Lanes<32> LW = lanes_of<32>(lane);
    wait_prior_grid();   // road extraction has completed (see launch_after)
    // per-event rules first, whatever the status, so that the key stays the
    // smallest over all rules
    check_events(words, event_off, dims->n_words, dims->n_events, event_road, status,
                 (uint64_t)blockIdx.x * blockDim.x + threadIdx.x,
                 (uint64_t)gridDim.x * blockDim.x);
    const BigList &bl = fr.bl;
    const unsigned long long rv = *(volatile unsigned long long *)bl.reserve;
    const uint32_t n_big = (uint32_t)rv, n_items = (uint32_t)(rv >> 32);
    if (blockIdx.x == 0 && threadIdx.x == 0) counts[1] = n_items;
    if (!status_ok(status)) return;
    const uint64_t R64 = counts[0];
    if (R64 > road_cap || R64 == 0) return;
    const uint32_t R = (uint32_t)R64;
    if constexpr (GROUP == 1) {
        if (counts[2] >= SCREEN_MEAN * R64) {
            const uint32_t n_pass = __reduce_add_sync(
                0xffffffffu,
                screen_path<GUARDED>(reinterpret_cast<ScreenSlot &>(sm),
                                     *reinterpret_cast<CandList *>(list), words, desc, F, q, cfg,
                                     sc, fr, n_big, n_items, R, roads_per_chunk, out));
            if (lane == 0 && n_pass)
                atomicAdd((unsigned long long *)(counts + 3), (unsigned long long)n_pass);
            return;
        }
    }
    const uint32_t sh = 32u - cfg.oshift, qsh = cfg.qshift + sh;
    const uint32_t init_chi = cfg.chi2_cut == 0xFFFFFFFFu ? 0xFFFFFFFFu : cfg.chi2_cut + 1u;
    // GROUP 32: lanes to a tiny road, so that chunks of 32, 16 or at most 8
    // roads fill the warp
    const uint32_t L = GROUP != 32 ? 1u : roads_per_chunk > 16 ? 1u : roads_per_chunk > 8 ? 2u : 4u;
    uint32_t n_rec = 0;    // entries of rl (uniform over the warp)
    uint32_t n_pass = 0;   // passing roads whose records this lane wrote, summed at exit
    // Each lane forms one listed record into the warp's road slot (free
    // between roads), then the warp stores the 6 * n_rec words with
    // consecutive lanes on consecutive words, so that the records of
    // consecutive roads go out as contiguous runs.
    auto flush = [&]() {
        __syncwarp();
        uint32_t *stage = reinterpret_cast<uint32_t *>(&sm);
        if ((uint32_t)lane < n_rec &&
            form_record(words, desc, rl.road[lane], rl.key[lane], F, q, cfg, stage + lane * 6))
            ++n_pass;
        __syncwarp();
        for (uint32_t e = (uint32_t)lane; e < n_rec * 6; e += 32) {
            const uint32_t i = e / 6;
            out[(size_t)rl.road[i] * 6 + (e - i * 6)] = stage[e];
        }
        n_rec = 0;
        __syncwarp();
    };

    // With four tiny roads per warp (GROUP 4) or one per lane (GROUP 32) a
    // batch without split roads skips phase 1 and hands every warp its first
    // chunk of phase 2 statically (warp w of block b takes chunk
    // w * gridDim.x + b, so that a batch of fewer chunks than warps spreads
    // over the SMs), the rest through the
    // counter counted from nw: the grid's warps then start without queueing
    // on one address, which for chunks this short is a large part of the
    // kernel (the paper's shape, 3000 events: 43 -> 37 us).  Otherwise every
    // claim goes through the counters (static first claims made the scaled
    // shape 6 % slower).
    const uint32_t nw = gridDim.x * (blockDim.x >> 5);
    const bool static_first = (GROUP == 4 || GROUP == 32) && n_items == 0;

    // phase 1: items of split roads
    // (GROUP 1: none, no claim: a grid's warps queue 3.5 us on one counter)
    while (GROUP == 1 ? n_items != 0 : !static_first) {
        uint32_t it = 0;
        if (lane == 0) it = atomicAdd(bl.counters + 0, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= n_items) break;
        const uint32_t j = find_slot(bl.item_off, n_big, it, lane);
        const uint32_t r = __ldg(bl.road + j);
        const uint32_t k = it - __ldg(bl.item_off + j);
        RoadDesc D;
        D.a = __ldg(&desc[r].a);
        D.b = __ldg(&desc[r].b);
        const Geo g = geo_of(D);
        road_setup<32>(sm, words, D, g, F, q, sh, cfg.xft_pairs, kColBias<GUARDED>, LW);
        const uint32_t a_lo = k * fr.rows;
        const uint32_t a_hi = min(a_lo + fr.rows, g.NA);
        const unsigned long long best = eval_rows<GUARDED, 32>(sm, g, a_lo, a_hi, qsh, init_chi, LW);
        uint32_t last = 0;
        if (lane == 0) {
            if (best != ~0ull) atomicMin(fr.key + r, best);
            __threadfence();
            last = (atomicSub(bl.pending + j, 1u) == 1u) ? 1u : 0u;
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last) {   // every item of road r is done: list it with its final key
            if (n_rec == 32) flush();
            if (lane == 0) {
                __threadfence();
                rl.key[n_rec] = __ldcg(fr.key + r);
                rl.road[n_rec] = r;
            }
            n_rec += 1;
        }
        __syncwarp();
    }

    // phase 2: chunks of consecutive roads, each fitted whole by this warp,
    // or two SMALL roads side by side by its two halves
    for (bool first = true;; first = false) {
        uint32_t c0, n;
        if constexpr (GROUP == 1) {
            uint32_t k = 0;
            if (lane == 0) k = atomicAdd(bl.counters + 1, 1u);
            k = __shfl_sync(0xffffffffu, k, 0);
            const uint32_t full = full_chunks(R, roads_per_chunk, nw);
            c0 = chunk_first(k, full, roads_per_chunk, R);
            if (c0 >= R) break;
            n = k < full ? roads_per_chunk : 1u;
        } else {
            uint32_t k = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;   // chunk index
            if (!(first && static_first)) {
                if (lane == 0) k = atomicAdd(bl.counters + 1, 1u) + (static_first ? nw : 0u);
                k = __shfl_sync(0xffffffffu, k, 0);
            }
            if ((uint64_t)k * roads_per_chunk >= R) break;
            c0 = k * roads_per_chunk;
            n = min(roads_per_chunk, R - c0);
        }
        // this lane's road of the chunk (GROUP 32: L lanes to a road)
        const uint32_t jr = (uint32_t)lane / L;
        uint4 da = make_uint4(0, 0, 0, 0), db = make_uint4(0, 0, 0, 0);
        if (jr < n) {
            da = __ldg(&desc[c0 + jr].a);
            db = __ldg(&desc[c0 + jr].b);
        }
        if constexpr (GROUP == 32) {
            // the chunk's TINY roads, L lanes each, their records formed by
            // their first lanes and stored at once as runs of consecutive
            // words ...
            const bool mine = jr < n && (db.x & GEO_TINY) && da.w <= fr.small_max;
            const uint32_t lm = __ballot_sync(0xffffffffu, mine);
            const bool first_lane = ((uint32_t)lane & (L - 1u)) == 0;
            if (lm) {
                LaneRecord rec;
                if (mine)
                    rec = lane_fit<GUARDED>(*reinterpret_cast<LaneTables *>(&sm), words, da, db, F,
                                            q, cfg, sh, qsh, init_chi, lane, L, lm);
                __syncwarp();
                uint32_t *stage = reinterpret_cast<uint32_t *>(&sm);
                if (mine && first_lane) {
#pragma unroll
                    for (int j = 0; j < 6; ++j) stage[jr * 6 + j] = rec.w[j];
                    n_pass += rec.pass ? 1u : 0u;
                }
                __syncwarp();
                for (uint32_t e = (uint32_t)lane; e < n * 6; e += 32) {
                    const uint32_t i = e / 6;
                    if ((lm >> (i * L)) & 1u) out[(size_t)(c0 + i) * 6 + (e - i * 6)] = stage[e];
                }
                __syncwarp();
            }
            // ... then the others (not split) one per warp
            uint32_t rest = __ballot_sync(0xffffffffu,
                                          first_lane && jr < n && !mine && da.w <= fr.small_max);
            while (rest) {
                const uint32_t src = (uint32_t)__ffs(rest) - 1u, jj = src / L;
                rest &= rest - 1u;
                const RoadDesc D = shfl_desc(da, db, src);
                if (n_rec == 32) flush();
                const unsigned long long best =
                    fit_road<GUARDED, 32>(sm, words, D, F, q, cfg, sh, qsh, init_chi, LW);
                if (lane == 0) {
                    rl.key[n_rec] = best;
                    rl.road[n_rec] = c0 + jj;
                }
                n_rec += 1;
                __syncwarp();
            }
        } else {
            for (uint32_t jj = 0; jj < n;) {
                const RoadDesc D = shfl_desc(da, db, jj);
                if (D.a.w > fr.small_max) {   // split road: done in phase 1
                    ++jj;
                    continue;
                }
                if (n_rec > 32 - GROUP) flush();   // room for GROUP more
                if constexpr (GROUP == 4) {
                    // four TINY roads with the same hits per layer and the same
                    // number of combinations to evaluate, so that the quarters
                    // run their loops in step
                    if ((D.b.x & GEO_TINY) && jj + 3 < n) {
                        // lane k holds road c0 + k: one vote over the next four
                        const bool same = (db.x & GEO_TINY) && da.y == D.a.y && da.w == D.a.w;
                        const uint32_t votes = __ballot_sync(0xffffffffu, same);
                        if (((votes >> jj) & 15u) == 15u) {
                            // this lane's quarter and road
                            const uint32_t qt = (uint32_t)lane >> 3;
                            QuarterSmem &qs = reinterpret_cast<QuarterSmem *>(&sm)[qt];
                            const RoadDesc Dq = shfl_desc(da, db, jj + qt);
                            const Lanes<8> LQ = lanes_of<8>(lane);
                            Geo g = geo_of(Dq);
                            unsigned long long best = ~0ull;
                            if (g.C_eval) {
                                quarter_geometry(g, Dq.a.y, cfg.xft_pairs);
                                road_setup<8>(qs, words, Dq, g, F, q, sh, cfg.xft_pairs,
                                              kColBias<GUARDED>, LQ);
                                best = quarter_key(
                                    eval_rows<GUARDED, 8>(qs, g, 0, g.NA, qsh, init_chi, LQ), g.NB,
                                    Dq.b.y);
                            }
                            if ((lane & 7) == 0) {
                                rl.key[n_rec + qt] = best;
                                rl.road[n_rec + qt] = c0 + jj + qt;
                            }
                            n_rec += 4;
                            jj += 4;
                            __syncwarp();
                            continue;
                        }
                    }
                }
                if constexpr (GROUP >= 2) {
                    // two SMALL roads of the same geometry (split, NBp, ntop and NA),
                    // so that the two halves run their loops in step
                    if ((D.b.x & GEO_SMALL) && jj + 1 < n) {
                        const RoadDesc D2 = shfl_desc(da, db, jj + 1);
                        if ((D2.b.x & GEO_SMALL) && ((D.b.x ^ D2.b.x) & 0x1FFFu) == 0 &&
                            D.b.z == D2.b.z && D2.a.w <= fr.small_max) {
                            const uint32_t h = (uint32_t)lane >> 4;   // this lane's half and road
                            HalfSmem &hs = reinterpret_cast<HalfSmem *>(&sm)[h];
                            const unsigned long long best = fit_road<GUARDED, 16>(
                                hs, words, h ? D2 : D, F, q, cfg, sh, qsh, init_chi,
                                lanes_of<16>(lane));
                            if ((lane & 15) == 0) {
                                rl.key[n_rec + h] = best;
                                rl.road[n_rec + h] = c0 + jj + h;
                            }
                            n_rec += 2;
                            jj += 2;
                            __syncwarp();
                            continue;
                        }
                    }
                }
                const unsigned long long best =
                    fit_road<GUARDED, 32>(sm, words, D, F, q, cfg, sh, qsh, init_chi, LW);
                if (lane == 0) {
                    rl.key[n_rec] = best;
                    rl.road[n_rec] = c0 + jj;
                }
                n_rec += 1;
                jj += 1;
                __syncwarp();
            }
        }
    }
    flush();
    n_pass = __reduce_add_sync(0xffffffffu, n_pass);
    if (lane == 0 && n_pass)
        atomicAdd((unsigned long long *)(counts + 3), (unsigned long long)n_pass);
}

}  // namespace

size_t fit_smem_bytes(int warps_per_block) {
    return (SLOT_BYTES + sizeof(RecordList)) * (size_t)warps_per_block;
}

namespace {

// see Screen: rounded up at every step
Screen make_screen(const svt_config &cfg) {
    const double u = 0x1p-24, P = std::ldexp(1.0, -(int)cfg.oshift);
    const double M = (6.0 * 0x1p30 + std::ldexp(1.0, 15 + (int)cfg.qshift)) * P + 1.0;
    const double delta = std::sqrt(3.0) * (0.5 + 10.0 * u * M) * (1.0 + 1e-6);
    const double cut = std::sqrt((double)std::min(cfg.chi2_cut, SAT)) + delta;
    Screen sc;
    sc.f_scale = (float)P;
    sc.q_scale = (float)std::ldexp(1.0, (int)cfg.qshift - (int)cfg.oshift);
    sc.delta = (float)(delta * (1.0 + 1e-6));
    sc.thr = (float)(cut * cut * (1.0 + 1e-5));
    return sc;
}

}  // namespace


int fit_persistent_blocks_per_sm(int warps_per_block, uint32_t group) {
    const size_t smem = fit_smem_bytes(warps_per_block);
    int occ = 1 << 30;
    auto one = [&](auto kernel) {
        int n = 0;
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, warps_per_block * 32, smem) !=
            cudaSuccess)
            n = 0;
        occ = n < occ ? n : occ;
    };
    // both instances of the group (the chi2 cut picks one at launch)
    if (group == 32) {
        one(k_fit_persistent<true, 32>);
        one(k_fit_persistent<false, 32>);
    } else if (group == 4) {
        one(k_fit_persistent<true, 4>);
        one(k_fit_persistent<false, 4>);
    } else if (group == 2) {
        one(k_fit_persistent<true, 2>);
        one(k_fit_persistent<false, 2>);
    } else {
        one(k_fit_persistent<true, 1>);
        one(k_fit_persistent<false, 1>);
    }
    return occ;
}

cudaError_t launch_fit_persistent(const uint32_t *words, const uint64_t *event_off,
                                  const Dims *dims, const uint32_t *event_road,
                                  const RoadDesc *desc, uint64_t *counts, uint64_t road_cap,
                                  const int16_t *F, const int16_t *q, const svt_config cfg,
                                  const FusedRoads fr, uint32_t roads_per_chunk, uint32_t group,
                                  uint32_t *out, unsigned long long *status,
                                  int warps_per_block, int grid, cudaStream_t st) {
    const size_t smem = fit_smem_bytes(warps_per_block);
    const bool guarded = cfg.chi2_cut < SAT;
    const Screen sc = make_screen(cfg);
    auto launch = [&](auto kernel) {
        launch_after(kernel, grid, warps_per_block * 32, smem, st, words, event_off, dims,
                     event_road, desc, counts, road_cap, F, q, cfg, sc, fr, roads_per_chunk, out,
                     status);
    };
    if (guarded) {
        if (group == 32) launch(k_fit_persistent<true, 32>);
        else if (group == 4) launch(k_fit_persistent<true, 4>);
        else if (group == 2) launch(k_fit_persistent<true, 2>);
        else launch(k_fit_persistent<true, 1>);
    } else {
        if (group == 32) launch(k_fit_persistent<false, 32>);
        else if (group == 4) launch(k_fit_persistent<false, 4>);
        else if (group == 2) launch(k_fit_persistent<false, 2>);
        else launch(k_fit_persistent<false, 1>);
    }
    return cudaGetLastError();
}

}  // namespace svt
