// Seed-and-verify search (sm_103a): the reads whose error-free parts lead to few
// places in the text are answered from those places; the tree search is left the
// rest.
//
// A transcript with at most b differences, cut at b + 1 parts of the read, leaves
// one part without any: that part occurs in the text as it is, on the
// transcript's diagonal.  So every place of every part, looked at base by base,
// gives every target within b differences.  With at most one gap a transcript is
// a prefix on one diagonal, a run of inserted or deleted bases, and a suffix on
// another; its target is (start on the first, end on the second), and the fewest
// mismatches over the gap's places is the target's least witness, as the other
// terms of the witness follow from the gap's length.  The search's limits (gap
// and seed limits, end window, N) are those of aln_search.cuh, read index p of
// the reverse strand being pattern index m - 1 - p here.  Both strands work on X:
// the reverse strand's pattern is the reverse complement of the read.
//
// A target's rows in the suffix array of its strand's text come from the derived
// inverse (its sampled entries and at most three LF steps).  All places of a
// target are found, so equal targets, which are neighbours in the suffix array,
// give its interval; targets of different lengths with the same interval merge as
// in the tree search.
//
// G lanes a read: one lane per (strand, part) finds the part's rows (one look-up
// in the table of k-mers, a few LF steps in a repeat), then the lanes share the
// places out.
//
// Where the tree search of a read of 100 bases expands about 1900 nodes, one after
// the other, this takes 2 (z + 1) look-ups at once and looks at about ten places
// (100 Mbp), each a read of the suffix array and of the text.  1 M reads of 100
// bases at z = 4 on 100 Mbp: 65 -> 3.0 ms; 400 000 reads of 36 to 250 bases on
// 3.1 Gbp: 738 -> 14.1 ms.  It is bound by the latency of
// those four dependent random reads and by instruction issue, not by bandwidth.
#pragma once

#include <cstdint>

#include "aln_search.cuh"

namespace aln {

#ifndef ALN_EXTEND
#define ALN_EXTEND 24
#endif
// Bases a part grows by at most, past the table's: 300 000 mates on 3.1 Gbp take
// 5.47 / 5.42 / 5.36 ms with 6 / 12 / 24, unique reads do not grow at all.
constexpr int kExtend = ALN_EXTEND;
constexpr uint32_t kWideRows = 1u << 20;  // a part's rows saturate here
#ifndef ALN_MANY_PLACES
#define ALN_MANY_PLACES 3
#endif
// Places per lane from which a pass starts over with fewer, longer parts.  1, 2, 3, 6
// and 8 are within 2 % of each other on the 3.1 Gbp batches (1 costs unique reads
// of 100 Mbp 13 %).
constexpr uint32_t kManyPlaces = ALN_MANY_PLACES;

// Row of the suffix of text w that starts at position pos (0 .. n).
__device__ __forceinline__ uint32_t row_of(const DIndex &X, int w, uint32_t pos) {
    const DText &T = X.t[w];
    const uint64_t s = (static_cast<uint64_t>(pos) + kIsaStep - 1) / kIsaStep;
    const uint64_t at = s * kIsaStep;
    uint32_t row = 0, steps = T.n - pos;  // past the last sampled position: from the suffix "$", row 0
    if (at <= T.n) {
        row = __ldg(X.isa[w] + s);
        steps = static_cast<uint32_t>(at) - pos;
    }
    for (; steps; steps--) row = lf_row(T, row);
    return row;
}

__device__ __forceinline__ uint32_t low_mask(int k) {  // the low k bits, k clamped to 0..32
    return __funnelshift_lc(0xFFFFFFFFu, 0u, static_cast<uint32_t>(max(k, 0)));
}

// Bits [from, to) of a read's mask that fall into its word w.
__device__ __forceinline__ uint32_t span_mask(int from, int to, int w) {
    return low_mask(to - 32 * w) & ~low_mask(from - 32 * w);
}

constexpr int kPlaneWords = 8;  // words of a mask of ALN_MAX_READ_LEN bases

// A pattern (a read on one strand, in text order) as bit planes in shared memory.
struct Pattern {
    uint32_t lo[kPlaneWords], hi[kPlaneWords], nn[kPlaneWords];
};

// mis = the pattern's mismatches (bit j = pattern index j) with the pattern's
// first base on text position x.
__device__ __forceinline__ void mismatches(const uint2 *text, const Pattern &P, long long x, int m,
                                           uint32_t mis[kPlaneWords]) {
    const uint2 *t = text + (x >> 5);
    const uint32_t s = static_cast<uint32_t>(x & 31);
    uint2 a = __ldg(t);
#pragma unroll
    for (int w = 0; w < kPlaneWords; w++) {
        mis[w] = 0;
        if (32 * w < m) {
            const uint2 b = __ldg(t + w + 1);
            const uint32_t lo = __funnelshift_r(a.x, b.x, s), hi = __funnelshift_r(a.y, b.y, s);
            mis[w] = ((lo ^ P.lo[w]) | (hi ^ P.hi[w]) | P.nn[w]) & low_mask(m - 32 * w);
            a = b;
        }
    }
}

__device__ __forceinline__ uint32_t count_in(const uint32_t mis[kPlaneWords], int from, int to) {
    uint32_t c = 0;
#pragma unroll
    for (int w = 0; w < kPlaneWords; w++) {
        if (32 * w >= to) break;
        c += __popc(mis[w] & span_mask(from, to, w));
    }
    return c;
}

// Index of the (r + 1)-th mismatch from the start (m if there are fewer).
__device__ __forceinline__ int nth_low(const uint32_t mis[kPlaneWords], uint32_t r, int m) {
    uint32_t x = 0;
    int at = -1;
#pragma unroll
    for (int w = 0; w < kPlaneWords; w++) {
        if (32 * w >= m) break;
        const uint32_t c = __popc(mis[w]);
        if (at < 0) {
            if (r < c) {
                x = mis[w];
                at = 32 * w;
            } else {
                r -= c;
            }
        }
    }
    if (at < 0) return m;
    for (; r; r--) x &= x - 1;
    return at + __ffs(x) - 1;
}

// Index of the (r + 1)-th mismatch from the end (-1 if there are fewer).
__device__ __forceinline__ int nth_high(const uint32_t mis[kPlaneWords], uint32_t r) {
    uint32_t x = 0;
    int at = -1;
#pragma unroll
    for (int w = kPlaneWords - 1; w >= 0; w--) {
        const uint32_t c = __popc(mis[w]);
        if (at < 0) {
            if (r < c) {
                x = mis[w];
                at = 32 * w;
            } else {
                r -= c;
            }
        }
    }
    if (at < 0) return -1;
    for (; r; r--) x &= ~(0x80000000u >> __clz(x));
    return at + 31 - __clz(x);
}

// The places of one gap of length g between a prefix with mismatches A and a
// suffix with mismatches B (a deletion, or an insertion of pattern bases
// [p, p + g)): the fewest mismatches over p in [plo, phi] that keep the seed
// limit, or none (> most).  Only the few gap lengths whose diagonals both match
// come past the two bounds below, so the walk over p is rare and short.
struct SeedZone {
    int from, to;      // pattern indices of the seed ([0, 0): no seed)
    uint32_t most;     // differences allowed in it
    bool reverse;      // the pattern is the reverse complement
};

__device__ __forceinline__ uint32_t best_gap(const uint32_t A[kPlaneWords], const uint32_t B[kPlaneWords], int m, int g,
                                             bool del, int plo, int phi, uint32_t most, const SeedZone &Z) {
    constexpr uint32_t kNone = 0xFFFFFFFFu;
    const int gi = del ? 0 : g;
    phi = min(phi, nth_low(A, most, m));           // the prefix has at most `most` mismatches
    plo = max(plo, nth_high(B, most) + 1 - gi);    // and so has the suffix
    if (plo > phi) return kNone;
    uint32_t a[kPlaneWords], b[kPlaneWords];
#pragma unroll
    for (int w = 0; w < kPlaneWords; w++) {
        a[w] = A[w];
        b[w] = B[w];
    }
    uint32_t f = count_in(A, 0, plo) + count_in(B, plo + gi, m);
    uint32_t sa = 0, sb = 0;
    const bool seeded = Z.to > Z.from;
    if (seeded) {
        sa = count_in(A, Z.from, min(Z.to, plo));
        sb = count_in(B, max(Z.from, plo + gi), Z.to);
    }
    uint32_t best = kNone;
    for (int p = plo;; p++) {
        bool ok = f <= most && f < best;
        if (ok && seeded) {
            // gap bases in the seed: inserted bases by index; a deletion at the
            // read index that follows it (p on the forward strand, and p - 1 in
            // pattern order on the reverse strand)
            const int at = Z.reverse ? p - 1 : p;
            const int in = del ? (at >= Z.from && at < Z.to ? g : 0) : max(0, min(Z.to, p + g) - max(Z.from, p));
            ok = sa + sb + static_cast<uint32_t>(in) <= Z.most;
        }
        if (ok) best = f;
        if (p >= phi) break;
        const uint32_t ia = (a[p >> 5] >> (p & 31)) & 1u, q = static_cast<uint32_t>(p + gi);
        const uint32_t ib = (b[q >> 5] >> (q & 31u)) & 1u;  // q < m: p < phi <= m - gi
        f += ia - ib;
        if (seeded) {
            if (p >= Z.from && p < Z.to) sa += ia;
            if (static_cast<int>(q) >= Z.from && static_cast<int>(q) < Z.to) sb -= ib;
        }
    }
    return best;
}

// Whether diagonal d can be the prefix (or, `ahead`, the suffix) of a target with
// a gap: its own mismatches and the end window bound the gap's place, and the
// bases past that place (of them, the 32 at the read's far end) have to fit a
// neighbouring diagonal.  One word a diagonal in the lane that found d, against
// the masks of the whole read by all lanes: what has no indel ends here, both the
// copies of a repeat and the read's own place.
__device__ __forceinline__ bool gap_fits(const uint2 *text, const Pattern &P, long long d, int m,
                                         const uint32_t mis[kPlaneWords], int F, int gmost, int e, bool ahead) {
    const int i = ahead ? 0 : max(m - 32, 0), w = i >> 5;
    const uint32_t s = static_cast<uint32_t>(i & 31);
    const int v = min(w + 1, kPlaneWords - 1);
    const uint32_t lo = __funnelshift_r(P.lo[w], P.lo[v], s), hi = __funnelshift_r(P.hi[w], P.hi[v], s);
    const uint32_t nn = __funnelshift_r(P.nn[w], P.nn[v], s);
    const int bound = ahead ? nth_high(mis, F - 1) + 1 : nth_low(mis, F - 1, m);
    // the 64 bases from 8 before the far word on diagonal d
    const long long x = d + i - 8;
    const uint2 *at = text + (x >> 5);
    const uint32_t t = static_cast<uint32_t>(x & 31);
    const uint2 a = __ldg(at), b = __ldg(at + 1), c = __ldg(at + 2);
    const uint32_t lo0 = __funnelshift_r(a.x, b.x, t), lo1 = __funnelshift_r(b.x, c.x, t);
    const uint32_t hi0 = __funnelshift_r(a.y, b.y, t), hi1 = __funnelshift_r(b.y, c.y, t);
    for (int q = 0; q < 2 * gmost; q++) {
        const int g = (q >> 1) + 1;
        const bool del = q & 1;
        const int window = del ? max(e, 1) : e, gi = del ? 0 : g;
        const uint32_t zone = ahead ? low_mask(max(bound - gi, window))
                                    : low_mask(m - i) & ~low_mask(min(bound, m - window - gi) + gi - i);
        const uint32_t by = static_cast<uint32_t>(del != ahead ? 8 + g : 8 - g);
        const uint32_t far = (__funnelshift_r(lo0, lo1, by) ^ lo) | (__funnelshift_r(hi0, hi1, by) ^ hi) | nn;
        if (__popc(far & zone) + g <= F) return true;
    }
    return false;
}

// Shared memory of one read's lanes.
template <int E>
struct SeedRead {
    Pattern pat[2];
    uint32_t bases[18];              // the read, 2 bits a base (two words past it)
    uint32_t count;                  // targets found (may pass E)
    uint32_t start[E], key[E];       // target start in X; the tree search's candidate key
    uint32_t row[E], end[E];         // its rows [row, end)
};

// `width` low-order bases from index i of the packed read.
__device__ __forceinline__ uint32_t bases_at(const uint32_t *bases, uint32_t i, uint32_t width) {
    const uint32_t w = i >> 4, s = 2 * (i & 15u);
    const uint32_t v = __funnelshift_r(bases[w], bases[w + 1], s);
    return v & low_mask(static_cast<int>(2 * width));
}

// Base order reversed in the low `width` bases.
__device__ __forceinline__ uint32_t reverse_bases(uint32_t v, uint32_t width) {
    const uint32_t r = __brev(v);
    const uint32_t x = ((r & 0x55555555u) << 1) | ((r >> 1) & 0x55555555u);
    return width ? x >> (32u - 2u * width) : 0u;
}

// Even and odd bits of a word, each as 16 bits.
__device__ __forceinline__ uint32_t even_bits(uint32_t x) {
    x &= 0x55555555u;
    x = (x | (x >> 1)) & 0x33333333u;
    x = (x | (x >> 2)) & 0x0F0F0F0Fu;
    x = (x | (x >> 4)) & 0x00FF00FFu;
    return (x | (x >> 8)) & 0x0000FFFFu;
}

template <int G>
__device__ __forceinline__ uint32_t group_min(uint32_t v) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) v = min(v, __shfl_xor_sync(0xFFFFFFFFu, v, o, G));
    return v;
}

template <int G>
__device__ __forceinline__ uint32_t group_sum(uint32_t v) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o, G);
    return v;
}

// X[a .. a+L) == X[b .. b+L)
__device__ __forceinline__ bool same_text(const uint2 *text, uint32_t a, uint32_t b, uint32_t L) {
    const uint2 *ta = text + (a >> 5), *tb = text + (b >> 5);
    const uint32_t sa = a & 31u, sb = b & 31u;
    for (uint32_t w = 0; 32 * w < L; w++) {
        const uint2 a0 = __ldg(ta + w), a1 = __ldg(ta + w + 1), b0 = __ldg(tb + w), b1 = __ldg(tb + w + 1);
        const uint32_t d = (__funnelshift_r(a0.x, a1.x, sa) ^ __funnelshift_r(b0.x, b1.x, sb)) |
                           (__funnelshift_r(a0.y, a1.y, sa) ^ __funnelshift_r(b0.y, b1.y, sb));
        if (d & low_mask(static_cast<int>(L - 32 * w))) return false;
    }
    return true;
}

__device__ __forceinline__ uint32_t key_diffs(uint32_t key) { return (key >> 28) & 7u; }

__device__ __forceinline__ uint32_t key_score(const SearchParams &p, uint32_t key) {
    return p.sc_mm * ((key >> 16) & 15u) + p.sc_go * ((key >> 24) & 15u) + p.sc_ge * ((key >> 20) & 15u);
}

__device__ __forceinline__ uint32_t target_key(uint32_t strand, uint32_t len, uint32_t mm, uint32_t g) {
    return (strand << 31) | ((mm + g) << 28) | ((g ? 1u : 0u) << 24) | ((g ? g - 1u : 0u) << 20) | (mm << 16) | len;
}

// A target found: recorded unless it is among the first `have`, those of the
// rounds before (two lanes may record it in one round; the reduction drops the
// second).
template <int E>
__device__ __forceinline__ void add_target(SeedRead<E> &S, uint32_t have, uint32_t at, uint32_t key) {
    for (uint32_t j = 0; j < have; j++)
        if (S.start[j] == at && S.key[j] == key) return;
    const uint32_t j = atomicAdd(&S.count, 1u);
    if (j < E) {
        S.start[j] = at;
        S.key[j] = key;
    }
}

__device__ __forceinline__ void put_hit(aln_hit *to, uint32_t k, uint32_t l, uint32_t key) {
    aln_hit h;
    h.k = k;
    h.l = l;
    h.aligned_len = static_cast<uint16_t>(key & 0xFFFFu);
    h.strand = static_cast<uint8_t>(key >> 31);
    h.n_diff = static_cast<uint8_t>(key_diffs(key));
    h.n_mm = static_cast<uint8_t>((key >> 16) & 15u);
    h.n_gapo = static_cast<uint8_t>((key >> 24) & 15u);
    h.n_gape = static_cast<uint8_t>((key >> 20) & 15u);
    h.reserved = 0;
    *to = h;
}

template <bool SCORE>
__device__ __forceinline__ void empty_result(aln_read_result *to, uint32_t flags) {
    aln_read_result out;
    out.c0 = out.c1 = 0;
    out.n_hits = 0;
    out.flags = static_cast<uint8_t>(flags);
    out.d_best = 255;
    out.best_score = SCORE ? 255 : 0;
    *to = out;
}

// Gapped targets of diagonal d by the lanes of its group, one (gap, side) a lane;
// returns the fewest differences this lane found.
template <int G, int E>
__device__ __forceinline__ uint32_t gap_targets(const uint2 *text, uint32_t n, SeedRead<E> &S, uint32_t have, int m,
                                             long long d, int first_end, int last_start, uint32_t F, uint32_t gmost,
                                             int e, SeedZone Z) {
    const uint32_t strand = Z.reverse ? 1u : 0u;
    const Pattern &P = S.pat[strand];
    uint32_t found = 255;
    for (uint32_t q = threadIdx.x & (G - 1); q < 4 * gmost; q += G) {
        const int g = static_cast<int>(q >> 2) + 1;
        const bool del = q & 1u, side = q & 2u;  // side 0: a part lies before the gap, 1: after it
        const long long other = side == del ? d - g : d + g;
        const long long a = side ? other : d;
        const int L = del ? m + g : m - g;
        int plo = del ? max(e, 1) : e;
        int phi = del ? m - plo : m - plo - g;
        if (side) phi = min(phi, last_start - (del ? 0 : g));
        else plo = max(plo, first_end);
        if (static_cast<uint32_t>(g) > F || L < 1 || a < 0 || a + L > static_cast<long long>(n) || plo > phi) continue;
        uint32_t pre[kPlaneWords], suf[kPlaneWords];  // mismatches on the prefix's and on the suffix's diagonal
        mismatches(text, P, a, m, pre);
        mismatches(text, P, side ? d : other, m, suf);
        const uint32_t f = best_gap(pre, suf, m, g, del, plo, phi, F - g, Z);
        if (f != 0xFFFFFFFFu) {
            add_target(S, have, static_cast<uint32_t>(a),
                       target_key(strand, static_cast<uint32_t>(L), f, static_cast<uint32_t>(g)));
            found = min(found, f + static_cast<uint32_t>(g));
        }
    }
    return found;
}

// Bitonic sort of a read's first P entries (a power of two, the same for every
// group of the warp) by its G lanes; less(i, j) compares two entries.
template <int G, int E, class Less>
__device__ __forceinline__ void sort_targets(SeedRead<E> &S, uint32_t P, Less less) {
    const uint32_t l = threadIdx.x & (G - 1);
    for (uint32_t k = 2; k <= P; k <<= 1)
        for (uint32_t j = k >> 1; j; j >>= 1) {
            for (uint32_t i = l; i < P / 2; i += G) {
                const uint32_t x = ((i & ~(j - 1u)) << 1) | (i & (j - 1u)), y = x | j;
                if (less(y, x) == ((x & k) == 0)) {
                    const uint32_t s = S.start[x], t = S.key[x], r = S.row[x], e = S.end[x];
                    S.start[x] = S.start[y];
                    S.key[x] = S.key[y];
                    S.row[x] = S.row[y];
                    S.end[x] = S.end[y];
                    S.start[y] = s;
                    S.key[y] = t;
                    S.row[y] = r;
                    S.end[y] = e;
                }
            }
            __syncwarp();
        }
}

// The entries of the first P that keep(e) holds for move to the front, in order;
// the others become entries that sort last.  Returns how many are kept.
template <int G, int E, class Keep>
__device__ __forceinline__ uint32_t pack_targets(SeedRead<E> &S, uint32_t P, unsigned group_lanes, Keep keep) {
    const uint32_t l = threadIdx.x & (G - 1);
    const unsigned before = (1u << (threadIdx.x & 31u)) - 1u;
    uint32_t n = 0;
    for (uint32_t i = 0; i < P; i += G) {  // an entry moves to a place at or before its own: behind what is still to be read
        const uint32_t e = i + l;
        const bool k = e < P && keep(e);
        uint32_t s = 0, t = 0, r = 0, d = 0;
        if (k) {
            s = S.start[e];
            t = S.key[e];
            r = S.row[e];
            d = S.end[e];
        }
        __syncwarp();
        const unsigned kept = __ballot_sync(0xFFFFFFFFu, k) & group_lanes;
        if (k) {
            const uint32_t to = n + __popc(kept & before);
            S.start[to] = s;
            S.key[to] = t;
            S.row[to] = r;
            S.end[to] = d;
        }
        n += __popc(kept);
        __syncwarp();
    }
    for (uint32_t e = l; e < P; e += G)
        if (e >= n) {
            S.start[e] = S.end[e] = 0;
            S.key[e] = S.row[e] = 0xFFFFFFFFu;
        }
    __syncwarp();
    return n;
}

// The result of a read from its cnt recorded targets with at most F differences:
// intervals, merged hits, strata, order.  Warp-wide, a group each; true if
// written (write, and no more hits than the tree search keeps).  By sorting: a
// read in a repeat has hundreds of targets, and comparing each with each kept one
// warp busy for milliseconds after the others had gone.
template <int G, int E, bool SCORE>
__device__ __noinline__ bool reduce_targets(const DIndex &X, const SearchParams &p, SeedRead<E> &S, uint32_t r,
                                            uint32_t cnt, uint32_t F, bool write, unsigned group_lanes,
                                            aln_read_result *res, aln_hit *hits) {
    constexpr uint32_t kNone = 0xFFFFFFFFu, kTarget = 0x8000FFFFu;  // a key's strand and length
    const uint32_t l = threadIdx.x & (G - 1), n = X.t[0].n;
    const uint32_t most = __reduce_max_sync(0xFFFFFFFFu, cnt);
    uint32_t P = 2;
    while (P < most) P <<= 1;
    // targets above the final budget leave; rows of the others
    for (uint32_t e = l; e < P; e += G) {
        uint32_t key = kNone, row = kNone;
        if (e < cnt && key_diffs(S.key[e]) <= F) {
            key = S.key[e];
            const uint32_t a = S.start[e];
            row = (key >> 31) ? row_of(X, 0, a) : row_of(X, 1, n - a - (key & 0xFFFFu));
        }
        S.key[e] = key;
        S.row[e] = row;
        S.end[e] = 0;
    }
    __syncwarp();
    // each target once, with its least witness (a part may have seen another place
    // for the gap than the best one)
    sort_targets<G, E>(S, P, [&](uint32_t i, uint32_t j) {
        const uint32_t a = S.key[i] & kTarget, b = S.key[j] & kTarget;
        if (a != b) return a < b;
        return S.row[i] != S.row[j] ? S.row[i] < S.row[j] : S.key[i] < S.key[j];
    });
    uint32_t have = pack_targets<G, E>(S, P, group_lanes, [&](uint32_t e) {
        return S.row[e] != kNone &&
               (e == 0 || S.row[e - 1] != S.row[e] || ((S.key[e - 1] ^ S.key[e]) & kTarget) != 0);
    });
    // equal targets of several places lie in neighbouring rows: the first of a run
    // stands for it
    for (uint32_t e = l; e < have; e += G) {
        const uint32_t key = S.key[e];
        const bool joins = e > 0 && S.row[e - 1] + 1u == S.row[e] && S.key[e - 1] == key &&
                           same_text(X.text, S.start[e - 1], S.start[e], key & 0xFFFFu);
        S.end[e] = joins ? 1u : 0u;
    }
    __syncwarp();
    for (uint32_t e = l; e < have; e += G)
        if (!S.end[e]) {
            uint32_t end = S.row[e] + 1u;
            for (uint32_t j = e + 1; j < have && S.end[j]; j++) end++;
            S.start[e] = end;  // the target's start is not needed any more
        }
    __syncwarp();
    for (uint32_t e = l; e < have; e += G) S.end[e] = S.end[e] ? 0u : S.start[e];
    __syncwarp();
    have = pack_targets<G, E>(S, P, group_lanes, [&](uint32_t e) { return S.end[e] != 0u; });
    // hits of equal rows on a strand (targets of several lengths) keep the least (score, witness)
    sort_targets<G, E>(S, P, [&](uint32_t i, uint32_t j) {
        const uint32_t a = S.key[i] >> 31, b = S.key[j] >> 31;
        if (a != b) return a < b;
        if (S.row[i] != S.row[j]) return S.row[i] < S.row[j];
        if (S.end[i] != S.end[j]) return S.end[i] < S.end[j];
        if (SCORE && key_score(p, S.key[i]) != key_score(p, S.key[j])) return key_score(p, S.key[i]) < key_score(p, S.key[j]);
        return S.key[i] < S.key[j];
    });
    have = pack_targets<G, E>(S, P, group_lanes, [&](uint32_t e) {
        return S.row[e] != kNone && (e == 0 || S.row[e - 1] != S.row[e] || S.end[e - 1] != S.end[e] ||
                                     ((S.key[e - 1] ^ S.key[e]) >> 31) != 0);
    });
    write = write && have <= static_cast<uint32_t>(kCandCap);  // more than that the tree search flags
    // the order (diffs or score, strand, k, l)
    auto value = [&](uint32_t e) { return SCORE ? key_score(p, S.key[e]) : key_diffs(S.key[e]); };
    sort_targets<G, E>(S, P, [&](uint32_t i, uint32_t j) {
        const bool in = S.row[i] != kNone, jn = S.row[j] != kNone;
        if (!in || !jn) return in && !jn;
        const uint32_t a = (value(i) << 1) | (S.key[i] >> 31), b = (value(j) << 1) | (S.key[j] >> 31);
        if (a != b) return a < b;
        return S.row[i] != S.row[j] ? S.row[i] < S.row[j] : S.end[i] < S.end[j];
    });
    uint32_t s1 = have ? value(0) : kNone, s2 = kNone, best = 255, c0 = 0, c1 = 0, n1 = 0, n2 = 0;
    if (SCORE) {
        for (uint32_t e = l; e < have; e += G)
            if (value(e) > s1) s2 = min(s2, value(e));
        s2 = group_min<G>(s2);
    } else {
        s2 = s1 + 1u;
    }
    for (uint32_t e = l; e < have; e += G) {
        const uint32_t v = value(e), w = S.end[e] - S.row[e];
        if (v == s1) {
            c0 += w;
            n1++;
            best = min(best, key_diffs(S.key[e]));
        } else if (v == s2) {
            c1 += w;
            n2++;
        }
    }
    best = group_min<G>(best);
    c0 = group_sum<G>(c0);
    c1 = group_sum<G>(c1);
    n1 = group_sum<G>(n1);
    n2 = group_sum<G>(n2);
    const bool many = SCORE && p.max_best && c0 > p.max_best;
    const uint32_t listed = SCORE ? n1 + (many ? 0u : n2) : have;
    if (write)
        for (uint32_t e = l; e < min(listed, p.hit_cap); e += G)
            put_hit(hits + static_cast<uint64_t>(r) * p.hit_cap + e, S.row[e], S.end[e] - 1u, S.key[e]);
    if (write && l == 0) {
        aln_read_result out;
        const bool any = listed > 0;
        const uint32_t flags = (many ? ALN_FLAG_MANY_BEST : 0u) | (listed > p.hit_cap ? ALN_FLAG_HIT_OVERFLOW : 0u);
        out.c0 = any ? c0 : 0u;
        out.c1 = any ? c1 : 0u;
        out.n_hits = static_cast<uint8_t>(min(listed, p.hit_cap));
        out.d_best = static_cast<uint8_t>(any ? best : 255u);
        out.best_score = static_cast<uint8_t>(SCORE ? (any ? min(s1, 254u) : 255u) : 0u);
        out.flags = static_cast<uint8_t>(flags);
        res[r] = out;
    }
    return write;
}

// What became of a read: its result is written; it has too many places or targets
// for this group (nothing is written then); or more places than a group of a whole
// warp takes, so that only the tree search is left.  Told apart, reads of the
// third kind save the wide kernel's try: 400 000 reads of 60 bases out of 30 000 copies
// take 33.4 ms, not 37.9 (the tree search alone 30.2), 100 000 of one letter 4.18, not
// 5.09 (4.18).
enum SeedAnswer : uint32_t { kSeedDone, kSeedWide, kSeedTree };

// The most places a read's search looks at.  16384 are half a millisecond of a warp,
// about what the tree search of such a read costs.
constexpr uint32_t kWidePlaces = 16384;

// Search of one read by the G lanes of a group; all 32 lanes of the warp call it
// together (other groups with their own reads, or with active = false).  The
// gapped stage is in line: 1 M reads take 3.41 ms with it in a function of its own and
// 3.00 without, 100 000 in the plain form 0.457 and 0.419.
template <int G, int E, bool SCORE>
__device__ SeedAnswer seed_search(const DIndex &X, const ReadBatch &rb, const SearchParams &p, SeedRead<E> &S, uint32_t r,
                            bool active, uint32_t max_places, aln_read_result *res, aln_hit *hits) {
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr uint32_t kHalf = G / 2;
    const uint32_t l = threadIdx.x & (G - 1);
    const uint32_t n = X.t[0].n;
    int m = 0;
    uint32_t z = 0;
    bool answer = false;  // a read that is not searched: its (empty) result is known
    uint32_t flags = 0;
    if (active) {
        m = rb.len[r];
        z = rb.z ? rb.z[r] : p.z;
        if (m > ALN_MAX_READ_LEN) flags |= ALN_FLAG_READ_TOO_LONG;
        if (z > ALN_MAX_Z || z > p.z) flags |= ALN_FLAG_BAD_LIMIT;
        answer = flags || m == 0;
        if (answer) m = 0;
    }
    const bool search = active && !answer;
    // ---- the read into shared memory: packed, and as planes of both strands
    __syncwarp();
    if (search) {
        const uint64_t off = rb.offset[r], last = (off + m - 1) >> 4;
        for (uint32_t w = l; w < 18; w += G) {
            uint32_t v = 0;
            if (16 * w < static_cast<uint32_t>(m)) {
                const uint64_t at = (off >> 4) + w;
                const uint32_t a = __ldg(rb.bases + at), b = at + 1 <= last ? __ldg(rb.bases + at + 1) : 0u;
                v = __funnelshift_r(a, b, 2 * static_cast<uint32_t>(off & 15u));
            }
            S.bases[w] = v;
        }
        const uint64_t nlast = (off + m - 1) >> 5;
        for (uint32_t w = l; w < kPlaneWords; w += G) {
            uint32_t v = 0;
            if (rb.nmask && 32 * w < static_cast<uint32_t>(m)) {
                const uint64_t at = (off >> 5) + w;
                const uint32_t a = __ldg(rb.nmask + at), b = at + 1 <= nlast ? __ldg(rb.nmask + at + 1) : 0u;
                v = __funnelshift_r(a, b, static_cast<uint32_t>(off & 31u));
            }
            S.pat[0].nn[w] = v & low_mask(m - static_cast<int>(32 * w));
        }
        if (l == 0) S.count = 0;
    }
    __syncwarp();
    if (search)
        for (uint32_t w = l; w < kPlaneWords; w += G) {
            const uint32_t a = S.bases[2 * w], b = S.bases[2 * w + 1];
            S.pat[0].lo[w] = even_bits(a) | (even_bits(b) << 16);
            S.pat[0].hi[w] = even_bits(a >> 1) | (even_bits(b >> 1) << 16);
        }
    __syncwarp();
    if (search)
        for (uint32_t w = l; w < kPlaneWords; w += G) {
            // pattern index 32 w + i of the reverse strand is read index m - 1 - 32 w - i:
            // read bits [m - 32 - 32 w, m - 32 w), in reverse
            const int at = m - 32 - 32 * static_cast<int>(w);
            const int q = at >> 5;
            const uint32_t s = static_cast<uint32_t>(at & 31);
            uint32_t v[3];
#pragma unroll
            for (int t = 0; t < 3; t++) {
                const uint32_t *src = t == 0 ? S.pat[0].lo : (t == 1 ? S.pat[0].hi : S.pat[0].nn);
                const uint32_t x0 = q >= 0 && q < kPlaneWords ? src[q] : 0u;
                const uint32_t x1 = q + 1 >= 0 && q + 1 < kPlaneWords ? src[q + 1] : 0u;
                v[t] = __brev(__funnelshift_r(x0, x1, s));
            }
            S.pat[1].lo[w] = ~v[0];
            S.pat[1].hi[w] = ~v[1];
            S.pat[1].nn[w] = v[2];
        }
    __syncwarp();

    const uint32_t strand = l / kHalf, part = l % kHalf;
    const uint32_t K = X.lo_k;
    const bool exhaustive = p.strata != ALN_STRATA_BEST1;
    const unsigned group_lanes = (G == 32 ? FULL : ((1u << (G & 31)) - 1u)) << ((threadIdx.x & 31u) / G * G);
    auto zone = [&](uint32_t s) {
        const int len = min(m, static_cast<int>(p.seed_len));
        return SeedZone{s ? m - len : 0, s ? m : len, p.seed_z, s != 0};
    };
    // ---- passes: every target within b differences.  b = z at once where the parts
    // are long enough to be rare; else, or where they still turn out to have many
    // places (a repeat), few long parts first: what they find bounds the
    // differences that the next pass has to look for.
    uint32_t b = z;
    bool stepping = exhaustive;  // b is 1, 3, 7 or what the targets found allow (or, of an exhaustive search, z)
    if (!exhaustive && static_cast<uint32_t>(m) < (z + 1) * K) {
        const uint32_t fit = static_cast<uint32_t>(m) / K;
        b = min(z, fit > 2 ? fit - 1 : 1u);
    }
    uint32_t F = z;            // differences a target may still have
    uint32_t dmin = 255;       // fewest found
    bool todo = search;
    SeedAnswer failed = kSeedDone;
    while (__any_sync(FULL, todo)) {
        // the rows of this lane's part
        uint32_t lo = 0, hi = 0, width = 0, ps = 0, pe = 0, off = 0;  // part [ps, pe) and first matched base, in pattern order
        uint32_t next = 0, bases = 0;                                 // read index of the next base outside, bases left
        if (todo && part <= b) {
            const uint32_t s0 = static_cast<uint32_t>(m) * part / (b + 1);
            const uint32_t s1 = static_cast<uint32_t>(m) * (part + 1) / (b + 1);
            ps = strand ? m - s1 : s0;
            pe = strand ? m - s0 : s1;
            bool clean = true;
            for (uint32_t w = s0 >> 5; 32 * w < s1; w++)
                clean = clean && !(S.pat[0].nn[w] & span_mask(static_cast<int>(s0), static_cast<int>(s1), static_cast<int>(w)));
            if (s1 == s0) {
                width = kWideRows;
            } else if (clean) {
                const uint32_t kk = min(K, s1 - s0);
                uint64_t id;  // the part's last kk bases in text order, first base highest
                if (strand) id = ~bases_at(S.bases, s0, kk) & low_mask(static_cast<int>(2 * kk));
                else id = reverse_bases(bases_at(S.bases, s1 - kk, kk), kk);
                const uint32_t sh = 2 * (K - kk);
                hi = __ldg(X.lo + ((id + 1) << sh));
                lo = __ldg(X.lo + (id << sh));
                // a shorter string's rows also hold the suffixes that end within K
                // bases, which sort below its first K-mer: at most one per length
                lo -= min(lo, K - kk);
                off = pe - kk;
                width = hi > lo ? min(hi - lo, kWideRows) : 0u;
                bases = s1 - s0 - kk;
                next = strand ? s0 + kk : s1 - 1 - kk;
            }
        }
        // Parts with several rows grow towards their first base while the group has
        // more places than two rounds look at: a base costs about a third of a
        // round, and leaves the copies of a repeat that differ there.
        for (int step = 0; step < kExtend; step++) {
            const uint32_t places = group_sum<G>(width);
            const bool go = todo && bases && width > 2 && places > 2 * G;
            if (!__any_sync(FULL, go)) break;
            if (go) {
                const uint32_t c = ((S.bases[next >> 4] >> (2 * (next & 15u))) & 3u) ^ (strand ? 3u : 0u);
                lo = lf_base(X.t[0], c, lo);
                hi = lf_base(X.t[0], c, hi);
                width = hi > lo ? min(hi - lo, kWideRows) : 0u;
                next += strand ? 1u : ~0u;
                off--;
                bases--;
            }
        }
        // places of the group, shared out in order
        uint32_t before = width;
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            const uint32_t u = __shfl_up_sync(FULL, before, o, G);
            if (l >= static_cast<uint32_t>(o)) before += u;
        }
        uint32_t total = __shfl_sync(FULL, before, G - 1, G);
        before -= width;
        const bool again = todo && !stepping && b > 1 && total > kManyPlaces * G;
        if (again) {
            stepping = true;
            total = 0;
        } else if (todo && total > max_places) {
            failed = total > kWidePlaces ? kSeedTree : kSeedWide;
            todo = false;
        }
        const uint32_t span = ps | (pe << 8) | (off << 16);
        // A group that has found more targets than it keeps is done: of a family of
        // thousands of similar copies it would look at every place for nothing (50 000
        // reads of 20 bases out of 5000 copies 1 % apart: the wide kernel 247 ms, now 10;
        // 20 000 of 36 bases at z = 3: 223 ms, now 30).
        for (uint32_t c0 = 0; __any_sync(FULL, todo && c0 < total && S.count <= static_cast<uint32_t>(E)); c0 += G) {
            const uint32_t c = c0 + l, found = S.count, have = min(found, static_cast<uint32_t>(E));
            __syncwarp();  // before lanes record targets
            uint32_t o = 0;  // the lane whose part has place c: the last one that starts at or before it
#pragma unroll
            for (int step = G / 2; step; step >>= 1) {
                const uint32_t u = __shfl_sync(FULL, before, static_cast<int>(o) + step, G);
                if (u <= c) o += step;
            }
            const uint32_t orow = __shfl_sync(FULL, lo, static_cast<int>(o), G) +
                                  (c - __shfl_sync(FULL, before, static_cast<int>(o), G));
            const uint32_t ospan = __shfl_sync(FULL, span, static_cast<int>(o), G);
            const uint32_t cs = o / kHalf;
            const int qs = static_cast<int>(ospan & 0xFFu), qe = static_cast<int>((ospan >> 8) & 0xFFu);
            bool live = todo && c < total && found <= static_cast<uint32_t>(E);
            long long d = 0;  // the diagonal: text position of pattern index 0
            if (live) {
                d = static_cast<long long>(__ldg(X.sa[0] + orow)) - static_cast<int>(ospan >> 16);
                live = d >= -static_cast<int>(z) && d + m <= static_cast<long long>(n) + static_cast<int>(z);
            }
            const Pattern &P = S.pat[cs];
            uint32_t mis[kPlaneWords];
            uint32_t mm = 255;
            if (live) {
                mismatches(X.text, P, d, m, mis);
                live = count_in(mis, qs, qe) == 0;  // else another part leads to what this diagonal has
            }
            if (live && d >= 0 && d + m <= static_cast<long long>(n)) {
                mm = 0;
#pragma unroll
                for (int w = 0; w < kPlaneWords; w++) mm += __popc(mis[w]);
                if (p.seed_len && mm <= z) {
                    const SeedZone Z = zone(cs);
                    if (count_in(mis, Z.from, Z.to) > Z.most) mm = 255;
                }
            }
            dmin = min(dmin, group_min<G>(mm));
            if (!exhaustive) F = min(z, dmin + 1);
            // gapless targets, one diagonal after the other (several parts lead to a
            // read's own place in one round): the group looks whether it has it already
            for (unsigned left = __ballot_sync(FULL, live && mm <= F) & group_lanes; __any_sync(FULL, left != 0);) {
                const int src = left ? __ffs(left) - 1 : static_cast<int>(threadIdx.x & 31u);
                const long long dd = __shfl_sync(FULL, d, src);
                const uint32_t ds = __shfl_sync(FULL, cs, src), dm = __shfl_sync(FULL, mm, src);
                const bool same = dd == d && ds == cs;
                const uint32_t key = target_key(ds, static_cast<uint32_t>(m), dm, 0u);
                bool known = false;
                for (uint32_t j = l; left && j < have; j += G)
                    known = known || (S.start[j] == static_cast<uint32_t>(dd) && S.key[j] == key);
                known = (__ballot_sync(FULL, known) & group_lanes) != 0;
                if (left && !known && src == static_cast<int>(threadIdx.x & 31u))
                    add_target(S, 0u, static_cast<uint32_t>(dd), key);
                left &= ~__ballot_sync(FULL, same);
            }
            // gapped targets: a diagonal that a gap may lead to or from is looked at by
            // the whole group, for all the parts that lead to it here
            const uint32_t gmost = p.max_gapo ? min(F, p.max_gape + 1u) : 0u;
            bool want = false;
            if (live && gmost) {
                const int f = static_cast<int>(F), gm = static_cast<int>(gmost), e = static_cast<int>(p.e);
                want = (count_in(mis, 0, qs) < F && gap_fits(X.text, P, d, m, mis, f, gm, e, false)) ||
                       (count_in(mis, qe, m) < F && gap_fits(X.text, P, d, m, mis, f, gm, e, true));
            }
            uint32_t dgap = 255;
            for (unsigned left = __ballot_sync(FULL, want) & group_lanes; __any_sync(FULL, left != 0);) {
                const int src = left ? __ffs(left) - 1 : static_cast<int>(threadIdx.x & 31u);
                const long long dd = __shfl_sync(FULL, d, src);
                const uint32_t ds = __shfl_sync(FULL, cs, src);
                const bool same = want && dd == d && ds == cs;
                const int fe = static_cast<int>(group_min<G>(same ? static_cast<uint32_t>(qe) : 255u));
                const int ls = 255 - static_cast<int>(group_min<G>(same ? 255u - static_cast<uint32_t>(qs) : 255u));
                if (left) {
                    const int e = static_cast<int>(p.e);
                    dgap = min(dgap, gap_targets<G, E>(X.text, n, S, have, m, dd, fe, ls, F, gmost, e, zone(ds)));
                }
                left &= ~__ballot_sync(FULL, same);
            }
            dmin = min(dmin, group_min<G>(dgap));
            if (!exhaustive) F = min(z, dmin + 1);
            __syncwarp();
        }
        if (todo) {
            if (S.count > static_cast<uint32_t>(E)) {
                failed = kSeedWide;
                todo = false;
            } else if (again) {
                b = 1;
            } else if (exhaustive || F <= b) {  // F = z while nothing is found
                todo = false;
            } else {
                b = stepping ? min(F, 2 * b + 1) : F;  // 1, 2, 3, ... takes 300 000 mates on 3.1 Gbp 5.78 ms, this 5.33
            }
        }
    }

    // ---- reduction of the targets: intervals, merged hits, strata, order
    const uint32_t cnt = search && !failed ? min(S.count, static_cast<uint32_t>(E)) : 0u;
    if (__all_sync(FULL, cnt <= 1u)) {  // the usual read: one target (its group's lanes 0), or none
        if (l == 0 && search && !failed) {
            const uint32_t key = cnt ? S.key[0] : 0u, a = S.start[0];
            const bool any = cnt && key_diffs(key) <= F;
            aln_read_result out;
            out.c0 = any ? 1u : 0u;
            out.c1 = 0;
            out.n_hits = any ? 1 : 0;
            out.flags = 0;
            out.d_best = static_cast<uint8_t>(any ? key_diffs(key) : 255u);
            out.best_score = static_cast<uint8_t>(SCORE ? (any ? min(key_score(p, key), 254u) : 255u) : 0u);
            if (any) {
                const uint32_t row = (key >> 31) ? row_of(X, 0, a) : row_of(X, 1, n - a - (key & 0xFFFFu));
                put_hit(hits + static_cast<uint64_t>(r) * p.hit_cap, row, row, key);
            }
            res[r] = out;
        } else if (l == 0 && answer) {
            empty_result<SCORE>(res + r, flags);
        }
        return failed;
    }
    const bool written = reduce_targets<G, E, SCORE>(X, p, S, r, cnt, F, search && !failed, group_lanes, res, hits);
    if (answer && l == 0) empty_result<SCORE>(res + r, flags);
    return failed ? failed : (search && !written ? kSeedWide : kSeedDone);
}

}  // namespace aln
