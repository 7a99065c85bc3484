// Arrays derived on the device from the uploaded index: the whole suffix array
// of both texts (the index keeps every sa_sample-th row), its inverse at every
// kIsaStep-th text position, the text X as bit planes, and for every string of
// lo_k bases the number of suffixes of X below it.  They follow from the image
// alone, so a search or a position look-up gives the same numbers with or without
// them; an index whose arrays would not fit comfortably is served from the image.
//
// The first three come from LF walks: from the sampled row r, whose value is
// known, LF leads to the row of the suffix one position earlier, and shows the
// base there, until the next sampled row.  Every row lies on exactly one such
// walk, so the n + 1 rows take n LF steps in all, one thread per sampled row.  The
// rows that the walks pass are counted: an image whose LF steps form a cycle
// without a sampled row would leave rows unwritten, and is not derived from.
// The table follows from the Occ counts, one base longer a launch: the suffixes
// below c s are those that start with a lower base and those of base c whose
// rest is below s.
#include <cuda_runtime.h>

#include "aln_device.cuh"
#include "aln_derive.h"

namespace aln {
namespace {

__device__ __forceinline__ void put_bases(uint2 *text, uint32_t word, uint32_t lo, uint32_t hi) {
    if (lo) atomicOr(&text[word].x, lo);
    if (hi) atomicOr(&text[word].y, hi);
}

constexpr uint32_t kWalkError = 1u;   // a walk left the text, missed its sample or passed its bound
constexpr uint32_t kTableError = 2u;  // an Occ count led past the last row

struct Report {                       // what the kernels tell the host, cleared first
    uint32_t err, pad;
    unsigned long long rows[2];       // rows that the walks of each text passed
};

// One thread per sampled row: the walk to the next sampled row.  Bound by the
// latency of one dependent half-block read a step (and by the scattered 4-byte
// stores); one thread per walk keeps the most walks in flight.  Both texts of
// 100 Mbp and the table add 9.7 ms to the upload.
__global__ void __launch_bounds__(256) sa_fill_kernel(DText T, uint32_t shift, uint32_t limit, uint32_t n_samples,
                                                      uint32_t *sa, uint32_t *isa, uint2 *text, Report *rep,
                                                      unsigned long long *rows) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = i < n_samples;
    const uint32_t mask = (1u << shift) - 1u;
    uint32_t row = i << shift, v = live ? T.sa_samp[i] : 0u, steps = 0, last = 0;
    bool bad = !live || v > T.n;
    uint32_t lo = 0, hi = 0, word = v >> 5;  // bases of the text word the walk is in
    while (!bad) {
        sa[row] = v;
        if (v % kIsaStep == 0) isa[v / kIsaStep] = row;
        if (row == T.primary) {  // SA[primary] = 0: the walk around the text ends here
            bad = v != 0;
            last = 1;
            break;
        }
        if (v == 0 || steps >= limit) {
            bad = true;
            break;
        }
        uint32_t c;
        row = lf_row(T, row, c);
        v--;
        steps++;
        if (text) {
            if (v >> 5 != word) {
                put_bases(text, word, lo, hi);
                lo = hi = 0;
                word = v >> 5;
            }
            lo |= (c & 1u) << (v & 31u);
            hi |= (c >> 1) << (v & 31u);
        }
        if (row > T.n) {
            bad = true;
        } else if ((row & mask) == 0) {
            bad = T.sa_samp[row >> shift] != v;
            break;
        }
    }
    if (text && !bad) put_bases(text, word, lo, hi);
    if (live && bad) atomicOr(&rep->err, kWalkError);
    const uint32_t all = __reduce_add_sync(0xFFFFFFFFu, bad ? 0u : steps + last);  // rows written
    if ((threadIdx.x & 31u) == 0) atomicAdd(rows, static_cast<unsigned long long>(all));
}

// lo[c 4^j + s] = number of suffixes below the string c s, from lo[s] over the
// 4^j strings s (first base highest), in place: a thread reads entry s alone and
// writes that entry and three past the level.  The levels are enqueued together, so
// each bounds what it read before it reads an Occ block there.
__global__ void __launch_bounds__(256) lo_level_kernel(DText T, uint64_t strings, uint32_t *lo, Report *rep) {
    const uint64_t s = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (s >= strings) return;
    uint32_t at = lo[s];
    if (at > T.n + 1u) {
        atomicOr(&rep->err, kTableError);
        at = 0;
    }
    const uint32_t b = at / kRowsPerBlock, o = at - b * kRowsPerBlock;
    HalfBlock H;
    load_half(T.blocks, b, o, H);
    uint32_t occ[4];
    occ4_in_half(H, o, occ);
    occ[0] -= at > T.primary ? 1u : 0u;
#pragma unroll
    for (int c = 0; c < 4; c++) lo[c * strings + s] = T.C1[c] + occ[c];
}

}  // namespace

static uint64_t text_words(uint64_t n) { return n / 32 + 1 + 2 * kTextPad; }

// Depth of the table: the strings number at most kLoStrings times the suffixes,
// so that a random string of that length is met less than once.
static uint32_t lo_depth(uint64_t n) {
    uint32_t k = 1;
    while (k < 16 && (4ull << (2 * k)) <= kLoStrings * (n + 1)) k++;
    return k;
}

static uint64_t lo_entries(uint64_t n) { return (1ull << (2 * lo_depth(n))) + 1; }

uint64_t derived_bytes(uint64_t n) {
    return 256 + 2 * derived_align(4 * (n + 1)) + 2 * derived_align(4 * (n / kIsaStep + 1)) +
           derived_align(8 * text_words(n)) + derived_align(4 * lo_entries(n));
}

// The derived arrays of index X in mem (derived_bytes(n) bytes), on stream st;
// *ok tells whether the image was consistent (walks that met their samples
// within 64 * sa_sample steps, the bound of a position look-up, and passed every
// row; counts that stay within the rows).
cudaError_t derive(DIndex &X, void *mem, cudaStream_t st, bool *ok) {
    const uint64_t n = X.t[0].n;
    char *p = static_cast<char *>(mem);
    auto take = [&](uint64_t bytes) {
        char *at = p;
        p += derived_align(bytes);
        return at;
    };
    *ok = false;
    Report *rep = reinterpret_cast<Report *>(take(256));
    uint32_t *sa[2], *isa[2];
    for (int w = 0; w < 2; w++) sa[w] = reinterpret_cast<uint32_t *>(take(4 * (n + 1)));
    for (int w = 0; w < 2; w++) isa[w] = reinterpret_cast<uint32_t *>(take(4 * (n / kIsaStep + 1)));
    uint2 *text = reinterpret_cast<uint2 *>(take(8 * text_words(n)));
    uint32_t *lo = reinterpret_cast<uint32_t *>(take(4 * lo_entries(n)));
    cudaError_t e = cudaMemsetAsync(rep, 0, 256, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(text, 0, 8 * text_words(n), st);
    if (e != cudaSuccess) return e;
    const uint32_t n_samples = static_cast<uint32_t>(n >> X.sa_shift) + 1u;
    for (int w = 0; w < 2; w++)
        sa_fill_kernel<<<(n_samples + 255u) / 256u, 256, 0, st>>>(X.t[w], X.sa_shift, 64u << X.sa_shift, n_samples,
                                                                  sa[w], isa[w], w ? nullptr : text + kTextPad, rep,
                                                                  &rep->rows[w]);
    const uint32_t depth = lo_depth(n), end = static_cast<uint32_t>(n + 1);
    if ((e = cudaMemsetAsync(lo, 0, 4, st)) != cudaSuccess) return e;  // no suffix is below the empty string
    for (uint32_t j = 0; j < depth; j++) {
        const uint64_t strings = 1ull << (2 * j);
        lo_level_kernel<<<static_cast<unsigned>((strings + 255) / 256), 256, 0, st>>>(X.t[0], strings, lo, rep);
    }
    e = cudaMemcpyAsync(lo + lo_entries(n) - 1, &end, 4, cudaMemcpyHostToDevice, st);
    Report got{};
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&got, rep, sizeof got, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess || got.err || got.rows[0] != n + 1 || got.rows[1] != n + 1) return e;
    for (int w = 0; w < 2; w++) {
        X.sa[w] = sa[w];
        X.isa[w] = isa[w];
    }
    X.text = text + kTextPad;
    X.lo = lo;
    X.lo_k = depth;
    *ok = true;
    return cudaSuccess;
}

}  // namespace aln
