// Arrays derived on the device from the uploaded index: the whole suffix array
// of both texts (the index keeps every sa_sample-th row).  They follow from the
// image alone, so a search or a position look-up gives the same numbers with or
// without them; an index whose arrays would not fit comfortably is served from
// the image.
//
// The suffix array comes from LF walks: from the sampled row r, whose value is
// known, LF leads to the row of the suffix one position earlier, until the next
// sampled row.  Every row lies on exactly one such walk, so the n + 1 rows take
// n LF steps in all, one thread per sampled row.
#include <cuda_runtime.h>

#include "aln_device.cuh"
#include "aln_derive.h"

namespace aln {
namespace {

constexpr uint32_t kWalkError = 1u;   // a walk left the text, missed its sample or passed its bound

// One thread per sampled row: the walk to the next sampled row.  Bound by the
// latency of one dependent half-block read a step (and by the scattered 4-byte
// stores); one thread per walk keeps the most walks in flight.  Both texts of
// 100 Mbp add about 8 ms to the upload.
__global__ void __launch_bounds__(256) sa_fill_kernel(DText T, uint32_t shift, uint32_t limit, uint32_t n_samples,
                                                      uint32_t *sa, uint32_t *err) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_samples) return;
    const uint32_t mask = (1u << shift) - 1u;
    uint32_t row = i << shift, v = T.sa_samp[i], steps = 0;
    bool bad = v > T.n;
    while (!bad) {
        sa[row] = v;
        if (row == T.primary) {  // SA[primary] = 0: the walk around the text ends here
            bad = v != 0;
            break;
        }
        if (v == 0 || steps >= limit) {
            bad = true;
            break;
        }
        row = lf_row(T, row);
        v--;
        steps++;
        if (row > T.n) {
            bad = true;
        } else if ((row & mask) == 0) {
            bad = T.sa_samp[row >> shift] != v;
            break;
        }
    }
    if (bad) atomicOr(err, kWalkError);
}

}  // namespace

uint64_t derived_bytes(uint64_t n) { return 256 + 2 * derived_align(4 * (n + 1)); }

// The derived arrays of index X in mem (derived_bytes(n) bytes), on stream st;
// *ok tells whether the image was consistent (walks that met their samples
// within 64 * sa_sample steps, the bound of a position look-up).
cudaError_t derive(DIndex &X, void *mem, cudaStream_t st, bool *ok) {
    const uint64_t n = X.t[0].n;
    char *p = static_cast<char *>(mem);
    uint32_t *err = reinterpret_cast<uint32_t *>(p);
    p += 256;
    *ok = false;
    cudaError_t e = cudaMemsetAsync(err, 0, 256, st);
    if (e != cudaSuccess) return e;
    const uint32_t n_samples = static_cast<uint32_t>(n >> X.sa_shift) + 1u;
    uint32_t *sa[2];
    for (int w = 0; w < 2; w++) {
        sa[w] = reinterpret_cast<uint32_t *>(p);
        p += derived_align(4 * (n + 1));
        sa_fill_kernel<<<(n_samples + 255u) / 256u, 256, 0, st>>>(X.t[w], X.sa_shift, 64u << X.sa_shift, n_samples,
                                                                  sa[w], err);
    }
    uint32_t bad = 1;
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bad, err, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess || bad) return e;
    X.sa[0] = sa[0];
    X.sa[1] = sa[1];
    *ok = true;
    return cudaSuccess;
}

}  // namespace aln
