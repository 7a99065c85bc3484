// Arrays derived on the device from an uploaded index (aln_derive.cu).
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace aln {

struct DIndex;

#ifndef ALN_LO_STRINGS
#define ALN_LO_STRINGS 4
#endif
// Strings in the k-mer table per suffix, at most: with 4 (14-mers at 100 Mbp, 1.1
// GB) 1 M reads take 3.0 ms, with 1 (13-mers) 4.1 ms, as every part then has a
// chance place or two.
constexpr uint64_t kLoStrings = ALN_LO_STRINGS;

constexpr uint64_t derived_align(uint64_t bytes) { return (bytes + 255u) & ~255ull; }

uint64_t derived_bytes(uint64_t n);
cudaError_t derive(DIndex &X, void *mem, cudaStream_t st, bool *ok);

}  // namespace aln
