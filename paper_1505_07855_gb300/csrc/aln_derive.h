// Arrays derived on the device from an uploaded index (aln_derive.cu).
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace aln {

struct DIndex;

constexpr uint64_t derived_align(uint64_t bytes) { return (bytes + 255u) & ~255ull; }

uint64_t derived_bytes(uint64_t n);
cudaError_t derive(DIndex &X, void *mem, cudaStream_t st, bool *ok);

}  // namespace aln
