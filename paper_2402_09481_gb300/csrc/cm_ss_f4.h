// The shared-seed product on tcgen05 (cm_ss_f4.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace cm {

// Longest input: its counts, all ones included, are checked exact in the
// accumulator.
constexpr uint64_t kSsF4MaxN = 1ull << 14;
// Bytes of the expanded matrix.
uint64_t ss_f4_bytes(uint64_t n, uint64_t m);
cudaError_t launch_ss_f4_rows(const uint64_t *y, uint64_t n, uint64_t m, void *T, int nsm, cudaStream_t st);
// The same from packed rows: bit j < n of row i < m at word i * gw + j / 32 (bits
// past n are 0).
cudaError_t launch_ss_f4_pack(const uint32_t *G, uint64_t gw, uint64_t n, uint64_t m, void *T, int nsm, cudaStream_t st);
cudaError_t launch_ss_f4(const void *T, uint64_t n, uint64_t m, const uint64_t *X, uint64_t count, uint64_t *Z,
                         uint32_t *status, int nsm, cudaStream_t st);

}  // namespace cm
