// srht.cuh -- interface of the fast projection onto the subsampled
// randomized Hadamard basis (srht.cu).
#pragma once

#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

namespace synax {

struct SrhtBasis {
    int lgM;                   // log2 Nside^2
    int n_basis;
    float scale;               // 1 / sqrt(12 Nside^2)
    const uint32_t* signs;     // device, one bit per pixel (1: the sign is -1)
    const int* rows;           // device, n_basis row indexes of H_12 (x) H_M
};

// Uploads H_12 (144 entries of +1 / -1, row major) and opts the kernels into
// their shared memory; call once per device before srht_project.
int srht_init(const int8_t* h12);

// The signs of npix pixels as one bit each.
void srht_pack_signs(const int8_t* sign, int npix, std::vector<uint32_t>& words);

// out[n][n_basis] = coefficients of maps [n][12 Nside^2] (device), enqueued on st.
int srht_project(const SrhtBasis& B, const float* maps, long long n, float* out, cudaStream_t st);

}  // namespace synax
