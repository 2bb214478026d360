// srht.cu -- projection of maps onto the surrogate's subsampled randomized
// Hadamard basis as a fast transform.
//
// The basis row r = a M + k of H_12 (x) H_M (M = Nside^2) gives, for a map x
// with signs s,
//   c_r = sum_b H_12[a][b] sum_t (-1)^popc(k & t) s_p x_p,  p = b M + t,
// that is a combination of the 12 base-pixel blocks followed by a
// Walsh-Hadamard transform of length M (Ailon & Chazelle 2006), of which only
// the seeded rows are kept.  Nothing of the n_basis x 12 Nside^2 matrix is
// formed or read.
//
// One CTA transforms G of the 12 combinations of one map in shared memory
// (4 G M bytes): the threads read the 12 blocks with 16-byte loads, form the
// G combinations and the two lowest bits of the transform in registers, and
// the other bits follow in one or two passes of up to 32 values per thread.
// Above M = 4096 the top bits (J = M / 4096) are summed on the way in, one CTA
// per (map, combinations, top index j), at the price of reading the map J
// times from L2.
//
// 384 maps of Nside 64 onto 3072 rows: 48.8 us (1.6 TB/s of the 80 MB it cannot
// do without) against 559 us as two BF16 GEMMs of the maps' hi + lo halves with
// the dense +-1 matrix; the coefficients' error falls from 1.2e-5 to 1.2e-7.
// Bound: the bytes of the maps (12 Nside^2 x 4 per map) from HBM.  A CTA with
// G < 12 reads its whole map, so the 12 / G CTAs of a map read it again from
// L2; fewer combinations per CTA give more CTAs for few maps.
#include <cuda_runtime.h>

#include <vector>

#include "srht.cuh"
#include "synax_internal.h"

namespace synax {
namespace {

constexpr int kSrhtThreads = 256;
constexpr int kMaxLg = 12;                 // transform length of a CTA, at most 4096

__constant__ float c_h12f[144];            // Paley's H_12, row a, column b

// Shared-memory place of element i: a 4-float gap every 128, so that both
// register passes (strides 4 and 2^(2 + P1)) touch 32 different banks.
__device__ __forceinline__ int padded(int i) { return i + ((i >> 7) << 2); }

template <int N>
__device__ __forceinline__ void wht_regs(float* v) {
#pragma unroll
    for (int h = 1; h < N; h <<= 1)
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (!(i & h)) {
                const float a = v[i], b = v[i + h];
                v[i] = a + b;
                v[i + h] = a - b;
            }
}

// Bits [B0, B0 + P) of G transforms of length 2^LG (blocks of `pitch` floats).
template <int LG, int G, int B0, int P>
__device__ __forceinline__ void wht_pass(float* sm, int pitch) {
    constexpr int N = 1 << P;
    constexpr int TASKS = G << (LG - P);
    for (int q = threadIdx.x; q < TASKS; q += kSrhtThreads) {
        const int g = q >> (LG - P), r = q & ((1 << (LG - P)) - 1);
        const int base = (r & ((1 << B0) - 1)) | ((r >> B0) << (B0 + P));
        float* p = sm + g * pitch;
        float v[N];
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = p[padded(base + (i << B0))];
        wht_regs<N>(v);
#pragma unroll
        for (int i = 0; i < N; ++i) p[padded(base + (i << B0))] = v[i];
    }
}

template <int LG>
constexpr int srht_pitch() {
    return (1 << LG) + ((1 << LG) >> 7) * 4;
}

// rows: basis row indexes r; signs: one bit per pixel (1 = negative).
template <int LG, int G>
__global__ void __launch_bounds__(kSrhtThreads)
k_srht(const float* __restrict__ maps, int lgM, const uint32_t* __restrict__ signs, const int* __restrict__ rows,
       int n_basis, float scale, int vec, float* __restrict__ out) {
    extern __shared__ float sm[];
    constexpr int PITCH = srht_pitch<LG>();
    constexpr int m = 1 << LG;
    constexpr int GROUPS = 12 / G;
    const int J = 1 << (lgM - LG);
    const int j = blockIdx.x % J;
    const int a0 = (blockIdx.x / J) % GROUPS * G;
    const long long map = blockIdx.x / (J * GROUPS);
    const int M = 1 << lgM;
    const float* x = maps + map * 12 * M;

    for (int t = 4 * threadIdx.x; t < m; t += 4 * kSrhtThreads) {
        float acc[G][4];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[g][e] = 0.0f;
        for (int q = 0; q < J; ++q) {
            const uint32_t top = (uint32_t)(__popc(q & j) & 1) * 15u;
            float4 v[12];
            uint32_t w[12];
#pragma unroll
            for (int b = 0; b < 12; ++b) {
                const int p = b * M + q * m + t;
                w[b] = __ldg(signs + (p >> 5));
                if (vec) {
                    v[b] = __ldg(reinterpret_cast<const float4*>(x + p));
                } else {
                    v[b] = make_float4(__ldg(x + p), __ldg(x + p + 1), __ldg(x + p + 2), __ldg(x + p + 3));
                }
            }
#pragma unroll
            for (int b = 0; b < 12; ++b) {
                const int p = b * M + q * m + t;
                const uint32_t s = (w[b] >> (p & 31)) ^ top;       // bits 0..3: the signs of the four pixels
                const float u[4] = {__uint_as_float(__float_as_uint(v[b].x) ^ (s << 31)),
                                    __uint_as_float(__float_as_uint(v[b].y) ^ ((s & 2u) << 30)),
                                    __uint_as_float(__float_as_uint(v[b].z) ^ ((s & 4u) << 29)),
                                    __uint_as_float(__float_as_uint(v[b].w) ^ ((s & 8u) << 28))};
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const float h = c_h12f[(a0 + g) * 12 + b];
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[g][e] = fmaf(h, u[e], acc[g][e]);
                }
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            wht_regs<4>(acc[g]);
            *reinterpret_cast<float4*>(sm + g * PITCH + padded(t)) =
                make_float4(acc[g][0], acc[g][1], acc[g][2], acc[g][3]);
        }
    }
    __syncthreads();
    constexpr int REST = LG - 2;
    constexpr int P1 = REST > 5 ? REST / 2 : REST;
    wht_pass<LG, G, 2, P1>(sm, PITCH);
    __syncthreads();
    if constexpr (REST > P1) {
        wht_pass<LG, G, 2 + P1, REST - P1>(sm, PITCH);
        __syncthreads();
    }
    float* o = out + map * n_basis;
    for (int i = threadIdx.x; i < n_basis; i += kSrhtThreads) {
        const int r = __ldg(rows + i);
        const int a = (r >> lgM) - a0, k = r & (M - 1);
        if (a >= 0 && a < G && (k >> LG) == j) o[i] = scale * sm[a * PITCH + padded(k & (m - 1))];
    }
}

template <int LG, int G>
cudaError_t attr() {
    return cudaFuncSetAttribute(k_srht<LG, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(G * srht_pitch<LG>() * sizeof(float)));
}

template <int LG, int G>
int launch(const SrhtBasis& B, const float* maps, long long n, float* out, cudaStream_t st) {
    const int per = (12 / G) << (B.lgM - LG);
    const int vec = ((uintptr_t)maps & 15) == 0;
    const size_t npix = (size_t)12 << B.lgM;
    const long long cap = (1LL << 30) / per;
    for (long long r0 = 0; r0 < n; r0 += cap) {
        const long long rows = n - r0 < cap ? n - r0 : cap;
        k_srht<LG, G><<<(unsigned)(rows * per), kSrhtThreads, G * srht_pitch<LG>() * sizeof(float), st>>>(
            maps + r0 * npix, B.lgM, B.signs, B.rows, B.n_basis, B.scale, vec, out + r0 * B.n_basis);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return record_cuda_error((int)e);
    }
    return SYNAX_OK;
}

// Combinations per CTA: 6 once that still gives two CTAs for every SM, 3
// for half as many maps, otherwise one, so that a single I/Q/U map spreads
// over 36 CTAs.
template <int LG>
int launch_lg(const SrhtBasis& B, const float* maps, long long n, float* out, cudaStream_t st) {
    const long long work = n << (B.lgM - LG);
    if (work >= 152) return launch<LG, 6>(B, maps, n, out, st);
    if (work >= 76) return launch<LG, 3>(B, maps, n, out, st);
    return launch<LG, 1>(B, maps, n, out, st);
}

}  // namespace

int srht_init(const int8_t* h12) {
    float h[144];
    for (int i = 0; i < 144; ++i) h[i] = (float)h12[i];
    cudaError_t e = cudaMemcpyToSymbol(c_h12f, h, sizeof h);
    if (e == cudaSuccess) e = attr<12, 6>();
    if (e == cudaSuccess) e = attr<12, 3>();
    return e == cudaSuccess ? SYNAX_OK : record_cuda_error((int)e);
}

void srht_pack_signs(const int8_t* sign, int npix, std::vector<uint32_t>& words) {
    words.assign((size_t)(npix + 31) / 32, 0u);
    for (int p = 0; p < npix; ++p)
        if (sign[p] < 0) words[p >> 5] |= 1u << (p & 31);
}

int srht_project(const SrhtBasis& B, const float* maps, long long n, float* out, cudaStream_t st) {
    if (n <= 0) return SYNAX_OK;
    switch (B.lgM < kMaxLg ? B.lgM : kMaxLg) {
    case 4: return launch_lg<4>(B, maps, n, out, st);
    case 6: return launch_lg<6>(B, maps, n, out, st);
    case 8: return launch_lg<8>(B, maps, n, out, st);
    case 10: return launch_lg<10>(B, maps, n, out, st);
    case 12: return launch_lg<12>(B, maps, n, out, st);
    default: return SYNAX_EINVAL;
    }
}

}  // namespace synax
