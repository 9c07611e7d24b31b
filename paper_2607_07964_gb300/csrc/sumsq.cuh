// Sums of squares along rows and along columns of a row-major fp32 matrix, in a fixed
// order (deterministic): fp32 partials over short runs, fp64 across runs and lanes.
//
// Both are HBM-bound single passes. They keep many independent loads in flight per thread
// (the runs are unrolled, loads first, then the FMA chain), which a one-load-per-iteration
// loop does not: with ~1 us DRAM latency that loop ran at a tenth of the copy bandwidth.
#pragma once

#include <stdint.h>

namespace kq {

// Column sums: block (CS_X, CS_Y); column j = blockIdx.x * CS_X + threadIdx.x; thread row y
// reads the CS_U-row runs starting at y * CS_U, stepping CS_Y * CS_U rows, the next run's loads in
// flight over the sums of the one before. Bound: HBM (3.6 TB/s at 14336 x 4096 from a cold L2:
// 112.6 -> 65.5 us with the loads ahead, 4096 x 4096 41.0 -> 26.6). A second thread row of loaders
// for each chain, its sums handed over through shared memory, took 69.6 and 26.6 us, and 22.5
// against 18.5 at 1024 x 8192.
// Registers (95 a thread: one CTA per SM; 64: two): one while every CTA has an SM of its own, 4096
// x 4096 18.8 us against 22.3 and 8192 x 1024 26.7 against 35.0; two beyond, where the second
// CTA fills the SM: 1024 x 8192 14.8 -> 12.4, 256 x 28672 22.6 -> 14.4 (18.5 without loads ahead,
// 56 registers), 8192 x 28672 187 -> 160 (197). Just past one CTA per SM it depends on the rows
// (scales of both sides, one and two: 256 x 4896 16.5 and 14.4, 4096 x 4896 39.0 and 43.1, 4096 x
// 7168 55.6 and 52.1, 14336 x 4896 154.9 and 148.6).
constexpr int CS_X = 32, CS_Y = 16, CS_U = 16;

inline int cs_per_sm(int64_t cols) { return cdiv(cols, CS_X) > num_sms() ? 2 : 1; }

// sum over r of M[r][j]^2; the result is valid in threadIdx.y == 0 (all threads must call).
__device__ __forceinline__ double col_sumsq(const float* __restrict__ M, int64_t rows, int64_t cols, int64_t j) {
    __shared__ double part[CS_Y][CS_X + 1];
    double acc = 0.0;
    if (j < cols) {
        const float* p0 = M + j;
        auto load = [&](int64_t r0, float (&v)[CS_U]) {
            if (r0 + CS_U <= rows) {
#pragma unroll
                for (int k = 0; k < CS_U; ++k) v[k] = __ldg(p0 + (r0 + k) * cols);
            } else {
#pragma unroll
                for (int k = 0; k < CS_U; ++k) v[k] = (r0 + k < rows) ? __ldg(p0 + (r0 + k) * cols) : 0.0f;
            }
        };
        float v[CS_U], nv[CS_U];
        int64_t r0 = static_cast<int64_t>(threadIdx.y) * CS_U;
        if (r0 < rows) load(r0, v);
        while (r0 < rows) {
            r0 += CS_Y * CS_U;
            if (r0 < rows) load(r0, nv);
            float p = 0.0f;
#pragma unroll
            for (int k = 0; k < CS_U; ++k) p = fmaf(v[k], v[k], p);
            acc += p;
#pragma unroll
            for (int k = 0; k < CS_U; ++k) v[k] = nv[k];
        }
    }
    part[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    double a = 0.0;
    if (threadIdx.y == 0)
        for (int y = 0; y < CS_Y; ++y) a += part[y][threadIdx.x];
    return a;
}

// Row sums: one warp per row. Lane l reads 4-float groups l, l + 32, ... (float4 when the
// row start is 16-byte aligned and the length a multiple of 4), RS_U groups per run.
constexpr int RS_U = 4;

// sum over j of row[j]^2, valid in every lane of the warp.
__device__ __forceinline__ double row_sumsq(const float* __restrict__ row, int64_t n) {
    const int lane = threadIdx.x & 31;
    double acc = 0.0;
    if ((n & 3) == 0 && (reinterpret_cast<uintptr_t>(row) & 15) == 0) {
        const float4* r4 = reinterpret_cast<const float4*>(row);
        const int64_t n4 = n >> 2;
        for (int64_t g0 = lane; g0 < n4; g0 += 32 * RS_U) {
            float4 v[RS_U];
#pragma unroll
            for (int u = 0; u < RS_U; ++u)
                v[u] = (g0 + 32 * u < n4) ? __ldg(r4 + g0 + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
            float p = 0.0f;
#pragma unroll
            for (int u = 0; u < RS_U; ++u) {
                p = fmaf(v[u].x, v[u].x, p);
                p = fmaf(v[u].y, v[u].y, p);
                p = fmaf(v[u].z, v[u].z, p);
                p = fmaf(v[u].w, v[u].w, p);
            }
            acc += p;
        }
    } else {
        for (int64_t j0 = lane; j0 < n; j0 += 32 * 4 * RS_U) {
            float v[4 * RS_U];
#pragma unroll
            for (int u = 0; u < 4 * RS_U; ++u) v[u] = (j0 + 32 * u < n) ? __ldg(row + j0 + 32 * u) : 0.0f;
            float p = 0.0f;
#pragma unroll
            for (int u = 0; u < 4 * RS_U; ++u) p = fmaf(v[u], v[u], p);
            acc += p;
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

}  // namespace kq
