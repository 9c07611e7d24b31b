// Inference with a quantized layer: y = W^ x with the incoherence processing reverted
// online (Sec. 3.2: "At inference, BiIP introduces no additional overhead beyond QuIP#";
// the reverted weight of Algorithm 2 is W^ = S_G^-1 U^T Q' V S_X^-1, Q' the dequantized
// codes). The dense W^ is never formed:
//   x' = V S_X^-1 x        fast Hadamard transform of each token (biip.cu row transform)
//   y' = Q' x'             dequantizing matrix-vector product over packed codes (this file)
//   y  = S_G^-1 U^T y'     fast Hadamard transform of each output
// so the cost is the code stream plus O(d log d) per token.
//
// Packed codes: each row of codes is stored as 32-bit words along d_in, word w holding codes
// w * (32 / pb) .. + (32 / pb) - 1, code t of the word in bits [t pb, t pb + pb); pb = bits for
// 2, 4 and 8-bit codes, and 4 for 3-bit codes (3-bit codes travel in 4-bit lanes).
//
// Three kernels: the transform of x (infer_rht_*: one CTA per token for n = 2^k, a cluster of
// seven or eight CTAs per token otherwise), the product (infer_mma_kernel: clusters of CTAs that
// split d_in, codes minus the middle code exact in bf16, x' an exact sum of three bf16 terms),
// the transform of y'. Each is launched as a programmatic dependent, so the next kernel's weights,
// scales and factors are on their way while the one before it finishes: a single-token call is
// bound by the latency of the three, not by its bytes. Per layer (24 layers of one size in a graph,
// distinct weights, 4 bits, one token): 4096 x 4096 10.3 us, 14336 x 4096 23.0, 4096 x 14336 20.7,
// 8192 x 8192 23.2; eight tokens 13.9, 31.9, 28.8, 33.2. The streaming kernel this replaces (TMA
// ring of weights, x' formed in every CTA, fp32 products) took 18.2, 42.9, 80.4, 61.3 us for one
// token and 33, 69 us for eight; where eight tokens' x' did not fit beside its ring (d_in = 8192,
// 14336), the row-per-warp fallback took 550-600 us.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "kq_common.cuh"
#include "rht.cuh"

namespace cg = cooperative_groups;

namespace kq {
namespace {

constexpr int KQ_INFER_MAX_B = 8;

inline int lane_bits(int bits) { return bits == 3 ? 4 : bits; }

// packed[r][w] = sum_t codes[r][w * cpw + t] << (t pb), one thread per word.
__global__ void pack_kernel(const uint8_t* __restrict__ codes, int64_t d_out, int64_t d_in, int pb,
                            uint32_t* __restrict__ packed) {
    const int cpw = 32 / pb;
    const int64_t wpr = d_in / cpw;
    const int64_t total = d_out * wpr;
    const uint32_t mask = (1u << pb) - 1u;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
         e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t r = e / wpr, w = e - r * wpr;
        const uint8_t* src = codes + r * d_in + w * cpw;
        uint32_t v = 0;
        for (int t = 0; t < cpw; ++t) v |= (static_cast<uint32_t>(src[t]) & mask) << (t * pb);
        packed[e] = v;
    }
}

__device__ __forceinline__ void prefetch_l2(const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(src)), "r"(bytes)
                 : "memory");
}

// 2^23 + code for the byte k of w (the bits 0x4B0000qq).
__device__ __forceinline__ float byte_raw(uint32_t w, int k) {
    return __int_as_float(static_cast<int>(__byte_perm(w, 0x4B000000u, 0x7440u | static_cast<uint32_t>(k))));
}

// ------------------------------------------------------------------- transforms of a token
// dst[b] = T (f (.) src[b]) / sqrt(n) (PRE: x' = V S_X^-1 x) or f (.) T src[b] / sqrt(n) (y =
// S_G^-1 U^T y'), T = H_n, f = sign / s, for one token b per CTA or cluster. Bound: latency (a few
// tens of KB per token). The first kernel of a call (PRE) waits for the work before it and only
// then lets the product kernel start: everything that work wrote (codes, grids, scales) is then
// there for the product's and the last transform's loads ahead of their own waits.
template <bool PRE>
__device__ __forceinline__ void rht_begin() {
    if constexpr (PRE) {
        pdl_wait();
        pdl_launch_dependents();
    }
}
template <bool PRE>
__device__ __forceinline__ void rht_wait() {
    if constexpr (!PRE) {
        pdl_launch_dependents();
        pdl_wait();
    }
}
__device__ __forceinline__ float rht_factor(const float* s, const int8_t* sign, int64_t j) {
    const float r = __frcp_rn(__ldg(s + j));
    return sign[j] < 0 ? -r : r;
}
// N of them at the places at(k): every load is issued before the first reciprocal (one at a time
// they cost a memory latency each: 12 us for 16, 28 us for 28).
template <int N, typename At>
__device__ __forceinline__ void rht_factors(const float* s, const int8_t* sign, float (&f)[N], At at) {
    int sg[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        f[k] = __ldg(s + at(k));
        sg[k] = __ldg(sign + at(k));
    }
    asm volatile("" ::: "memory");
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const float r = __frcp_rn(f[k]);
        f[k] = sg[k] < 0 ? -r : r;
    }
}

// A thread's 16 consecutive values of a token, and the same times the factors at j0 ..
// (16-byte loads, all issued before the first use).
__device__ __forceinline__ void load16(const float* src, float (&x)[16]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(src) + q);   // written by the kernel before
        x[4 * q] = v.x;
        x[4 * q + 1] = v.y;
        x[4 * q + 2] = v.z;
        x[4 * q + 3] = v.w;
    }
}
__device__ __forceinline__ void load16_scaled(const float* src, const float* s, const int8_t* sign, float (&x)[16]) {
    float4 sv[4];
    char4 sg[4];
    load16(src, x);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        sv[q] = __ldg(reinterpret_cast<const float4*>(s) + q);
        sg[q] = __ldg(reinterpret_cast<const char4*>(sign) + q);
    }
    asm volatile("" ::: "memory");
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float f[4] = {__frcp_rn(sv[q].x), __frcp_rn(sv[q].y), __frcp_rn(sv[q].z), __frcp_rn(sv[q].w)};
        const int8_t g[4] = {static_cast<int8_t>(sg[q].x), static_cast<int8_t>(sg[q].y), static_cast<int8_t>(sg[q].z),
                             static_cast<int8_t>(sg[q].w)};
#pragma unroll
        for (int u = 0; u < 4; ++u) x[4 * q + u] *= g[u] < 0 ? -f[u] : f[u];
    }
}

// One cluster of NC CTAs per token, CTA c holding the slice [c L, c L + L) of src (L = n / NC).
// With T = H_A (x) H_P (index a P + b, b fastest): for n = 2^k, NC = 8 CTAs (A = 8, P = L) or one
// CTA for n < 64; for n = 28 P, NC = 7 CTAs of four length-P pieces each (A = 28). Each CTA
// applies H_P to its pieces in shared memory; after a cluster barrier, column b of the A x P
// array is gathered from the CTAs' shared memory (distributed shared memory) and mixed by H_A.
template <int NC, bool PRE>
__global__ void __launch_bounds__(256) infer_rht_kernel(const float* __restrict__ src, int n, int lg_p,
                                                        const float* __restrict__ sc, const int8_t* __restrict__ sign,
                                                        float* __restrict__ dst) {
    extern __shared__ __align__(16) float ov[];
    constexpr int A = NC == 7 ? 28 : NC;    // rows of the A x P array
    constexpr int PER = A / NC;              // rows a CTA holds
    const int P = 1 << lg_p;
    const int L = PER * P;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = NC > 1 ? static_cast<int>(cl.block_rank()) : 0;
    const int64_t b = blockIdx.x / NC;
    rht_begin<PRE>();
    rht_wait<PRE>();
    const float* in = src + b * n + static_cast<int64_t>(rank) * L;
    for (int q = threadIdx.x; q < L; q += blockDim.x) {
        const float v = __ldcg(in + q);
        ov[q] = PRE ? v * rht_factor(sc, sign, static_cast<int64_t>(rank) * L + q) : v;
    }
    __syncthreads();
    block_rht_inplace(ov, L, lg_p, false, F_NONE, F_NONE, sign, sc, 1.0f);
    if constexpr (NC > 1) cl.sync();
    const float isn = rsqrtf(static_cast<float>(n));
    // columns [c0, c1) of this CTA
    const int per_cta = (P + NC - 1) / NC;
    const int c0 = rank * per_cta, c1 = min(P, c0 + per_cta);
    float* out = dst + b * n;
    for (int col = c0 + static_cast<int>(threadIdx.x); col < c1; col += blockDim.x) {
        float f[A], xa[A];
        if constexpr (PRE) {
#pragma unroll
            for (int a = 0; a < A; ++a) f[a] = 1.0f;
        } else {
            rht_factors(sc, sign, f, [&](int a) { return a * P + col; });
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const float* rv = NC > 1 ? cl.map_shared_rank(ov, c) : ov;
#pragma unroll
            for (int q = 0; q < PER; ++q) xa[c * PER + q] = rv[q * P + col];
        }
        auto put = [&](int a, float v) { out[static_cast<int64_t>(a) * P + col] = v * isn * f[a]; };
        if constexpr (A == 28) {
            mix28_paley(xa, put);
        } else {
            float x8[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) x8[q] = q < A ? xa[q] : 0.0f;
            if constexpr (A == 8) fwht_reg<8>(x8);
#pragma unroll
            for (int q = 0; q < A; ++q) put(q, x8[q]);
        }
    }
    if constexpr (NC > 1) cl.sync();   // keep this CTA's slice alive until every CTA has read it
}

// n = 2^LG, one CTA per token, in registers (n / 16 threads of 16 values).
template <int LG, bool PRE>
__global__ void __launch_bounds__((1 << LG) / 16) infer_rht_reg_kernel(const float* __restrict__ src, int n,
                                                                       const float* __restrict__ sc,
                                                                       const int8_t* __restrict__ sign,
                                                                       float* __restrict__ dst) {
    constexpr int NPH = rr_phases(LG);
    constexpr uint32_t ML = rr_mask(LG, NPH - 1);
    extern __shared__ __align__(16) float osm[];
    const int t = threadIdx.x;
    const int tl = deposit_bits<((1u << LG) - 1u) & ~ML>(t);
    float f[16], xr[16];   // f: of the outputs (!PRE)
    rht_begin<PRE>();
    if constexpr (!PRE) rht_factors(sc, sign, f, [&](int k) { return tl | deposit_bits<ML>(k); });
    rht_wait<PRE>();
    const float isn = rsqrtf(static_cast<float>(n));
    const int64_t b = blockIdx.x;
    if constexpr (PRE) load16_scaled(src + b * n + 16 * t, sc + 16 * t, sign + 16 * t, xr);
    else load16(src + b * n + 16 * t, xr);
    fwht_kbits<0xFu>(xr);
    rr_transpose<LG, 1>(xr, osm, t);
    if constexpr (NPH > 2) rr_transpose<LG, 2>(xr, osm, t);
    if constexpr (NPH > 3) rr_transpose<LG, 3>(xr, osm, t);
    float* out = dst + b * n;
#pragma unroll
    for (int k = 0; k < 16; ++k) out[tl | deposit_bits<ML>(k)] = PRE ? xr[k] * isn : xr[k] * isn * f[k];
}

// n = 28 P, P = 2^LG (512, 1024): a cluster of seven CTAs per token, four rows of P each (P / 16
// threads a row, H_P in registers); then each CTA mixes a seventh of the columns, one per
// thread, from the seven CTAs' shared memory. (One CTA of 896 threads did all of it before:
// 27 us at n = 14336 from cold caches.)
template <int LG, bool PRE>
__global__ void __launch_bounds__((1 << LG) / 4) infer_rht28_reg_kernel(const float* __restrict__ src, int n,
                                                                        const float* __restrict__ sc,
                                                                        const int8_t* __restrict__ sign,
                                                                        float* __restrict__ dst) {
    constexpr int P = 1 << LG, TR = P / 16, NPH = rr_phases(LG), PC = (P + 6) / 7;
    static_assert(PC <= 4 * TR, "one column per thread");
    constexpr uint32_t ML = rr_mask(LG, NPH - 1);
    extern __shared__ __align__(16) float osm[];   // [4][P + P / 32] exchange buffers, then [4][P] rows
    cg::cluster_group cl = cg::this_cluster();
    const int rank = static_cast<int>(cl.block_rank());
    const int64_t b = blockIdx.x / 7;
    const int row = threadIdx.x / TR, t = threadIdx.x - row * TR;
    const int tl = deposit_bits<((1u << LG) - 1u) & ~ML>(t);
    const int col = rank * PC + static_cast<int>(threadIdx.x);
    const bool mixes = static_cast<int>(threadIdx.x) < PC && col < P;
    float f[28], xr[16];   // f: of the outputs (!PRE)
    rht_begin<PRE>();
    if constexpr (!PRE) rht_factors(sc, sign, f, [&](int a) { return a * P + (mixes ? col : 0); });
    rht_wait<PRE>();
    const float isn = rsqrtf(static_cast<float>(n));
    const int j0 = (4 * rank + row) * P + 16 * t;
    if constexpr (PRE) load16_scaled(src + b * n + j0, sc + j0, sign + j0, xr);
    else load16(src + b * n + j0, xr);
    float* buf = osm + row * (P + P / 32);
    fwht_kbits<0xFu>(xr);
    rr_transpose<LG, 1>(xr, buf, t);
    if constexpr (NPH > 2) rr_transpose<LG, 2>(xr, buf, t);
    __syncthreads();   // every row's exchange buffer has been read
#pragma unroll
    for (int k = 0; k < 16; ++k) osm[row * P + (tl | deposit_bits<ML>(k))] = xr[k];
    cl.sync();
    if (mixes) {
        float xa[28];
#pragma unroll
        for (int c = 0; c < 7; ++c) {
            const float* rv = cl.map_shared_rank(osm, c);
#pragma unroll
            for (int q = 0; q < 4; ++q) xa[4 * c + q] = rv[q * P + col];
        }
        float* out = dst + b * n + col;
        mix28_paley(xa, [&](int a, float v) { out[a * P] = PRE ? v * isn : v * isn * f[a]; });
    }
    cl.sync();   // keep this CTA's rows alive until every CTA has read them
}

// ---------------------------------------------------------------- product on the tensor cores
// y' = Q' x'. A cluster of C CTAs takes 128 rows, each CTA a range of the 128-column groups; its 8
// warps take 16 rows each. A lane reads its rows' codes straight from global memory (rows g and
// g + 8 of the warp's 16, the 32 codes 32 t .. of each group, g = lane / 4, t = lane % 4), turns
// pairs of them into bf16 (q - c, c the middle code: exact) and multiplies with mma.sync
// m16n8k16: the k order inside a group is whatever pairs the codes' bits give, and x' is
// staged in that order. x' = hi + mid + lo, three bf16 terms (exact to fp32's 24 bits), and the
// terms of the tokens are the columns n = 3 token + term, so that every product is exact, sums are
// fp32, and one or two tokens take one product per k step (NC = 1), five two, eight three. Per
// group and column
//   y'_r += scale_rg (sum (q - c) x' - (zero_rg - c) sum x'),
// the column sums from the same instruction with a matrix of ones. The C CTAs' sums are added
// through distributed shared memory in rank order, the three terms last.
constexpr int IM_ROWS = 128;             // rows per cluster
constexpr int IM_KLD = 72;               // 32-bit words per (k step, term): 32 lanes x 2, padded so
                                         // that the staging stores of four k steps hit other banks
constexpr int IM_GW = 8 * IM_KLD;        // words per (group, term)

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint2 b) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}
__device__ __forceinline__ uint32_t bf16x2_bits(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// The 32 codes of a lane's part of a group: 32 PB / 32 = PB words.
template <int PB>
struct LaneCodes {
    uint32_t w[PB];
    __device__ __forceinline__ void load(const uint8_t* p) {
        if constexpr (PB == 2) {
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
            w[0] = v.x;
            w[1] = v.y;
        } else {
#pragma unroll
            for (int q = 0; q < PB / 4; ++q) {
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(p) + q);
                w[4 * q] = v.x;
                w[4 * q + 1] = v.y;
                w[4 * q + 2] = v.z;
                w[4 * q + 3] = v.w;
            }
        }
    }
    // pair `i` (0 or 1) of k step s as bf16 (q - c): codes at bits sh and sh + 16 of a word (PB 2,
    // 4), bytes 2 i and 2 i + 1 of word s (PB 8)
    __device__ __forceinline__ uint32_t pair(int s, int i, uint32_t c2, float c) const {
        if constexpr (PB == 8) {
            const float m = 8388608.0f + c;
            return bf16x2_bits(byte_raw(w[s], 2 * i) - m, byte_raw(w[s], 2 * i + 1) - m);
        } else {
            constexpr int SPW = 8 / PB;   // k steps per word
            const uint32_t sh = static_cast<uint32_t>(PB * (2 * (s % SPW) + i));
            constexpr uint32_t mask = PB == 2 ? 0x00030003u : 0x000F000Fu;
            const uint32_t u = ((w[s / SPW] >> sh) & mask) | 0x43004300u;   // 128 + q
            const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&u),
                                             *reinterpret_cast<const __nv_bfloat162*>(&c2));
            return *reinterpret_cast<const uint32_t*>(&d);
        }
    }
};
// Columns (within a group) of pair p = 0 .. 63, and its k step, lane part t and pair index.
template <int PB>
__device__ __forceinline__ void pair_place(int p, int& c0, int& c1, int& s, int& t, int& i) {
    constexpr int PPW = 16 / PB;        // pairs per word
    constexpr int WPL = PB;             // words per lane part
    const int w = p / PPW, k = p % PPW;
    t = w / WPL;
    s = (w % WPL) * (PPW / 2) + k / 2;
    i = k & 1;
    if constexpr (PB == 8) {
        c0 = 4 * w + 2 * k;
        c1 = c0 + 1;
    } else {
        c0 = 2 * PPW * w + k;
        c1 = c0 + PPW;
    }
}

template <int PB, int NC>
__global__ void __launch_bounds__(256, 2) infer_mma_kernel(const uint8_t* __restrict__ packed,
                                                           const float* __restrict__ scale,
                                                           const int32_t* __restrict__ zero, int d_out, int d_in,
                                                           int ng, int mid, const float* __restrict__ x, int B,
                                                           float* __restrict__ yp, int gmax) {
    // [NC][gmax][8][IM_KLD] x' terms (the partial sums y' [128][8 NC] after the products),
    // [gmax][8 NC] column sums, [gmax][128] (scale, zero - c)
    extern __shared__ __align__(16) uint32_t im[];
    const int nterm = gmax * IM_GW;
    float* gs = reinterpret_cast<float*>(im + max(NC * nterm, IM_ROWS * 8 * NC));
    float2* sz = reinterpret_cast<float2*>(gs + gmax * 8 * NC);
    float* part = reinterpret_cast<float*>(im);
    cg::cluster_group cl = cg::this_cluster();
    const int C = static_cast<int>(cl.num_blocks()), rank = static_cast<int>(cl.block_rank());
    const int G = d_in / 128;
    const int g0 = rank * G / C, g1 = (rank + 1) * G / C;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t rt0 = static_cast<int64_t>(blockIdx.x / C) * IM_ROWS;
    const int64_t rowbytes = static_cast<int64_t>(d_in) / 8 * PB;
    // weights, scales and zero points were there before the preceding kernel (see rht_begin)
    if (threadIdx.x < IM_ROWS && rt0 + threadIdx.x < d_out)
        prefetch_l2(packed + (rt0 + threadIdx.x) * rowbytes + g0 * 16 * PB, static_cast<uint32_t>((g1 - g0) * 16 * PB));
    const bool grouped = ng > 1;
    const int ngl = grouped ? g1 - g0 : 1;   // grids per row here
#pragma unroll 4
    for (int e = threadIdx.x; e < ngl * IM_ROWS; e += 256) {
        const int r = e / ngl, g = e - r * ngl;
        const int64_t gi = min(rt0 + r, static_cast<int64_t>(d_out) - 1) * ng + (grouped ? g0 + g : 0);
        sz[g * IM_ROWS + r] = make_float2(__ldg(scale + gi), static_cast<float>(__ldg(zero + gi) - mid));
    }
    const int gl = lane >> 2, t = lane & 3;
    const uint8_t* pa = packed + min(rt0 + warp * 16 + gl, static_cast<int64_t>(d_out) - 1) * rowbytes + t * 4 * PB;
    const uint8_t* pb = packed + min(rt0 + warp * 16 + gl + 8, static_cast<int64_t>(d_out) - 1) * rowbytes + t * 4 * PB;
    constexpr int D = PB == 8 ? 2 : 4;   // groups in flight
    LaneCodes<PB> wa[D], wb[D];
#pragma unroll
    for (int d = 0; d < D; ++d)
        if (g0 + d < g1) {
            wa[d].load(pa + (g0 + d) * (16 * PB));
            wb[d].load(pb + (g0 + d) * (16 * PB));
        }
    pdl_launch_dependents();
    pdl_wait();
    // stage x': a warp per group, the loads of all its tokens in flight, two pairs of columns a lane.
    // (Tokens past B repeat the last one; columns past them hold anything: it stays in their sums.)
    int pc[2][2], po[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        int sp, tt, i;
        pair_place<PB>(lane + 32 * h, pc[h][0], pc[h][1], sp, tt, i);
        po[h] = sp * IM_KLD + 2 * tt + i;
    }
    for (int g = warp; g < g1 - g0; g += 8) {
        const float* xg = x + static_cast<int64_t>(g0 + g) * 128;
        constexpr int TB = NC == 1 ? 2 : NC == 2 ? 5 : 8;   // most tokens
        float v[TB][4];
#pragma unroll
        for (int u = 0; u < TB; ++u) {
            const float* xb = xg + static_cast<int64_t>(min(u, B - 1)) * d_in;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                v[u][2 * h] = __ldcg(xb + pc[h][0]);
                v[u][2 * h + 1] = __ldcg(xb + pc[h][1]);
            }
        }
#pragma unroll
        for (int u = 0; u < TB; ++u) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float r0 = v[u][2 * h], r1 = v[u][2 * h + 1];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const int n = 3 * u + k;
                    const uint32_t hb = bf16x2_bits(r0, r1);
                    im[(n >> 3) * nterm + g * IM_GW + po[h] + (n & 7) * 8] = hb;
                    r0 -= __uint_as_float(hb << 16);
                    r1 -= __uint_as_float(hb & 0xFFFF0000u);
                }
            }
        }
        __syncwarp();
        const uint32_t ones[4] = {0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u};
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int s = 0; s < 8; ++s)
                mma_bf16(acc, ones, *reinterpret_cast<const uint2*>(im + c * nterm + g * IM_GW + s * IM_KLD + 2 * lane));
            if (gl == 0) *reinterpret_cast<float2*>(gs + (g * NC + c) * 8 + 2 * t) = make_float2(acc[0], acc[1]);
        }
    }
    __syncthreads();
    const float cf = static_cast<float>(mid);
    const uint32_t c2 = bf16x2_bits(128.0f + cf, 128.0f + cf);
    float y[NC][4] = {};
    for (int gb = g0; gb < g1; gb += D) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const int g = gb + d;
            if (g < g1) {
                const uint32_t* xg = im + (g - g0) * IM_GW + 2 * lane;
                float acc[NC][4] = {};
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    const uint32_t a[4] = {wa[d].pair(s, 0, c2, cf), wb[d].pair(s, 0, c2, cf), wa[d].pair(s, 1, c2, cf),
                                           wb[d].pair(s, 1, c2, cf)};
#pragma unroll
                    for (int c = 0; c < NC; ++c) mma_bf16(acc[c], a, *reinterpret_cast<const uint2*>(xg + c * nterm + s * IM_KLD));
                }
                if (g + D < g1) {
                    wa[d].load(pa + (g + D) * (16 * PB));
                    wb[d].load(pb + (g + D) * (16 * PB));
                }
                const float2* szg = sz + (grouped ? g - g0 : 0) * IM_ROWS + warp * 16 + gl;
                const float2 s1 = szg[0], s2 = szg[8];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const float2 sx = *reinterpret_cast<const float2*>(gs + ((g - g0) * NC + c) * 8 + 2 * t);
                    y[c][0] = fmaf(s1.x, fmaf(-s1.y, sx.x, acc[c][0]), y[c][0]);
                    y[c][1] = fmaf(s1.x, fmaf(-s1.y, sx.y, acc[c][1]), y[c][1]);
                    y[c][2] = fmaf(s2.x, fmaf(-s2.y, sx.x, acc[c][2]), y[c][2]);
                    y[c][3] = fmaf(s2.x, fmaf(-s2.y, sx.y, acc[c][3]), y[c][3]);
                }
            }
        }
    }
    __syncthreads();   // x' has been read: its space takes the partial sums
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        float* pr = part + (warp * 16 + gl) * 8 * NC + 8 * c + 2 * t;
        *reinterpret_cast<float2*>(pr) = make_float2(y[c][0], y[c][1]);
        *reinterpret_cast<float2*>(pr + 64 * NC) = make_float2(y[c][2], y[c][3]);
    }
    cl.sync();
    // rows [rank per, (rank + 1) per) of every CTA's sums, column by column; then the three terms
    const int per = IM_ROWS / C;   // C divides 128
    float* tot = gs;               // [per][8 NC] (the column sums and grids have been read)
    for (int e = threadIdx.x; e < per * 8 * NC; e += blockDim.x) {
        float v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = c < C ? cl.map_shared_rank(part, c)[rank * per * 8 * NC + e] : 0.0f;
        float a = v[0];
#pragma unroll
        for (int c = 1; c < 8; ++c) a += v[c];
        tot[e] = a;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < per * B; e += blockDim.x) {
        const int tok = e / per, rl = e - tok * per;
        const float* p = tot + rl * 8 * NC + 3 * tok;
        const int64_t r = rt0 + rank * per + rl;
        if (r < d_out && KQ_IN_RANGE(static_cast<int64_t>(tok) * d_out + r, static_cast<int64_t>(B) * d_out))
            yp[static_cast<int64_t>(tok) * d_out + r] = p[0] + (p[1] + p[2]);
    }
    cl.sync();   // keep this CTA's sums alive until every CTA has read them
}

constexpr size_t kInferSmemMax = 226 * 1024;

// The transform of B tokens (PRE: x' = V S_X^-1 x; else y = S_G^-1 U^T y'): in registers for
// n = 2^k (9 <= k <= 14), n = 28 * 512 and 28 * 1024, else infer_rht_kernel (n = 28 P: clusters of
// 7, n = 2^k >= 64: clusters of 8, smaller: one CTA).
template <int LG, bool PRE>
kq_status launch_rht_reg(int64_t B, cudaStream_t st, const float* src, int n, const float* sc, const int8_t* sign,
                         float* dst) {
    constexpr int P = 1 << LG;
    constexpr size_t smem = static_cast<size_t>(P + P / 32) * sizeof(float);
    static std::atomic<uint64_t> attr{0};
    KQ_TRY(once_per_device(attr, [&]() -> kq_status {
        KQ_CUDA(cudaFuncSetAttribute(infer_rht_reg_kernel<LG, PRE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(smem)));
        return KQ_OK;
    }));
    KQ_CUDA(launch_dependent(infer_rht_reg_kernel<LG, PRE>, dim3(static_cast<unsigned>(B)), dim3(P / 16), smem, st, 1u, true,
                             src, n, sc, sign, dst));
    KQ_LAUNCH_CHECK("infer_rht_reg_kernel");
    return KQ_OK;
}

template <bool PRE>
kq_status launch_rht(int64_t B, cudaStream_t st, const float* src, int n, int lg, int h28, const float* sc,
                     const int8_t* sign, float* dst) {
    const unsigned nb = static_cast<unsigned>(B);
    if (h28 && (lg == 9 || lg == 10)) {
        const size_t smem = 4 * (size_t{1} << lg) * 33 / 32 * sizeof(float);
        if (lg == 9)
            KQ_CUDA(launch_dependent(infer_rht28_reg_kernel<9, PRE>, dim3(7 * nb), dim3(128), smem, st, 7u, true, src, n, sc,
                                     sign, dst));
        else
            KQ_CUDA(launch_dependent(infer_rht28_reg_kernel<10, PRE>, dim3(7 * nb), dim3(256), smem, st, 7u, true, src, n,
                                     sc, sign, dst));
        KQ_LAUNCH_CHECK("infer_rht28_reg_kernel");
        return KQ_OK;
    }
    if (!h28) {
        switch (lg) {
            case 9: return launch_rht_reg<9, PRE>(B, st, src, n, sc, sign, dst);
            case 10: return launch_rht_reg<10, PRE>(B, st, src, n, sc, sign, dst);
            case 11: return launch_rht_reg<11, PRE>(B, st, src, n, sc, sign, dst);
            case 12: return launch_rht_reg<12, PRE>(B, st, src, n, sc, sign, dst);
            case 13: return launch_rht_reg<13, PRE>(B, st, src, n, sc, sign, dst);
            case 14: return launch_rht_reg<14, PRE>(B, st, src, n, sc, sign, dst);
            default: break;
        }
    }
    if (h28)
        KQ_CUDA(launch_dependent(infer_rht_kernel<7, PRE>, dim3(7 * nb), dim3(256), (size_t{4} << lg) * sizeof(float), st, 7u,
                                 true, src, n, lg, sc, sign, dst));
    else if (n >= 64)
        KQ_CUDA(launch_dependent(infer_rht_kernel<8, PRE>, dim3(8 * nb), dim3(256), (size_t{1} << (lg - 3)) * sizeof(float),
                                 st, 8u, true, src, n, lg - 3, sc, sign, dst));
    else
        KQ_CUDA(launch_dependent(infer_rht_kernel<1, PRE>, dim3(nb), dim3(256), (size_t{1} << lg) * sizeof(float), st, 1u,
                                 true, src, n, lg, sc, sign, dst));
    KQ_LAUNCH_CHECK("infer_rht_kernel");
    return KQ_OK;
}

// Cluster size and shared memory of infer_mma_kernel: CTAs until they cover the SMs or the cluster
// has 8 (portable), and until a CTA's part of x' leaves room for a second CTA on the SM (or, at
// the largest d_in, fits at all).
struct MmaPlan {
    int C, gmax;
    size_t smem;
};
inline bool infer_mma_plan(int64_t d_out, int64_t d_in, int nc, MmaPlan* p) {
    const int64_t G = d_in / 128, tiles = cdiv(d_out, IM_ROWS);
    auto bytes = [&](int64_t g) {
        const int64_t part = IM_ROWS * 8 * nc;   // partial sums; their totals take at most as much
        return static_cast<size_t>(std::max(g * nc * IM_GW, part) + std::max(g * (8 * nc + 2 * IM_ROWS), part)) * 4;
    };
    const int sms = num_sms();
    p->C = 1;
    while (p->C < 8 && 2 * p->C <= G && (tiles * p->C < sms || bytes(cdiv(G, p->C)) > 112 * 1024)) p->C *= 2;
    p->gmax = static_cast<int>(cdiv(G, p->C));
    p->smem = bytes(p->gmax);
    return p->smem <= kInferSmemMax;
}

inline int mma_nc(int64_t B) { return B <= 2 ? 1 : B <= 5 ? 2 : 3; }   // column tiles of 8 for 3 B terms

// Tokens of one product and its plan: all of them, or half where the terms of six to eight tokens do
// not fit (d_in = 32768: 257 KB for a CTA's eighth of the groups, 182 KB for three or four tokens, which
// have one plan); 0 if no product takes this size.
inline int64_t mma_tokens(int64_t B, int64_t d_out, int64_t d_in, MmaPlan* p) {
    if (infer_mma_plan(d_out, d_in, mma_nc(B), p)) return B;
    const int64_t h = cdiv(B, 2);
    return infer_mma_plan(d_out, d_in, mma_nc(h), p) ? h : 0;
}

template <int PB, int NC>
kq_status launch_mma_nc(const MmaPlan& p, int64_t B, cudaStream_t st, const uint32_t* packed, const float* scale,
                        const int32_t* zero, int64_t d_out, int64_t d_in, int ng, int mid, const float* x, float* yp) {
    static std::atomic<uint64_t> attr{0};
    KQ_TRY(once_per_device(attr, [&]() -> kq_status {
        KQ_CUDA(cudaFuncSetAttribute(infer_mma_kernel<PB, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(kInferSmemMax)));
        return KQ_OK;
    }));
    KQ_CUDA(launch_dependent(infer_mma_kernel<PB, NC>, dim3(static_cast<unsigned>(cdiv(d_out, IM_ROWS) * p.C)), dim3(256),
                             p.smem, st, static_cast<unsigned>(p.C), true, reinterpret_cast<const uint8_t*>(packed), scale,
                             zero, static_cast<int>(d_out), static_cast<int>(d_in), ng, mid, x, static_cast<int>(B), yp,
                             p.gmax));
    KQ_LAUNCH_CHECK("infer_mma_kernel");
    return KQ_OK;
}
template <int PB>
kq_status launch_mma(const MmaPlan& p, int64_t B, cudaStream_t st, const uint32_t* packed, const float* scale,
                     const int32_t* zero, int64_t d_out, int64_t d_in, int ng, int mid, const float* x, float* yp) {
    switch (mma_nc(B)) {
        case 1: return launch_mma_nc<PB, 1>(p, B, st, packed, scale, zero, d_out, d_in, ng, mid, x, yp);
        case 2: return launch_mma_nc<PB, 2>(p, B, st, packed, scale, zero, d_out, d_in, ng, mid, x, yp);
        default: return launch_mma_nc<PB, 3>(p, B, st, packed, scale, zero, d_out, d_in, ng, mid, x, yp);
    }
}

// The sizes this call takes: d_in a rotation size of the library (2^k up to 2^15, 28 * 2^k up to
// 28 * 1024); d_out too, or 28 * 2048 and 65536 with 16-byte aligned grids while the tokens' x' (33 floats for
// 32) and eight rows of codes and grids are at most 226 KB. The kernels need neither condition (see
// infer_mma_plan for theirs): they say which of these two d_out the call takes, and d_in * B for them.
inline bool rotation_size(int64_t n) { return n % 28 == 0 ? n <= 28 * 1024 : n <= 32768; }
inline bool sizes_ok(int64_t B, int64_t d_out, int64_t d_in, int pb, int64_t ng, const void* scale, const void* zero) {
    if (!rotation_size(d_in)) return false;
    if (rotation_size(d_out)) return true;
    const int64_t S = cdiv(d_in / 8 * pb / 16, 32);
    const int64_t xbytes = B * S * (32 / pb) * 132 * 4;
    const int64_t rows = 2 * (4 * (d_in / 8 * pb) + 32 * ng + (4 * S * B + 3) / 4 * 16);
    return d_out <= 65536 && ((reinterpret_cast<uintptr_t>(scale) | reinterpret_cast<uintptr_t>(zero)) & 15u) == 0 &&
           xbytes + rows <= static_cast<int64_t>(kInferSmemMax);
}

// n = 28 * 2^k or 2^k: (k, has28); false if neither.
inline bool rht_plan(int64_t n, int* lg, int* h28) {
    int64_t p = n;
    *h28 = 0;
    if (n % 28 == 0) {
        p = n / 28;
        *h28 = 1;
    }
    if (p < 1 || (p & (p - 1))) return false;
    int k = 0;
    while ((int64_t{1} << k) < p) ++k;
    *lg = k;
    return true;
}

inline size_t al256(size_t b) { return (b + 255) & ~static_cast<size_t>(255); }

}  // namespace

KQ_DEBUG_UNIT(infer)
}  // namespace kq

using namespace kq;

extern "C" size_t kq_packed_codes_bytes(int64_t d_out, int64_t d_in, int bits) {
    if (d_out < 1 || d_in < 1 || bits < 1 || bits > 8 || bits == 5 || bits == 6 || bits == 7 || bits == 1) return 0;
    return static_cast<size_t>(d_out) * static_cast<size_t>(d_in) * lane_bits(bits) / 8;
}

extern "C" kq_status kq_pack_codes(const uint8_t* codes, int64_t d_out, int64_t d_in, int bits, uint32_t* packed,
                                   kq_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (!codes || !packed || d_out < 1 || d_in < 1) {
        set_error("kq_pack_codes: invalid arguments");
        return KQ_ERR_INVALID_ARG;
    }
    if (kq_packed_codes_bytes(d_out, d_in, bits) == 0 || (d_in % 128) != 0 ||
        (reinterpret_cast<uintptr_t>(packed) & 15u)) {
        set_error("kq_pack_codes: bits must be 2, 3, 4 or 8, d_in a multiple of 128, packed 16-byte aligned");
        return KQ_ERR_UNSUPPORTED;
    }
    const int pb = lane_bits(bits);
    const int64_t words = d_out * d_in / (32 / pb);
    const int64_t grid = std::min<int64_t>(cdiv(words, 256), static_cast<int64_t>(num_sms()) * 16);
    pack_kernel<<<static_cast<unsigned>(grid), 256, 0, stream>>>(codes, d_out, d_in, pb, packed);
    KQ_LAUNCH_CHECK("pack_kernel");
    return KQ_OK;
}

extern "C" size_t kq_infer_workspace(int64_t B, int64_t d_in, int64_t d_out) {
    if (B < 1 || d_in < 1 || d_out < 1) return 0;
    return al256(static_cast<size_t>(B) * d_in * sizeof(float)) + al256(static_cast<size_t>(B) * d_out * sizeof(float));
}

extern "C" kq_status kq_infer(const uint32_t* packed, const float* scale, const int32_t* zero, int64_t d_out,
                              int64_t d_in, int bits, int group, const float* s_x, const float* s_g,
                              const int8_t* sign_u, const int8_t* sign_v, const float* x, int64_t B, float* y,
                              int* info, void* ws, size_t ws_bytes, kq_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (!packed || !scale || !zero || !s_x || !s_g || !sign_u || !sign_v || !x || !y || d_out < 1 || d_in < 1 || B < 1 ||
        B > KQ_INFER_MAX_B) {
        set_error("kq_infer: invalid arguments (B must be 1..%d)", KQ_INFER_MAX_B);
        return KQ_ERR_INVALID_ARG;
    }
    if (kq_packed_codes_bytes(d_out, d_in, bits) == 0 || (d_in % 128) != 0 || (group != 0 && group != 128) ||
        (reinterpret_cast<uintptr_t>(packed) & 15u) || (reinterpret_cast<uintptr_t>(x) & 15u) ||
        (reinterpret_cast<uintptr_t>(s_x) & 15u) || (reinterpret_cast<uintptr_t>(sign_v) & 3u) ||
        (reinterpret_cast<uintptr_t>(s_g) & 15u) || (reinterpret_cast<uintptr_t>(sign_u) & 3u) ||
        (reinterpret_cast<uintptr_t>(y) & 15u) || (d_out % 4) != 0) {
        set_error("kq_infer: bits in {2, 3, 4, 8}, d_in %% 128 == 0, d_out %% 4 == 0, group 0 or 128, 16-byte "
                  "aligned codes, x, y, s_x, s_g, 4-byte aligned signs");
        return KQ_ERR_UNSUPPORTED;
    }
    if (!ws || ws_bytes < kq_infer_workspace(B, d_in, d_out) || (reinterpret_cast<uintptr_t>(ws) & 255u)) {
        set_error("kq_infer: workspace must be 256-byte aligned and hold %zu bytes", kq_infer_workspace(B, d_in, d_out));
        return KQ_ERR_WORKSPACE;
    }
    float* xt = static_cast<float*>(ws);   // x' of the tokens; y' behind it (see kq_infer_workspace)
    float* yp = reinterpret_cast<float*>(static_cast<uint8_t*>(ws) + al256(static_cast<size_t>(B) * d_in * sizeof(float)));
    const int pb = lane_bits(bits);
    int lgi = 0, h28i = 0, lgo = 0, h28o = 0;
    if (!rht_plan(d_in, &lgi, &h28i) || !rht_plan(d_out, &lgo, &h28o)) {
        set_error("kq_infer: d_in=%lld or d_out=%lld has no Hadamard construction", (long long)d_in, (long long)d_out);
        return KQ_ERR_UNSUPPORTED;
    }
    const int ng = group ? static_cast<int>(d_in / group) : 1;
    const int di = static_cast<int>(d_in), dn = static_cast<int>(d_out);
    MmaPlan plan;
    const int64_t per = mma_tokens(B, d_out, d_in, &plan);
    if (!sizes_ok(B, d_out, d_in, pb, ng, scale, zero) || per == 0) {
        set_error("kq_infer: d_in=%lld or d_out=%lld is beyond the rotation sizes", (long long)d_in, (long long)d_out);
        return KQ_ERR_UNSUPPORTED;
    }
    (void)info;   // no kernel of this call waits on a copy
    KQ_TRY(launch_rht<true>(B, stream, x, di, lgi, h28i, s_x, sign_v, xt));
    const int mid = 1 << (bits - 1);
    for (int64_t t0 = 0; t0 < B; t0 += per) {
        const int64_t n = std::min(per, B - t0);
        const float* xn = xt + t0 * d_in;
        float* yn = yp + t0 * d_out;
        if (pb == 2) KQ_TRY(launch_mma<2>(plan, n, stream, packed, scale, zero, d_out, d_in, ng, mid, xn, yn));
        else if (pb == 4) KQ_TRY(launch_mma<4>(plan, n, stream, packed, scale, zero, d_out, d_in, ng, mid, xn, yn));
        else KQ_TRY(launch_mma<8>(plan, n, stream, packed, scale, zero, d_out, d_in, ng, mid, xn, yn));
    }
    return launch_rht<false>(B, stream, yp, dn, lgo, h28o, s_g, sign_u, y);
}
