// Stage 4: the column-wise OBS sweep with b-bit asymmetric grids.
//
// Paper: Sec. 2.1 Eq. (obs_update) (compensation -(w_p - q_p)/[H^-1]_pp [H^-1]_{p,p+1:}),
// Algorithm 2 (inner column loop over a block of B columns with error E, then the lazy
// trailing update W[:, i+B:] -= E R[i:i+B, i+B:]), Proposition 1 (H_G cancels, so only
// L = R^T enters). With the GPTAQ correction P (Proposition 1, Algorithm 2) each column j
// also adds w_j P[j, k] to the later columns k, w_j being column j's value just before it
// is quantized; the lazy update then subtracts [E | -Wpre] [R ; P]. GPTQ mode: no P.
//
// Every fp32 operation is written with an explicit round-to-nearest intrinsic so the
// compiler cannot contract or reorder it; the order is:
//   grid      scale = (xmax - xmin) / (2^b - 1), zero = rint(-xmin / scale)
//   column j  q = clamp(rint(w / scale) + zero, 0, 2^b - 1); what = scale * (q - zero)
//             E = (w - what) / R_jj;  w_k = fma(-E, R_jk, w_k) for k in (j, block end)
//             with P: w_k = fma(w_j, P_jk, fma(-E, R_jk, w_k))
//   trailing  acc = fma(E_k, R_kc, acc) over ascending k; with P continuing
//             acc = fma(-wpre_k, P_kc, acc) over ascending k; w_c = w_c - acc
// Kernels:
//   rowgrid_kernel   per-row grid (group = 0) from the whole row before the sweep
//   pack_r_kernel    the diagonal 128 x 128 blocks of R as the block kernel's 16 x 16 tiles, and
//                    the blocks of R right of them, for the fused update
//   obs_block_kernel 32 rows per CTA, lane = row, 16 columns per warp
//   trailing_kernel  128 x 128 output tiles of the shared tile GEMM (tile_gemm.cuh)
//   colloss_kernel   col_loss[j] = sum over rows of E_j^2, fixed order (sumsq.cuh)
#include <math.h>

#include <cstdlib>
#include <type_traits>

#include "kq_common.cuh"
#include "tile_gemm.cuh"
#include "sumsq.cuh"
#include "trail_tc.cuh"

namespace kq {
namespace {

constexpr int BLK = 128;          // block size B (Algorithm 2); the only supported value
constexpr int SPB = 8;            // blocks per super-panel of the two-level lazy update

struct Grid {
    float scale, zero;
};

__device__ __forceinline__ Grid make_grid(float xmin, float xmax, float maxq) {
    xmin = fminf(xmin, 0.0f);
    xmax = fmaxf(xmax, 0.0f);
    if (xmin == 0.0f && xmax == 0.0f) {
        xmin = -1.0f;
        xmax = 1.0f;
    }
    Grid g;
    g.scale = __fdiv_rn(__fsub_rn(xmax, xmin), maxq);
    g.zero = rintf(__fdiv_rn(-xmin, g.scale));
    return g;
}

__device__ __forceinline__ float warp_min(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Per-row grid from the whole row (group = 0). Warp per row.
__global__ void rowgrid_kernel(const float* __restrict__ W, int64_t d_out, int64_t d_in, int bits,
                               float* __restrict__ scale, int32_t* __restrict__ zero,
                               float* __restrict__ gscale, float* __restrict__ gzero) {
    const int64_t r = static_cast<int64_t>(blockIdx.x) * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x & 31;
    if (r >= d_out) return;
    float mn = 0.0f, mx = 0.0f;
    for (int64_t j = lane; j < d_in; j += 32) {
        const float v = W[r * d_in + j];
        mn = fminf(mn, v);
        mx = fmaxf(mx, v);
    }
    mn = warp_min(mn);
    mx = warp_max(mx);
    const Grid g = make_grid(mn, mx, static_cast<float>((1 << bits) - 1));
    if (lane == 0 && KQ_IN_RANGE(r, d_out)) {
        scale[r] = g.scale;
        zero[r] = static_cast<int32_t>(g.zero);
        gscale[r] = g.scale;
        gzero[r] = g.zero;
    }
}

// One block [i0, e) of the sweep. A CTA takes 32 rows, lane = row, and its 8 warps take 16
// consecutive columns each (warp s: columns i0 + 16 s ..), held in registers. The column loop
// is a serial chain per row: quantize w_j, form E_j, update w_{j+1}. Warp o runs the chain of
// its 16 columns with every value of a row in one lane (no exchange inside the 16 columns),
// and after every 4 columns publishes their E (and with P the values before quantization)
// through shared memory and one mbarrier arrival; the warps s > o, which own the later
// columns, then apply those 4 columns' updates while warp o goes on, so that warp o + 1
// starts its own chain a few fma after warp o's last column. Every column still receives
// the updates j = 0, 1, ... in order with the definition's operations.
// Bound: the chain's latency, ~20 dependent operations a column (two corrected divisions of 5,
// rounding 2, clamp 2, product, difference, update): 140-165 cycles a column measured, plus
// ~350-500 cycles for each of the seven hand-overs and ~5000 before the first column.
// 4096 rows (128 CTAs): 30.3 k cycles, 14.6 us a block; the form with 8 lanes per row and a
// shuffle per column took 25 us. With it the sweep of 1024 x 8192 went from 2.62 to 1.75 ms,
// of 14336 x 4096 (three CTAs per SM) from 3.40 to 2.29 ms (2.23 with the column sums' loads ahead). A fully unrolled chain with one
// register per column and range tests that branch took 270 cycles a column; packed pairs
// (f32x2 fma) for the updates, 16 against 30 instructions, took 170 to 145.
constexpr int CW = 16;                      // columns per warp
constexpr int NWARP = BLK / CW;             // 8 warps
constexpr int OBS_ROWS = 32;                // rows per CTA
constexpr int OBS_THREADS = 32 * NWARP;
constexpr int PUB = 4;                      // columns per publication
constexpr int NPUB = BLK / PUB;             // publications (one mbarrier each)
constexpr int ELD = OBS_ROWS + 2;           // column stride of the exchange tiles [16][ELD]: 8 rows x 4
                                            // column quads of a transposing access hit 32 banks
constexpr int XT = CW * ELD;                // floats of one warp's exchange tile
constexpr int PLD = BLK + 4;                // row stride of the staged E_prev
// Packed diagonal block of R: the 16 x 16 tiles (o, s), o <= s, the only ones the block's
// column loop reads (36 of 64), tile s (s + 1) / 2 + o, row-major; the diagonal tiles (s, s)
// with row jj shifted left by 4 (jj / 4): [jj][t] = R[jj][4 (jj / 4) + t] (0 past the tile). The
// chain shifts its registers the same way after every 4 columns, so its loop has fixed
// register indices and a body of 4 columns.
constexpr int RT = CW * CW;
constexpr int RTILES = NWARP * (NWARP + 1) / 2;
constexpr int RPACK = RTILES * RT;          // 9216 floats, 36 KB
__host__ __device__ constexpr int rtile(int o, int s) { return (s * (s + 1) / 2 + o) * RT; }
// Shared memory: R's tiles (with P also P's), the exchange tiles of E (with P also of Wpre).
// 54 KB (GPTQ mode): four CTAs per SM by shared memory, or one beside a 129 KB far-update CTA.
constexpr int obs_smem(bool hasp) { return (hasp ? 2 : 1) * (RPACK + NWARP * XT) * static_cast<int>(sizeof(float)); }
static_assert(OBS_ROWS * PLD <= NWARP * XT, "E_prev is staged in the exchange tiles");
// How the previous block's lazy update of this block column is applied.
enum { FUSE_NONE = 0, FUSE_FP32 = 1, FUSE_MMA = 2 };

// Rp[b][tile(o, s)][jj][t] = R[i0 + 16 o + jj][i0 + 16 s + t] = Lt[i0 + 16 s + t][i0 + 16 o + jj]
// (0 outside the matrix; diagonal tiles shifted as above), i0 = b BLK, b = blockIdx.y: tile `tile` by 256 threads.
__device__ __forceinline__ void pack_r_tile(const float* __restrict__ Lt, int64_t n, float* __restrict__ Rp, int tile) {
    __shared__ float t[CW][CW + 1];
    const int tx = threadIdx.x % CW, ty = threadIdx.x / CW;
    int s = 0, o = tile;
    while (o > s) {
        o -= s + 1;
        ++s;
    }
    const int64_t i0 = static_cast<int64_t>(blockIdx.y) * BLK;
    const int64_t c = i0 + CW * s + ty, j = i0 + CW * o + tx;
    t[ty][tx] = (c < n && j < n) ? Lt[c * n + j] : 0.0f;
    __syncthreads();
    const int64_t e = static_cast<int64_t>(blockIdx.y) * RPACK + rtile(o, s) + ty * CW + tx;
    const int jj = ty;
    int tt = tx;   // column within the tile
    if (o == s) tt += PUB * (jj / PUB);
    if (KQ_IN_RANGE(e, static_cast<int64_t>(gridDim.y) * RPACK)) Rp[e] = tt < CW ? t[tt][jj] : 0.0f;
}

// The block of R right of diagonal block b (rows i0 + k, columns i0 + BLK + c; 0 outside the
// matrix) for the fused update. FRAG = false: Rq[b][s][k][t], c = 16 s + t: warp s reads a row
// of 16 columns as four uniform 16-byte loads. FRAG = true: Rq[b][s][ks][lane][4] =
// (R[8 ks + t4][c], R[8 ks + t4 + 4][c], the same at c + 8), c = 16 s + g, g = lane / 4,
// t4 = lane % 4: the B fragments of mma.sync m16n8k8 for warp s's two column tiles, one
// 16-byte load per lane and k step. b = blockIdx.y; warp s's part by 256 threads.
template <bool FRAG>
__device__ __forceinline__ void pack_rq_part(const float* __restrict__ Lt, int64_t n, float* __restrict__ Rq, int s) {
    const int64_t i0 = static_cast<int64_t>(blockIdx.y) * BLK, i1 = i0 + BLK + CW * s;
    float* out = Rq + static_cast<int64_t>(blockIdx.y) * BLK * BLK + s * BLK * CW;
    __shared__ float t[CW][BLK + 1];
    for (int e = threadIdx.x; e < CW * BLK; e += blockDim.x) {
        const int c = e / BLK, k = e % BLK;
        t[c][k] = (i1 + c < n && i0 + k < n) ? Lt[(i1 + c) * n + i0 + k] : 0.0f;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < CW * BLK; e += blockDim.x) {
        float v;
        if constexpr (FRAG) {
            const int u = e & 3, lane = (e >> 2) & 31, ks = e >> 7;
            v = t[(lane >> 2) + 8 * (u >> 1)][8 * ks + (lane & 3) + 4 * (u & 1)];
        } else {
            v = t[e % CW][e / CW];
        }
        if (KQ_IN_RANGE(e, CW * BLK)) out[e] = v;
    }
}

// Both packings in one launch: a launch costs a short sweep as much as the copying does.
// Grid (RTILES, blocks), or with RQ != PACK_NONE (RTILES + NWARP, blocks); block 256.
enum { PACK_NONE = 0, PACK_ROWS = 1, PACK_FRAG = 2 };
template <int RQ>
__global__ void __launch_bounds__(256) pack_r_kernel(const float* __restrict__ Lt, int64_t n, float* __restrict__ Rp,
                                                     float* __restrict__ Rq) {
    const int x = static_cast<int>(blockIdx.x);
    if (x < RTILES) {
        pack_r_tile(Lt, n, Rp, x);
    } else if constexpr (RQ != PACK_NONE) {
        if (blockIdx.y + 1 < gridDim.y) pack_rq_part<RQ == PACK_FRAG>(Lt, n, Rq, x - RTILES);   // the last block has no next
    }
}

// Warp `warp`'s 16 columns of the CTA's rows in the transposing layout: lane (8 rows x 4 quads)
// holds rows r0 + 8 it + lane / 4, columns c0 + 4 (lane % 4) .. + 3 of M (0 past row d_out or
// column cend).
template <bool VEC>
__device__ __forceinline__ void load_quads(const float* M, int64_t r0, int64_t d_out, int64_t d_in,
                                           int64_t c0, int64_t cend, float4 (&v)[4]) {
    const int lane = threadIdx.x & 31;
    const int64_t c = c0 + 4 * (lane & 3);
    if (VEC && r0 + OBS_ROWS <= d_out && c0 + CW <= cend) {   // the whole tile
        const float* p = M + (r0 + (lane >> 2)) * d_in + c;
#pragma unroll
        for (int it = 0; it < 4; ++it) v[it] = *reinterpret_cast<const float4*>(p + it * 8 * d_in);
        return;
    }
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int64_t r = r0 + 8 * it + (lane >> 2);
        v[it] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (r >= d_out) continue;
        const float* p = M + r * d_in + c;
        if (VEC && c + 3 < cend) {
            v[it] = *reinterpret_cast<const float4*>(p);
        } else {
            if (c < cend) v[it].x = p[0];
            if (c + 1 < cend) v[it].y = p[1];
            if (c + 2 < cend) v[it].z = p[2];
            if (c + 3 < cend) v[it].w = p[3];
        }
    }
}

template <bool VEC>
__device__ __forceinline__ void store_quad(float* M, int64_t r, int64_t d_out, int64_t d_in, int64_t c, int64_t cend,
                                           const float (&v)[4]) {
    if (r >= d_out || c >= cend || !KQ_IN_RANGE(r * d_in + (c + 3 < cend ? c + 3 : cend - 1), d_out * d_in)) return;
    float* p = M + r * d_in + c;
    if (VEC && c + 3 < cend) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (c + u < cend) p[u] = v[u];
    }
}

// The previous block's lazy update of warp s's 16 columns for the CTA's 32 rows on the tensor
// cores (mma.sync m16n8k8 tf32, 3xTF32 split, ascending k): C = E_prev R_prev,this with E_prev
// staged in Es ([32][PLD]) and the lane's B fragments of every k step in registers (each CTA
// reads every fragment once). c[mt][nt]: rows 16 mt, columns 8 nt of the warp's 32 x 16 tile.
__device__ __forceinline__ void prev_block_update_mma(const float* Es, const float4 (&frag)[BLK / 8], float (&c)[2][2][4]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) c[mt][nt][e] = 0.0f;
#pragma unroll
    for (int ks = 0; ks < BLK / 8; ++ks) {
        const float4 bf = frag[ks];
        const float b[2][2] = {{bf.x, bf.y}, {bf.z, bf.w}};
        uint32_t bh[2][2], bl[2][2];
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float hi = tf32_hi(b[nt][e]);
                bh[nt][e] = __float_as_uint(hi);
                bl[nt][e] = __float_as_uint(b[nt][e] - hi);
            }
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            const float* a0p = Es + (16 * mt + g) * PLD + 8 * ks;
            const float* a1p = a0p + 8 * PLD;
            const float a[4] = {a0p[t4], a1p[t4], a0p[t4 + 4], a1p[t4 + 4]};
            uint32_t ah[4], al[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float hi = tf32_hi(a[e]);
                ah[e] = __float_as_uint(hi);
                al[e] = __float_as_uint(a[e] - hi);
            }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                mma_tf32(c[mt][nt], al, bh[nt]);
                mma_tf32(c[mt][nt], ah, bl[nt]);
                mma_tf32(c[mt][nt], ah, bh[nt]);
            }
        }
    }
}

// The same in fp32 in the order of the trailing update (acc = fma(E_k, R_kc, acc) over
// ascending k) for the lane's row; rq: warp s's columns of R_prev,this ([BLK][16]).
__device__ __forceinline__ void prev_block_update(const float* Es, const float* __restrict__ rq, float (&acc)[CW]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int t = 0; t < CW; ++t) acc[t] = 0.0f;
#pragma unroll 2
    for (int k = 0; k < BLK; k += 4) {
        const float4 e4 = *reinterpret_cast<const float4*>(Es + lane * PLD + k);
        const float ek[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4* rr = reinterpret_cast<const float4*>(rq + (k + u) * CW);
#pragma unroll
            for (int v = 0; v < CW / 4; ++v) {
                const float4 x = __ldg(rr + v);
                acc[4 * v] = __fmaf_rn(ek[u], x.x, acc[4 * v]);
                acc[4 * v + 1] = __fmaf_rn(ek[u], x.y, acc[4 * v + 1]);
                acc[4 * v + 2] = __fmaf_rn(ek[u], x.z, acc[4 * v + 2]);
                acc[4 * v + 3] = __fmaf_rn(ek[u], x.w, acc[4 * v + 3]);
            }
        }
    }
}

// One row's grid and the constants of its column steps: the integer t = q - zero is
// rint(w / scale) clamped to [lo, hi] (the same number as clamp(rint + zero, 0, maxq) - zero:
// all are integers below 2^24 or clamped alike).
struct RowGrid {
    float scale, ys, zero, lo, hi;
};

// What the column steps of a publication met: ok() when div_rn_fast was exact in all of them
// (reciprocals aside). A quotient w / scale only has to round to the right integer: below 1/4
// any error is harmless and above it the residuals are exact for every w, so w needs no lower
// bound; the dividend of E must be 0 or at least 2^-60. nan collects 0 * w.
struct StepRange {
    float mx = 0.0f, mn = 1.0f, nan = 0.0f;
    __device__ __forceinline__ bool ok() const { return (mx <= 0x1p60f) & (mn >= 0x1p-60f) & (nan == 0.0f); }
};

// One column step: t and E for the value w (d.x = 1 / R_jj, d.y = R_jj). !EXACT: div_rn_fast's
// operations, written out; the sign of a zero quotient does not matter to the rounding of the
// first division, which skips the a == 0 case; rounding is the addition of 1.5 * 2^23 (to
// nearest even below 2^22; beyond, the clamp decides).
template <bool EXACT>
__device__ __forceinline__ void column_step(float w, const RowGrid& g, float2 d, float& t, float& err, StepRange& sr) {
    if constexpr (EXACT) {
        t = fminf(fmaxf(rintf(__fdiv_rn(w, g.scale)), g.lo), g.hi);
        err = __fdiv_rn(__fsub_rn(w, __fmul_rn(g.scale, t)), d.y);
    } else {
        const float q0 = __fmul_rn(w, g.ys);
        const float q1 = __fmaf_rn(__fmaf_rn(-q0, g.scale, w), g.ys, q0);
        const float q2 = __fmaf_rn(__fmaf_rn(-q1, g.scale, w), g.ys, q1);
        t = fminf(fmaxf(__fsub_rn(__fadd_rn(q2, 12582912.0f), 12582912.0f), g.lo), g.hi);
        const float dif = __fsub_rn(w, __fmul_rn(g.scale, t));
        err = div_rn_fast(dif, d.y, d.x);
        sr.mx = fmaxf(sr.mx, fmaxf(fabsf(w), fabsf(dif)));
        sr.mn = fminf(sr.mn, dif == 0.0f ? 1.0f : fabsf(dif));
        sr.nan = __fmaf_rn(w, 0.0f, sr.nan);
    }
}

// A thread whose wait ran out: NaN in its part of what the later updates read, so that even without a
// word in info the columns after these and col_loss are NaN, not sums of what the workspace held.
// (Places from the special registers again: nothing is kept in registers for this.)
__device__ __forceinline__ void give_up(float* E, float* Eh, float* El, int64_t d_out, int64_t d_in, int64_t i0, int* info) {
    uint32_t tid, cta;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
    asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(cta));
    record_error(info, -KQ_ERR_TIMEOUT);
    const int64_t r = static_cast<int64_t>(cta) * OBS_ROWS + (tid & 31), c0 = i0 + CW * (tid >> 5);
    if (r >= d_out) return;
#pragma unroll 1
    for (int64_t c = c0; c < min(c0 + CW, d_in); ++c) {
        E[r * d_in + c] = __int_as_float(0x7FFFFFFF);
        if (Eh) Eh[r * d_in + c] = El[r * d_in + c] = __int_as_float(0x7FFFFFFF);
    }
}

// VEC: d_in % 16 == 0 and W and codes 16-byte aligned, so a lane's columns of W, E
// and codes move as 16-byte vectors. HASP: with the GPTAQ correction; Pp is P's
// diagonal block packed like R's, and the block's -Wpre goes to Q (fp32 trailing update)
// or to Qh + Ql (tensor-core trailing update). FUSE: the previous block's update of this
// block column first (Rq: pack_rq_part's layout for that form). One CTA per 32 rows.
template <bool VEC, bool HASP, int FUSE, int PER_SM = 2>
__global__ void __launch_bounds__(OBS_THREADS, PER_SM) obs_block_kernel(
    const float* W, int64_t d_out, int64_t d_in, const float* __restrict__ Rp, int64_t i0,
    int bits, int group, const float* __restrict__ gscale, const float* __restrict__ gzero,
    uint8_t* __restrict__ codes, float* __restrict__ scale, int32_t* __restrict__ zero,
    float* E, float* __restrict__ pre_q, float* __restrict__ Eh, float* __restrict__ El,
    const float* __restrict__ Pp, float* __restrict__ Q, float* __restrict__ Qh, float* __restrict__ Ql,
    const float* __restrict__ Rq, int* info) {
    extern __shared__ __align__(16) float Rs[];   // R's tiles, exchange tiles, with P: P's tiles, Wpre's exchange tiles
    float* Xs = Rs + RPACK;
    float* Ps = Xs + NWARP * XT;
    float* Qs = Ps + RPACK;
    __shared__ uint64_t pub[NPUB];
    __shared__ float mnmx[2][NWARP][OBS_ROWS];
    __shared__ float2 rds[BLK];
    __shared__ int abort_flag, ieee_only;
    const int lane = threadIdx.x & 31, s = threadIdx.x >> 5;
    const int nb = static_cast<int>(min(static_cast<int64_t>(BLK), d_in - i0));
    const int64_t row0 = static_cast<int64_t>(blockIdx.x) * OBS_ROWS;
    const int64_t r = row0 + lane;
    const bool live = r < d_out;
    const int64_t cend = i0 + nb, c0 = i0 + CW * s;
    if (threadIdx.x == 0) {
        for (int k = 0; k < NPUB; ++k) mbar_init(&pub[k], 1);
        fence_mbar_init();
        abort_flag = 0;
        ieee_only = 0;
    }
    // R (and P) do not depend on the kernel before this one (see block_launch): ahead of the wait
    for (int e = threadIdx.x; e < RPACK / 4; e += OBS_THREADS) cp_async16(Rs + 4 * e, Rp + 4 * e, 16);
    if constexpr (HASP)
        for (int e = threadIdx.x; e < RPACK / 4; e += OBS_THREADS) cp_async16(Ps + 4 * e, Pp + 4 * e, 16);
    cp_async_commit();
    float4 frag[FUSE == FUSE_MMA ? BLK / 8 : 1];
    if constexpr (FUSE == FUSE_MMA) {
#pragma unroll
        for (int ks = 0; ks < BLK / 8; ++ks) frag[ks] = __ldg(reinterpret_cast<const float4*>(Rq + s * BLK * CW) + 32 * ks + lane);
    }
    pdl_wait();
    if constexpr (FUSE != FUSE_NONE) {   // E_prev (128 columns) of the CTA's rows into the exchange tiles
        for (int q = threadIdx.x; q < OBS_ROWS * (BLK / 4); q += OBS_THREADS) {
            const int rr = q / (BLK / 4), c4 = 4 * (q % (BLK / 4));
            const bool lv = row0 + rr < d_out;
            const float* src = E + (row0 + rr) * d_in + (i0 - BLK) + c4;
            if constexpr (VEC) {
                cp_async16(Xs + rr * PLD + c4, lv ? src : E, lv ? 16 : 0);
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) Xs[rr * PLD + c4 + u] = lv ? src[u] : 0.0f;
            }
        }
        cp_async_commit();
    }
    float4 wq4[4];
    load_quads<VEC>(W, row0, d_out, d_in, c0, cend, wq4);
    float* xt = Xs + s * XT;                     // this warp's exchange tile
    const int qr = lane >> 2, qc = 4 * (lane & 3);   // this lane's place in the transposing layout
    float2 w[CW / 2];   // the warp's 16 columns of the lane's row, in pairs
    if constexpr (FUSE == FUSE_MMA) {
        cp_async_wait<0>();
        __syncthreads();
        float c[2][2][4];
        prev_block_update_mma(Xs, frag, c);
        __syncthreads();   // every warp is done with E_prev
        const int g = lane >> 2, t2 = 2 * (lane & 3);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                float* x = xt + (8 * nt + t2) * ELD + 16 * mt + g;
                x[0] = c[mt][nt][0];
                x[ELD] = c[mt][nt][1];
                x[8] = c[mt][nt][2];
                x[ELD + 8] = c[mt][nt][3];
            }
        __syncwarp();
#pragma unroll
        for (int it = 0; it < 4; ++it) {   // W - C in place: each lane its own elements
            float* x = xt + qc * ELD + 8 * it + qr;
            x[0] = __fsub_rn(wq4[it].x, x[0]);
            x[ELD] = __fsub_rn(wq4[it].y, x[ELD]);
            x[2 * ELD] = __fsub_rn(wq4[it].z, x[2 * ELD]);
            x[3 * ELD] = __fsub_rn(wq4[it].w, x[3 * ELD]);
        }
    } else {
        float acc[CW];
        if constexpr (FUSE == FUSE_FP32) {
            cp_async_wait<0>();
            __syncthreads();
            prev_block_update(Xs, Rq + s * BLK * CW, acc);
            __syncthreads();   // every warp is done with E_prev
        }
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            float* x = xt + qc * ELD + 8 * it + qr;
            x[0] = wq4[it].x;
            x[ELD] = wq4[it].y;
            x[2 * ELD] = wq4[it].z;
            x[3 * ELD] = wq4[it].w;
        }
        if constexpr (FUSE == FUSE_FP32) {
            __syncwarp();
#pragma unroll
            for (int t = 0; t < CW; ++t) xt[t * ELD + lane] = __fsub_rn(xt[t * ELD + lane], acc[t]);
        }
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < CW / 2; ++t) w[t] = make_float2(xt[2 * t * ELD + lane], xt[(2 * t + 1) * ELD + lane]);
    // The grid of the row: the minimum and maximum of the whole block (values past the end are 0,
    // which the definition includes anyway).
    if (group) {
        float mn = 0.0f, mx = 0.0f;
#pragma unroll
        for (int t = 0; t < CW / 2; ++t) {
            mn = fminf(mn, fminf(w[t].x, w[t].y));
            mx = fmaxf(mx, fmaxf(w[t].x, w[t].y));
        }
        mnmx[0][s][lane] = mn;
        mnmx[1][s][lane] = mx;
    }
    cp_async_wait<0>();
    __syncthreads();
    if (threadIdx.x < BLK) {   // reciprocals of the block's diagonal R_jj for the divisions
        const int j = threadIdx.x;
        // (columns past the end: finite steps, nothing kept)
        const float dj = j < nb ? Rs[rtile(j / CW, j / CW) + (j % CW) * CW + j % PUB] : 1.0f;
        const float y = div_recip(dj);
        rds[j] = make_float2(y, dj);
        if (y == 0.0f) ieee_only = 1;
    }
    const float maxq = static_cast<float>((1 << bits) - 1);
    RowGrid g;
    if (group) {
        float mn = mnmx[0][0][lane], mx = mnmx[1][0][lane];
#pragma unroll
        for (int k = 1; k < NWARP; ++k) {
            mn = fminf(mn, mnmx[0][k][lane]);
            mx = fmaxf(mx, mnmx[1][k][lane]);
        }
        const Grid gr = make_grid(mn, mx, maxq);
        g.scale = gr.scale;
        g.zero = gr.zero;
        const int64_t ngroups = (d_in + BLK - 1) / BLK, gi = r * ngroups + i0 / BLK;   // group == BLK
        if (live && s == 0 && KQ_IN_RANGE(gi, d_out * ngroups)) {
            scale[gi] = g.scale;
            zero[gi] = static_cast<int32_t>(g.zero);
        }
    } else {
        g.scale = live ? gscale[r] : 1.0f;
        g.zero = live ? gzero[r] : 0.0f;
    }
    if (!(fabsf(g.zero) <= 3.402823466e38f)) {   // scale underflowed to 0, or infinite: codes 0, E NaN
        g.scale = __int_as_float(0x7FFFFFFF);
        g.zero = 0.0f;
    }
    g.ys = div_recip(g.scale);
    g.lo = __fsub_rn(0.0f, g.zero);
    g.hi = __fsub_rn(maxq, g.zero);
    __syncthreads();
    if (CW * s >= nb) return;   // no columns (a last block narrower than 128)
    // The earlier warps' columns.
    for (int o = 0; o < s; ++o) {
        const float* rt = Rs + rtile(o, s);
        const float* ex = Xs + o * XT;
#pragma unroll 1
        for (int p = 0; p < CW / PUB; ++p) {
            if (!mbar_wait(&pub[o * (CW / PUB) + p], 0, &abort_flag)) {
                give_up(E, Eh, El, d_out, d_in, i0, info);
                return;
            }
#pragma unroll
            for (int u = 0; u < PUB; ++u) {
                const int jj = PUB * p + u;
                const float ne = -ex[jj * ELD + lane];
                const float2 ne2 = make_float2(ne, ne);
                const float4* rr = reinterpret_cast<const float4*>(rt + jj * CW);
                float2 wp2 = make_float2(0.0f, 0.0f);
                if constexpr (HASP) wp2.x = wp2.y = Qs[o * XT + jj * ELD + lane];
                (void)wp2;
#pragma unroll
                for (int v = 0; v < CW / 4; ++v) {
                    const float4 x = rr[v];
                    w[2 * v] = __ffma2_rn(ne2, make_float2(x.x, x.y), w[2 * v]);
                    w[2 * v + 1] = __ffma2_rn(ne2, make_float2(x.z, x.w), w[2 * v + 1]);
                    if constexpr (HASP) {
                        const float4 y = reinterpret_cast<const float4*>(Ps + rtile(o, s) + jj * CW)[v];
                        w[2 * v] = __ffma2_rn(wp2, make_float2(y.x, y.y), w[2 * v]);
                        w[2 * v + 1] = __ffma2_rn(wp2, make_float2(y.z, y.w), w[2 * v + 1]);
                    }
                }
            }
        }
    }
    if (CW * (s + 1) >= nb) pdl_launch_dependents();   // the last warp: an eighth of the chain to go
    // This warp's chain, 4 columns (w[0], w[1]) per turn of the loop, the last of which moves the
    // later columns down by 4; the first 8 columns update 16 registers, the last 8 only 8.
    const float* rt = Rs + rtile(s, s);
    const float* pt = Ps + rtile(s, s);
    (void)pt;
    const bool want_pre = pre_q != nullptr && live;
    const bool fast = (g.ys != 0.0f) & (ieee_only == 0) & (c0 + CW <= cend);
    bool finite = true;   // every value quantized was finite
    uint32_t cq[CW / PUB] = {};
    // Column u of turn p; N live pairs. The update touches the pairs from the one that holds
    // column u + 1 on (a value that is no longer read in a pair's lower half does no harm).
    auto column = [&](auto exact_tag, auto live_tag, auto u_tag, int p, float& e, float& wpre, float& t, StepRange& sr) {
        constexpr int N = decltype(live_tag)::value, u = decltype(u_tag)::value;
        const int jj = PUB * p + u;
        const float* rr = rt + jj * CW;
        wpre = (u & 1) ? w[u / 2].y : w[u / 2].x;
        column_step<decltype(exact_tag)::value>(wpre, g, rds[CW * s + jj], t, e, sr);
        const float2 ne2 = make_float2(-e, -e), wp2 = make_float2(wpre, wpre);
        (void)wp2;
        constexpr int V0 = (u + 1) / 2;
        constexpr int SH = u == PUB - 1 ? PUB / 2 : 0;
#pragma unroll
        for (int v = V0; v < N; ++v) {
            float2 x = __ffma2_rn(ne2, *reinterpret_cast<const float2*>(rr + 2 * v), w[v]);
            if constexpr (HASP) x = __ffma2_rn(wp2, *reinterpret_cast<const float2*>(pt + jj * CW + 2 * v), x);
            w[v - SH] = x;
        }
    };
    auto columns = [&](auto exact_tag, auto live_tag, int p, float (&e)[PUB], float (&wpre)[PUB], float (&tq)[PUB], StepRange& sr) {
        column(exact_tag, live_tag, std::integral_constant<int, 0>{}, p, e[0], wpre[0], tq[0], sr);
        column(exact_tag, live_tag, std::integral_constant<int, 1>{}, p, e[1], wpre[1], tq[1], sr);
        column(exact_tag, live_tag, std::integral_constant<int, 2>{}, p, e[2], wpre[2], tq[2], sr);
        column(exact_tag, live_tag, std::integral_constant<int, 3>{}, p, e[3], wpre[3], tq[3], sr);
    };
    static_assert(PUB == 4, "columns() writes out the 4 columns of a turn");
    const float czero = __fadd_rn(g.zero, 8388608.0f);   // t + czero = 2^23 + code
#pragma unroll 1
    for (int p = 0; p < CW / PUB; ++p) {
        float e[PUB], wpre[PUB], tq[PUB];
        StepRange sr;
        // the columns left, in their own (not yet published) rows of the exchange tile
#pragma unroll
        for (int t = 0; t < CW / 2; ++t)
            if (PUB * p + 2 * t < CW) {
                xt[(PUB * p + 2 * t) * ELD + lane] = w[t].x;
                xt[(PUB * p + 2 * t + 1) * ELD + lane] = w[t].y;
            }
        if (p < CW / PUB / 2)
            columns(std::false_type{}, std::integral_constant<int, CW / 2>{}, p, e, wpre, tq, sr);
        else
            columns(std::false_type{}, std::integral_constant<int, CW / 4>{}, p, e, wpre, tq, sr);
        uint32_t word = 0u;
        if (__builtin_expect(sr.ok() & fast, 1)) {
            uint32_t cb[PUB];
#pragma unroll
            for (int u = 0; u < PUB; ++u) {
                xt[(PUB * p + u) * ELD + lane] = e[u];
                if constexpr (HASP) Qs[s * XT + (PUB * p + u) * ELD + lane] = wpre[u];
                cb[u] = __float_as_uint(__fadd_rn(tq[u], czero));
            }
            word = __byte_perm(__byte_perm(cb[0], cb[1], 0x0040), __byte_perm(cb[2], cb[3], 0x0040), 0x5410);
            if (want_pre) {
#pragma unroll
                for (int u = 0; u < PUB; ++u)
                    if (KQ_IN_RANGE(r * d_in + c0 + PUB * p + u, d_out * d_in)) pre_q[r * d_in + c0 + PUB * p + u] = wpre[u];
            }
        } else {   // an operand outside the fast division's range (or past the end): these columns again,
                   // with IEEE divisions
#pragma unroll
            for (int t = 0; t < CW / 2; ++t)
                if (PUB * p + 2 * t < CW)
                    w[t] = make_float2(xt[(PUB * p + 2 * t) * ELD + lane], xt[(PUB * p + 2 * t + 1) * ELD + lane]);
            columns(std::true_type{}, std::integral_constant<int, CW / 2>{}, p, e, wpre, tq, sr);
#pragma unroll
            for (int u = 0; u < PUB; ++u) {
                const int jj = PUB * p + u;
                xt[jj * ELD + lane] = e[u];
                if constexpr (HASP) Qs[s * XT + jj * ELD + lane] = wpre[u];
                word |= (__float_as_uint(__fadd_rn(tq[u], czero)) & 255u) << (8 * u);
                finite = finite & ((fabsf(wpre[u]) <= 3.402823466e38f) | (CW * s + jj >= nb));
                if (want_pre && c0 + jj < cend && KQ_IN_RANGE(r * d_in + c0 + jj, d_out * d_in)) pre_q[r * d_in + c0 + jj] = wpre[u];
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&pub[s * (CW / PUB) + p]);
#pragma unroll
        for (int v = 0; v + 1 < CW / PUB; ++v) cq[v] = cq[v + 1];
        cq[CW / PUB - 1] = word;
    }
    if (!__all_sync(0xffffffffu, finite) && lane == 0) record_error(info, -KQ_ERR_NONFINITE);
    if (live && KQ_IN_RANGE(r * d_in + (c0 + CW <= cend ? c0 + CW : cend) - 1, d_out * d_in)) {
        uint8_t* cp = codes + r * d_in + c0;
        if (VEC && c0 + CW <= cend) {
            *reinterpret_cast<uint4*>(cp) = make_uint4(cq[0], cq[1], cq[2], cq[3]);
        } else {
#pragma unroll
            for (int t = 0; t < CW; ++t)
                if (c0 + t < cend) cp[t] = static_cast<uint8_t>(cq[t >> 2] >> (8 * (t & 3)));
        }
    }
    // E (and its tf32 split, and -Wpre) row by row from the exchange tile.
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int64_t rr = row0 + 8 * it + qr;
        float v[4], h[4], l[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = xt[(qc + u) * ELD + 8 * it + qr];
        store_quad<VEC>(E, rr, d_out, d_in, c0 + qc, cend, v);
        if (Eh) {   // tensor-core trailing update: E = E_hi + E_lo
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                h[u] = tf32_hi(v[u]);
                l[u] = v[u] - h[u];
            }
            store_quad<VEC>(Eh, rr, d_out, d_in, c0 + qc, cend, h);
            store_quad<VEC>(El, rr, d_out, d_in, c0 + qc, cend, l);
        }
        if constexpr (HASP) {   // -Wpre of the block, for the trailing update
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = -Qs[s * XT + (qc + u) * ELD + 8 * it + qr];
            if (Qh) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    h[u] = tf32_hi(v[u]);
                    l[u] = v[u] - h[u];
                }
                store_quad<VEC>(Qh, rr, d_out, d_in, c0 + qc, cend, h);
                store_quad<VEC>(Ql, rr, d_out, d_in, c0 + qc, cend, l);
            } else {
                store_quad<VEC>(Q, rr, d_out, d_in, c0 + qc, cend, v);
            }
        }
    }
}

// W[:, cb:ce] -= E[:, i0:i0+kb] R[i0:i0+kb, cb:ce] with R[k][c] = Lt[c][k]: 128 x 128 output
// tiles of the shared tile GEMM (acc = fma(E_k, R_kc, acc) over ascending k), then w = w - acc.
// With P (Q = -Wpre, P[k][c] = Pt[c][k]) the sum continues with acc = fma(Q_k, P_kc, acc).
template <bool VEC>
__global__ void __launch_bounds__(G_THREADS, 2) trailing_kernel(float* __restrict__ W, const float* __restrict__ E,
                                                                const float* __restrict__ Lt, int64_t d_out,
                                                                int64_t d_in, int64_t i0, int kb, int64_t cb,
                                                                int64_t ce, const float* __restrict__ Q,
                                                                const float* __restrict__ Pt) {
    extern __shared__ __align__(16) float sm[];
    const int64_t r0 = static_cast<int64_t>(blockIdx.y) * GT;
    const int64_t c0 = cb + static_cast<int64_t>(blockIdx.x) * GT;
    const int arows = static_cast<int>(min(static_cast<int64_t>(GT), d_out - r0));
    const int bcols = static_cast<int>(min(static_cast<int64_t>(GT), ce - c0));
    float acc[8][8];
    gemm_tile<false, VEC>(E + r0 * d_in + i0, d_in, arows, Lt + c0 * d_in + i0, d_in, bcols, kb, acc, sm);
    if (Pt) gemm_tile<false, VEC, false>(Q + r0 * d_in + i0, d_in, arows, Pt + c0 * d_in + i0, d_in, bcols, kb, acc, sm);
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    // Read-modify-write of W in two halves of 32 values, all loads of a half issued before
    // its stores, so the memory latency is paid twice rather than 64 times.
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float wv[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int rr = gt_row(ty, 4 * h + i), cc = gt_col<false>(tx, j);
                wv[i][j] = (rr < arows && cc < bcols) ? W[(r0 + rr) * d_in + c0 + cc] : 0.0f;
            }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int rr = gt_row(ty, 4 * h + i), cc = gt_col<false>(tx, j);
                if (rr < arows && cc < bcols && KQ_IN_RANGE((r0 + rr) * d_in + c0 + cc, d_out * d_in))
                    W[(r0 + rr) * d_in + c0 + cc] = __fsub_rn(wv[i][j], acc[4 * h + i][j]);
            }
    }
}

// col_loss[j] = sum over rows of E[r][j]^2 in a fixed order (fp32 runs, fp64 across them).
// Block (CS_X, CS_Y).
template <int PER_SM>
__global__ void __launch_bounds__(CS_X * CS_Y, PER_SM) colloss_kernel(const float* __restrict__ E, int64_t d_out, int64_t d_in,
                                                                      float* __restrict__ col_loss) {
    const int64_t j = static_cast<int64_t>(blockIdx.x) * CS_X + threadIdx.x;
    const double a = col_sumsq(E, d_out, d_in, j);
    if (threadIdx.y == 0 && j < d_in && KQ_IN_RANGE(j, d_in)) col_loss[j] = static_cast<float>(a);
}

struct ObsWs {
    float* Rp;      // packed diagonal blocks of R, nblk x BLK x BLK
    float* Rq;      // packed blocks of R right of them (block b: rows of b, columns of b + 1)
    float* E;       // d_out x d_in
    float* gscale;  // d_out
    float* gzero;   // d_out
    float* Eh;      // tensor-core mode: E_hi, E_lo [d_out x d_in], Lt_hi, Lt_lo [d_in x d_in]
    float* El;
    float* Lh;
    float* Ll;
    float* Pp;      // with P: packed diagonal blocks of P; -Wpre [d_out x d_in] (fp32 mode)
    float* Q;
    float* Qh;      // with P, tensor-core mode: (-Wpre)_hi, _lo [d_out x d_in], Pt_hi, Pt_lo
    float* Ql;
    float* Ph;
    float* Pl;
};

inline size_t align256(size_t b) { return (b + 255) & ~static_cast<size_t>(255); }

size_t ws_base_bytes(int64_t d_out, int64_t d_in) {
    return align256((2 * static_cast<size_t>(cdiv(d_in, BLK)) * BLK * BLK + static_cast<size_t>(d_out) * d_in +
                     2 * static_cast<size_t>(d_out)) * sizeof(float));
}

// Byte sizes of the parts in carve order.
struct WsParts {
    size_t base, blk, wide, sq;
};
WsParts parts_of(int64_t d_out, int64_t d_in) {
    WsParts p;
    p.base = ws_base_bytes(d_out, d_in);
    p.blk = align256(static_cast<size_t>(cdiv(d_in, BLK)) * BLK * BLK * sizeof(float));
    p.wide = align256(static_cast<size_t>(d_out) * d_in * sizeof(float));
    p.sq = align256(static_cast<size_t>(d_in) * d_in * sizeof(float));
    return p;
}

size_t ws_bytes_of(int64_t d_out, int64_t d_in, int mode, bool with_p) {
    const WsParts p = parts_of(d_out, d_in);
    const bool tc = mode == KQ_TRAIL_3XTF32;
    size_t b = p.base;
    if (tc) b += 2 * p.wide + 2 * p.sq;
    if (with_p) b += p.blk + (tc ? 2 * p.wide + 2 * p.sq : p.wide);
    return b + 256;
}

ObsWs carve(void* ws, int64_t d_out, int64_t d_in, int mode, bool with_p) {
    const WsParts sz = parts_of(d_out, d_in);
    const bool tc = mode == KQ_TRAIL_3XTF32;
    ObsWs o;
    o.Rp = static_cast<float*>(ws);
    o.Rq = o.Rp + cdiv(d_in, BLK) * BLK * BLK;
    o.E = o.Rq + cdiv(d_in, BLK) * BLK * BLK;
    o.gscale = o.E + d_out * d_in;
    o.gzero = o.gscale + d_out;
    o.Eh = o.El = o.Lh = o.Ll = o.Pp = o.Q = o.Qh = o.Ql = o.Ph = o.Pl = nullptr;
    uint8_t* p = static_cast<uint8_t*>(ws) + sz.base;
    auto take = [&](size_t bytes) {
        float* f = reinterpret_cast<float*>(p);
        p += bytes;
        return f;
    };
    if (tc) {
        o.Eh = take(sz.wide);
        o.El = take(sz.wide);
        o.Lh = take(sz.sq);
        o.Ll = take(sz.sq);
    }
    if (with_p) {
        o.Pp = take(sz.blk);
        if (tc) {
            o.Qh = take(sz.wide);
            o.Ql = take(sz.wide);
            o.Ph = take(sz.sq);
            o.Pl = take(sz.sq);
        } else {
            o.Q = take(sz.wide);
        }
    }
    return o;
}

}  // namespace

KQ_DEBUG_UNIT(obs)
}  // namespace kq

using namespace kq;

extern "C" size_t kq_obs_quantize_workspace(int64_t d_out, int64_t d_in, int block, int mode, int with_p) {
    (void)block;
    if (d_out < 1 || d_in < 1 || (mode != KQ_TRAIL_FP32 && mode != KQ_TRAIL_3XTF32)) return 0;
    return ws_bytes_of(d_out, d_in, mode, with_p != 0);
}

extern "C" kq_status kq_obs_quantize(float* W, int64_t d_out, int64_t d_in, const float* Lt, const float* Pt,
                                     int bits, int group, int block, int mode, uint8_t* codes, float* scale,
                                     int32_t* zero, float* col_loss, float* pre_q, int* info, void* ws,
                                     size_t ws_bytes, kq_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (!W || !Lt || !codes || !scale || !zero || d_out < 1 || d_in < 1 || bits < 1 || bits > 8) {
        set_error("kq_obs_quantize: invalid arguments");
        return KQ_ERR_INVALID_ARG;
    }
    if (block != BLK || (group != 0 && group != block)) {
        set_error("kq_obs_quantize: block must be %d and group 0 or equal to block", BLK);
        return KQ_ERR_UNSUPPORTED;
    }
    if (mode != KQ_TRAIL_FP32 && mode != KQ_TRAIL_3XTF32) {
        set_error("kq_obs_quantize: unknown trailing-update mode %d", mode);
        return KQ_ERR_INVALID_ARG;
    }
    const bool tc = mode == KQ_TRAIL_3XTF32;
    const bool hp = Pt != nullptr;
    if (tc && ((d_in % 4) != 0 || (reinterpret_cast<uintptr_t>(W) & 15u) != 0)) {
        set_error("kq_obs_quantize: the tensor-core trailing update needs d_in %% 4 == 0 and a 16-byte aligned W");
        return KQ_ERR_UNSUPPORTED;
    }
    if (hp && ((d_in % 16) != 0 || (reinterpret_cast<uintptr_t>(W) & 15u) || (reinterpret_cast<uintptr_t>(codes) & 15u) ||
               (reinterpret_cast<uintptr_t>(Pt) & 15u))) {
        set_error("kq_obs_quantize: the drift correction needs d_in %% 16 == 0 and 16-byte aligned W, codes, Pt");
        return KQ_ERR_UNSUPPORTED;
    }
    if (!ws || ws_bytes < ws_bytes_of(d_out, d_in, mode, hp) || (reinterpret_cast<uintptr_t>(ws) & 255u)) {
        set_error("kq_obs_quantize: workspace must be 256-byte aligned and hold %zu bytes",
                  ws_bytes_of(d_out, d_in, mode, hp));
        return KQ_ERR_WORKSPACE;
    }
    static std::atomic<uint64_t> attr{0};
    KQ_TRY(once_per_device(attr, [&]() -> kq_status {
        // The whole shared memory of the SM, so that a CTA fits beside a far-update CTA.
        auto block_attr = [](auto* kern, bool with_p) -> kq_status {
            KQ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, obs_smem(with_p)));
            KQ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         cudaSharedmemCarveoutMaxShared));
            return KQ_OK;
        };
        KQ_TRY(block_attr(obs_block_kernel<true, false, FUSE_NONE>, false));
        KQ_TRY(block_attr(obs_block_kernel<true, false, FUSE_NONE, 3>, false));
        KQ_TRY(block_attr(obs_block_kernel<true, false, FUSE_FP32>, false));
        KQ_TRY(block_attr(obs_block_kernel<true, false, FUSE_MMA>, false));
        KQ_TRY(block_attr(obs_block_kernel<false, false, FUSE_NONE>, false));
        KQ_TRY(block_attr(obs_block_kernel<false, false, FUSE_FP32>, false));
        KQ_TRY(block_attr(obs_block_kernel<true, true, FUSE_NONE>, true));
        KQ_CUDA(cudaFuncSetAttribute(trailing_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(G_SMEM)));
        KQ_CUDA(cudaFuncSetAttribute(trailing_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(G_SMEM)));
        return KQ_OK;
    }));
    ObsWs o = carve(ws, d_out, d_in, mode, hp);
    TrailMaps maps;
    if (group == 0) {
        rowgrid_kernel<<<static_cast<unsigned>(cdiv(d_out, 8)), 256, 0, stream>>>(W, d_out, d_in, bits, scale,
                                                                                zero, o.gscale, o.gzero);
        KQ_LAUNCH_CHECK("rowgrid_kernel");
    }
    const bool vec = (d_in % 4 == 0) && (reinterpret_cast<uintptr_t>(Lt) % 16 == 0);
    const bool bvec = (d_in % 16 == 0) && (reinterpret_cast<uintptr_t>(W) % 16 == 0) &&
                      (reinterpret_cast<uintptr_t>(codes) % 16 == 0);
    const int64_t nblk = cdiv(d_in, BLK);
    const int64_t row_ctas = cdiv(d_out, OBS_ROWS);
    // the blocks of R right of the diagonal ones, for the fused update: as mma.sync fragments in
    // the 3xTF32 mode, as rows otherwise
    const bool fuse_ok = !hp && nblk > 1 && row_ctas <= static_cast<int64_t>(num_sms()) &&
                         d_out * d_in <= (int64_t{24} << 20);
    const bool mma_fused = fuse_ok && tc && bvec;
    {
        const dim3 pgrid(RTILES + (fuse_ok ? NWARP : 0), static_cast<unsigned>(nblk));
        if (mma_fused)
            pack_r_kernel<PACK_FRAG><<<pgrid, 256, 0, stream>>>(Lt, d_in, o.Rp, o.Rq);
        else if (fuse_ok)
            pack_r_kernel<PACK_ROWS><<<pgrid, 256, 0, stream>>>(Lt, d_in, o.Rp, o.Rq);
        else
            pack_r_kernel<PACK_NONE><<<pgrid, 256, 0, stream>>>(Lt, d_in, o.Rp, nullptr);
        KQ_LAUNCH_CHECK("pack_r_kernel");
    }
    // L split for the trailing updates, unless there are none: one block, or two with the fused update
    if (tc && nblk > (fuse_ok ? 2 : 1)) {
        kq_status st0 = split_tf32(Lt, d_in * d_in, o.Lh, o.Ll, stream);
        if (st0 != KQ_OK) return st0;
        if ((st0 = maps.init(o.Eh, o.El, o.Lh, o.Ll, d_out, d_in)) != KQ_OK) return st0;
        if ((st0 = maps.set_w(W, d_out, d_in)) != KQ_OK) return st0;
        if (hp) {
            if ((st0 = split_tf32(Pt, d_in * d_in, o.Ph, o.Pl, stream)) != KQ_OK) return st0;
            if ((st0 = maps.init_p(o.Qh, o.Ql, o.Ph, o.Pl, d_out, d_in)) != KQ_OK) return st0;
        }
    }
    if (hp) {   // P[i0 + j][i0 + c] = Pt[i0 + c][i0 + j]: the same packing as R from Lt
        pack_r_kernel<PACK_NONE><<<dim3(RTILES, static_cast<unsigned>(nblk)), 256, 0, stream>>>(Pt, d_in, o.Pp, nullptr);
        KQ_LAUNCH_CHECK("pack_r_kernel");
    }
    // GPTQ mode: block b's kernel first applies the previous block's update of its own
    // columns (E_{b-1} R_{b-1,b}, fused), and the update of the columns beyond block b + 1
    // runs on a library side stream beside block b + 1, whose CTAs share the SMs with it.
    // Block b waits only for the far update of block b - 2 (the last one that writes its
    // columns); the two far-update events alternate. With P: after block b the update of
    // block column b + 1 runs on the caller's stream (the next block kernel waits for it),
    // the columns beyond on the side stream beside block b + 1.
    // Every column receives the block updates in block order either way. The fused update
    // is fp32 in the trailing update's order in the fp32 mode, and on the tensor cores
    // (mma.sync, 3xTF32) in the 3xTF32 mode, like the far updates there.
    SideStream* side = nblk > 2 ? side_stream(stream) : nullptr;
    bool forked = false;
    bool far_pending[2] = {false, false};
    // 128 x 64 far-update tiles (a CTA fits beside a block-kernel CTA) while the block kernel
    // runs one CTA per SM and the far updates take about as long as the block kernels
    // (their mean, ~d_out d_in / 2 multiply-adds per block, against ~35 us a block: up to
    // d_out d_in ~ 24M). Otherwise nothing fits beside the block kernel, or the sweep waits
    // on the far updates, and 128 x 128 tiles are faster.
    const bool narrow = !hp && row_ctas <= static_cast<int64_t>(num_sms()) && d_out * d_in <= (int64_t{24} << 20);
    // The previous block's update fused into the block kernel: only then, so that nothing
    // but the far update shares the SMs with the block kernel.
    const bool fuse = narrow;
    auto trailing = [&](int64_t i0, int kb, int64_t cb, int64_t ce, cudaStream_t st) -> kq_status {
        if (tc) return trail_tc(maps, W, d_out, d_in, i0, cb, ce, hp, narrow, kb, info, st);
        dim3 grid(static_cast<unsigned>(cdiv(ce - cb, GT)), static_cast<unsigned>(cdiv(d_out, GT)));
        if (vec)
            trailing_kernel<true><<<grid, G_THREADS, G_SMEM, st>>>(W, o.E, Lt, d_out, d_in, i0, kb, cb, ce, o.Q, Pt);
        else
            trailing_kernel<false><<<grid, G_THREADS, G_SMEM, st>>>(W, o.E, Lt, d_out, d_in, i0, kb, cb, ce, o.Q, Pt);
        KQ_LAUNCH_CHECK("trailing_kernel");
        return KQ_OK;
    };
    // `after_kernel`: the call before this one on the stream was a block kernel or a trailing
    // update, and nothing was waited for in between. The kernel is then launched as its
    // programmatic dependent: it stages R (packed before that kernel began) while the other
    // drains. A block kernel lets its own dependent start only after its own wait, so
    // everything before the kernel it depends on has finished.
    auto block_launch = [&](int64_t b, const float* rq, bool after_kernel) -> kq_status {
        auto go = [&](auto* kern) -> kq_status {
            KQ_CUDA(launch_dependent(kern, dim3(static_cast<unsigned>(row_ctas)), dim3(OBS_THREADS), obs_smem(hp), stream, 1u,
                                     after_kernel, W, d_out, d_in, o.Rp + b * RPACK, b * BLK, bits, group, o.gscale, o.gzero,
                                     codes, scale, zero, o.E, pre_q, o.Eh, o.El, hp ? o.Pp + b * RPACK : nullptr, o.Q, o.Qh,
                                     o.Ql, rq, info));
            KQ_LAUNCH_CHECK("obs_block_kernel");
            return KQ_OK;
        };
        if (hp) return go(obs_block_kernel<true, true, FUSE_NONE>);
        // three CTAs per SM (80 registers, some 30 % more cycles a column) once two do not hold every row
        if (!rq && bvec && row_ctas > 2 * static_cast<int64_t>(num_sms())) return go(obs_block_kernel<true, false, FUSE_NONE, 3>);
        if (!rq) return bvec ? go(obs_block_kernel<true, false, FUSE_NONE>) : go(obs_block_kernel<false, false, FUSE_NONE>);
        if (mma_fused) return go(obs_block_kernel<true, false, FUSE_MMA>);
        return bvec ? go(obs_block_kernel<true, false, FUSE_FP32>) : go(obs_block_kernel<false, false, FUSE_FP32>);
    };
    // Two levels for the large layers on the tensor cores (super-panels of SPB blocks, the
    // GPTQ lazy update grouped once more): inside a super-panel each block updates the next
    // block column on the caller's stream and the rest of the super-panel's columns on the
    // side stream (K = 128); after a super-panel's last block one update with the whole
    // super-panel's K covers every column beyond it -- the next super-panel's columns on the
    // caller's stream, the rest on the second side stream beside the next super-panel's
    // blocks -- so each W tile beyond is read and written once per super-panel instead of
    // once per block. Every column still receives the block updates in block order (the
    // long update drains its accumulator into W one block's K at a time).
    const bool two_level = tc && !hp && !fuse && nblk > SPB;
    if (two_level) {
        constexpr int64_t SPW = static_cast<int64_t>(SPB) * BLK;
        bool in_pending = false;    // the in-panel update of the previous block (side stream)
        bool far_pending = false;   // the far update of the previous super-panel (second side stream)
        cudaStream_t s_in = side ? side->s : stream;
        cudaStream_t s_far = side ? side->s2 : stream;
        for (int64_t b = 0; b < nblk; ++b) {
            const int64_t i0 = b * BLK;
            kq_status st = block_launch(b, nullptr, b > 0);
            if (st != KQ_OK) return st;
            const int64_t nb0 = i0 + BLK;                               // next block column
            if (nb0 >= d_in) break;
            const int64_t sp0 = (b / SPB) * SPW;                         // this super-panel
            const int64_t spe = std::min(d_in, sp0 + SPW);
            if (side) KQ_CUDA(cudaEventRecord(side->ev[0], stream));     // E of this block ready
            if (nb0 < spe) {
                if (in_pending) {   // it wrote the next block column too
                    KQ_CUDA(cudaStreamWaitEvent(stream, side->ev[1], 0));
                    in_pending = false;
                }
                const int64_t nb1 = std::min(spe, nb0 + BLK);
                st = trailing(i0, BLK, nb0, nb1, stream);
                if (st != KQ_OK) return st;
                if (nb1 < spe) {
                    if (side) KQ_CUDA(cudaStreamWaitEvent(s_in, side->ev[0], 0));
                    st = trailing(i0, BLK, nb1, spe, s_in);
                    if (st != KQ_OK) return st;
                    if (side) {
                        KQ_CUDA(cudaEventRecord(side->ev[1], s_in));
                        in_pending = true;
                    }
                }
            } else {
                const int64_t sp1 = std::min(d_in, spe + SPW);           // the next super-panel's end
                if (far_pending) {   // the previous super-panel's far update wrote these columns
                    KQ_CUDA(cudaStreamWaitEvent(stream, side->ev2[0], 0));
                    far_pending = false;
                }
                st = trail_tc_long(maps, d_out, d_in, sp0, static_cast<int>(spe - sp0), spe, sp1, info, stream);
                if (st != KQ_OK) return st;
                if (sp1 < d_in) {
                    if (side) KQ_CUDA(cudaStreamWaitEvent(s_far, side->ev[0], 0));
                    st = trail_tc_long(maps, d_out, d_in, sp0, static_cast<int>(spe - sp0), sp1, d_in, info, s_far);
                    if (st != KQ_OK) return st;
                    if (side) {
                        KQ_CUDA(cudaEventRecord(side->ev2[0], s_far));
                        far_pending = true;
                    }
                }
            }
        }
        if (in_pending) KQ_CUDA(cudaStreamWaitEvent(stream, side->ev[1], 0));
        if (far_pending) KQ_CUDA(cudaStreamWaitEvent(stream, side->ev2[0], 0));
    } else if (fuse && tc) {
        // Pairs of blocks (2s, 2s + 1). Block 2s + 1 applies block 2s's update of its columns
        // itself; after the pair, its update (K = 256, still applied 128 of K at a time) of
        // the next pair's columns runs on the caller's stream just before the next pair,
        // and that of the columns beyond on the side stream beside the next pair. The
        // next-pair update waits for the side update of the pair before (it wrote the same
        // columns); the side updates alternate two events.
        bool rest_pending[2] = {false, false};
        for (int64_t b = 0; b < nblk; ++b) {
            const int64_t i0 = b * BLK;
            const int64_t pr = b / 2;
            kq_status st;
            if ((b & 1) == 0 && b >= 2) {
                if (rest_pending[pr & 1]) {   // the side update of pair pr - 2
                    KQ_CUDA(cudaStreamWaitEvent(stream, side->ev2[pr & 1], 0));
                    rest_pending[pr & 1] = false;
                }
                st = trailing(i0 - 2 * BLK, 2 * BLK, i0, std::min<int64_t>(d_in, i0 + 2 * BLK), stream);
                if (st != KQ_OK) return st;
            }
            st = block_launch(b, (b & 1) ? o.Rq + (b - 1) * BLK * BLK : nullptr, b > 0);
            if (st != KQ_OK) return st;
            if ((b & 1) == 0) continue;
            const int64_t nb2 = std::min<int64_t>(d_in, i0 + 3 * BLK);   // beyond the next pair
            if (nb2 >= d_in) continue;
            cudaStream_t fs = stream;
            if (side) {
                KQ_CUDA(cudaEventRecord(side->ev[0], stream));   // E of the pair ready
                KQ_CUDA(cudaStreamWaitEvent(side->s, side->ev[0], 0));
                fs = side->s;
            }
            st = trailing(i0 - BLK, 2 * BLK, nb2, d_in, fs);
            if (st != KQ_OK) return st;
            if (side) {
                KQ_CUDA(cudaEventRecord(side->ev2[pr & 1], side->s));
                rest_pending[pr & 1] = true;
            }
        }
        for (int q = 0; q < 2; ++q)
            if (rest_pending[q]) KQ_CUDA(cudaStreamWaitEvent(stream, side->ev2[q], 0));
    } else {
        for (int64_t i0 = 0; i0 < d_in; i0 += BLK) {
            const int64_t b = i0 / BLK;
            const int kb = static_cast<int>(std::min<int64_t>(BLK, d_in - i0));
            const float* rq = fuse && b > 0 ? o.Rq + (b - 1) * BLK * BLK : nullptr;
            const bool waits = fuse && far_pending[b & 1];
            if (waits) {   // the far update of block b - 2
                KQ_CUDA(cudaStreamWaitEvent(stream, side->ev2[b & 1], 0));
                far_pending[b & 1] = false;
            }
            kq_status st = block_launch(b, rq, b > 0 && !waits);
            if (st != KQ_OK) return st;
            const int64_t nb0 = i0 + kb;                                // next block column
            if (nb0 >= d_in) break;
            const int64_t nb1 = std::min<int64_t>(d_in, nb0 + BLK);    // columns beyond it: [nb1, d_in)
            const bool fork = side && nb1 < d_in;
            if (fork) KQ_CUDA(cudaEventRecord(side->ev[0], stream));           // E of this block ready
            if (!fuse) {
                if (forked) KQ_CUDA(cudaStreamWaitEvent(stream, side->ev[1], 0));  // previous far update done
                st = trailing(i0, kb, nb0, nb1, stream);
                if (st != KQ_OK) return st;
            }
            if (nb1 < d_in) {
                cudaStream_t fs = stream;
                if (fork) {
                    KQ_CUDA(cudaStreamWaitEvent(side->s, side->ev[0], 0));
                    fs = side->s;
                }
                st = trailing(i0, kb, nb1, d_in, fs);
                if (st != KQ_OK) return st;
                if (fork) {
                    KQ_CUDA(cudaEventRecord(fuse ? side->ev2[b & 1] : side->ev[1], side->s));
                    if (fuse)
                        far_pending[b & 1] = true;
                    else
                        forked = true;
                }
            }
        }
        for (int q = 0; q < 2; ++q)
            if (far_pending[q]) KQ_CUDA(cudaStreamWaitEvent(stream, side->ev2[q], 0));
    }
    if (forked) KQ_CUDA(cudaStreamWaitEvent(stream, side->ev[1], 0));
    if (col_loss) {
        auto* kern = cs_per_sm(d_in) == 2 ? colloss_kernel<2> : colloss_kernel<1>;
        kern<<<static_cast<unsigned>(cdiv(d_in, CS_X)), dim3(CS_X, CS_Y), 0, stream>>>(o.E, d_out, d_in, col_loss);
        KQ_LAUNCH_CHECK("colloss_kernel");
    }
    return KQ_OK;
}
