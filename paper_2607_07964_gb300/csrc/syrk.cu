// Stage 1: Kronecker-factor accumulation H (+)= A^T A on the 5th-generation tensor cores.
//
// Paper: Sec. 2.1 Eq. (ptq_obj) (H_X = X X^T, tokens as columns there), Sec. 3.1 Eq. (kfac)
// (H = H_X (x) H_G), Algorithm 1 ("online statistics"). Tokens are rows here, so the
// factor is A^T A for A [T x d].
//
// Design (sm_103a):
//   * one CTA per 128 x 256 output tile of the lower triangle (row tile i, column tile j,
//     128 i + 127 >= 256 j); the tile is mirrored into the upper triangle on write-out;
//   * warp 0 issues TMA loads of 64-token x 64-feature boxes (128-byte swizzle) into a
//     4-stage ring; both operands are slices of the same A, read MN-major (features
//     contiguous), so no transpose pass is needed;
//   * warp 1 allocates 512 TMEM columns and issues tcgen05.mma kind::f16 (bf16 x bf16 ->
//     fp32, M = 128, N = 256, K = 16) into one of two 256-column accumulators;
//   * warps 2..9 drain an accumulator every KQ_SYRK_CHUNK_TOKENS tokens into an fp32
//     running sum held in registers (each thread owns 128 columns of one row), while the
//     MMAs continue into the other accumulator. This bounds how many tensor-core
//     additions any fp32 partial sum sees;
//   * a factor with few tiles (a narrow d) leaves most SMs idle: a cluster of KS = 4 CTAs then
//     shares each tile, CTA r taking the token chunks r, r + KS, ... and owning 128 / KS rows of
//     the running sum. Each drained chunk goes to the owners' inboxes through distributed
//     shared memory, and the owners add the chunks in token order, so H has the bits one CTA
//     would give it. d = 1024, T = 262144 (20 tiles): 1384 -> 1047 us; d = 1400, T = 131072: 1134
//     -> 620 us. What bounds it then is the exchange (~4 us a half tile: remote stores, their
//     release, the owner's answer), so quarter tiles in two slots (1470 us) and clusters of two
//     (d = 2048: 1597 against 1386 us) were slower. Splitting the columns instead (64 per CTA,
//     the row panel multicast) took 1217 us at d = 1024: a CTA's time per 64 tokens is then bound
//     by the bytes into its SM (50-70 per cycle) and the row operand, not by N;
//   * every mbarrier wait is bounded (kq::mbar_wait); a timeout is reported as
//     -KQ_ERR_TIMEOUT in *info and the CTA drains its own copies and MMAs before exit.
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "kq_common.cuh"
#include "trail_tc.cuh"

namespace kq {
namespace {

constexpr int BM = 128;   // output rows per tile (MMA M, TMEM lanes)
constexpr int BN = 256;   // output columns per tile (MMA N)
constexpr int BK = 64;    // tokens per pipeline stage
constexpr int BOX_BYTES = BK * 64 * 2;          // one 64-token x 64-feature bf16 box
constexpr int A_BYTES = BK * BM * 2;            // 16 KB
constexpr int B_BYTES = BK * BN * 2;            // 32 KB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;  // 48 KB
constexpr int NUM_THREADS = 320;                // 10 warps
// Ring stages of a CTA, and its inbox when KS CTAs share a tile: per source CTA 128 / KS rows x 128
// columns (half a tile at a time), 64 KB in all.
__host__ __device__ constexpr int stages_of(int ks) { return ks == 1 ? 4 : 3; }
constexpr int INBOX_BYTES = BM * 128 * 4;
constexpr int smem_bytes(int ks) { return stages_of(ks) * STAGE_BYTES + (ks == 1 ? 0 : INBOX_BYTES) + 1024 + 256; }
constexpr uint32_t TMEM_COLS = 512;
// Canonical MN-major SW128 layout: atoms of 64 features x 8 tokens (1 KB). Along the MN
// dimension atoms are one TMA box apart; along K they are 1 KB apart.
constexpr uint32_t LBO = BOX_BYTES;   // next 64 features
constexpr uint32_t SBO = 1024;        // next 8 tokens

// Tile order of the lower triangle (tile (i, j) needs i >= 2 j): bands of BAND column tiles,
// each band row by row, BAND tiles per row once past the diagonal. The CTAs resident at
// one time (about one per SM) then cover ~19 row panels x 8 column panels, i.e. ~4.5k of
// the d features, instead of one column panel and ~150 row panels (~20k features): every
// resident set streams all T tokens of its features from HBM, so this is what keeps a
// large factor (d = 14336, 28672) from re-reading X several times over.
constexpr int BAND = 8;
// Tiles of a band's first r rows past its start (row k of the band holds min(w, k / 2 + 1)).
__host__ __device__ constexpr int band_tiles(int r, int w) {
    return r <= 2 * w ? (r / 2) * (r / 2 + 1) + (r & 1) * (r / 2 + 1) : w * (w + 1) + (r - 2 * w) * w;
}
__device__ __forceinline__ void tile_of(int bid, int n_row_tiles, int n_col_tiles, int* ti, int* tj) {
    for (int j0 = 0; j0 < n_col_tiles; j0 += BAND) {
        const int w = min(BAND, n_col_tiles - j0);
        const int rows = n_row_tiles - 2 * j0;
        const int cnt = band_tiles(rows, w);
        if (bid >= cnt) {
            bid -= cnt;
            continue;
        }
        int k = 0;
        if (bid >= w * (w + 1) && rows > 2 * w) {   // past the triangle: w tiles a row
            k = 2 * w + (bid - w * (w + 1)) / w;
            bid = (bid - w * (w + 1)) % w;
        } else {
            while (bid >= min(w, k / 2 + 1)) bid -= min(w, k++ / 2 + 1);
        }
        *ti = 2 * j0 + k;
        *tj = j0 + bid;
        return;
    }
    *ti = 0;   // not reached for bid < the number of lower tiles
    *tj = 0;
}

__device__ __forceinline__ bool wait_noabort(uint64_t* bar, uint32_t parity) {
    int dummy = 0;
    return mbar_wait(bar, parity, &dummy);
}

__device__ __forceinline__ void st_cluster_f4(uint32_t addr, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

// The body shared by the two Gram products.
//   CROSS = false (SYRK): H (+)= A^T A, lower 128 x 256 tiles mirrored on write-out; every
//     operand box comes from map a0.
//   CROSS = true: D (+)= (A_hi + A_lo)^T B over all tiles, no symmetry: the K loop runs over
//     the T tokens of the pair (a0 = A_hi, b) and then over the pair (a1 = A_lo, b).
template <bool CROSS, int KS>
__device__ __forceinline__ void gram_tc_body(const CUtensorMap* a0, const CUtensorMap* a1,
                                             const CUtensorMap* bmap, float* __restrict__ H, int d,
                                             int T, int n_row_tiles, int tile0, int chunk_stages, int accumulate,
                                             int* info) {
    constexpr int STAGES = stages_of(KS);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    float* inbox = reinterpret_cast<float*>(smem + STAGES * STAGE_BYTES);   // KS > 1
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES + (KS > 1 ? INBOX_BYTES : 0));
    uint64_t* empty = full + STAGES;
    uint64_t* tfull = empty + STAGES;
    uint64_t* tempty = tfull + 2;
    uint64_t* mma_done = tempty + 2;
    uint64_t* in_full = mma_done + 1;     // [KS] a source's part of the inbox is there
    uint64_t* in_free = in_full + KS;     // [KS] an owner has read this CTA's part of its inbox
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(in_free + KS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int tile = tile0 + static_cast<int>(blockIdx.x) / KS;
    const int rank = KS > 1 ? static_cast<int>(cluster_ctarank()) : 0;
    int ti, tj;
    if (CROSS) {
        ti = tile % n_row_tiles;
        tj = tile / n_row_tiles;
    } else {
        tile_of(tile, n_row_tiles, (d + BN - 1) / BN, &ti, &tj);
    }
    const int i0 = ti * BM;
    const int j0 = tj * BN;
    const int nk1 = (T + BK - 1) / BK;          // stages per pass over the tokens
    const int nk = CROSS ? 2 * nk1 : nk1;
    const int nchunks = (nk + chunk_stages - 1) / chunk_stages;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], 8);
        }
        mbar_init(mma_done, 1);
        for (int r = 0; KS > 1 && r < KS; ++r) {
            mbar_init(&in_full[r], 8 / KS);
            mbar_init(&in_free[r], 8);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, TMEM_COLS);
        tmem_relinquish();
    }
    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(a0);
        if (CROSS) {
            tma_prefetch_desc(a1);
            tma_prefetch_desc(bmap);
        }
    }
    tc_fence_before();
    if constexpr (KS > 1)
        cluster_barrier();   // every CTA's barriers are set up before another one signals them
    else
        __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // This CTA's chunks c = rank, rank + KS, ..., its stages counted by ks (the ring position).

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int issued = 0;
            for (int k = rank * chunk_stages; k < nk; k += (KS > 1 && (k + 1) % chunk_stages == 0) ? (KS - 1) * chunk_stages + 1 : 1) {
                const int s = issued % STAGES;
                const uint32_t u = static_cast<uint32_t>(issued / STAGES);
                if (!mbar_wait(&empty[s], (u & 1u) ^ 1u, abort_flag)) break;
                mbar_arrive_expect_tx(&full[s], STAGE_BYTES);
                uint8_t* a = smem + s * STAGE_BYTES;
                uint8_t* b = a + A_BYTES;
                const bool second = CROSS && k >= nk1;
                const int y = (second ? k - nk1 : k) * BK;
                const CUtensorMap* am = second ? a1 : a0;
                const CUtensorMap* bm = CROSS ? bmap : a0;
                tma_load_2d(a, am, &full[s], i0, y);
                tma_load_2d(a + BOX_BYTES, am, &full[s], i0 + 64, y);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    tma_load_2d(b + q * BOX_BYTES, bm, &full[s], j0 + 64 * q, y);
                ++issued;
            }
            // Drain: every issued load must have landed before the CTA may exit.
            for (int k = (issued > STAGES ? issued - STAGES : 0); k < issued; ++k)
                wait_noabort(&full[k % STAGES], static_cast<uint32_t>(k / STAGES) & 1u);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16_mn_major(BM, BN);
            int k = 0;   // stages of this CTA so far
            bool ok = true;
            for (int c = rank, m = 0; c < nchunks && ok; c += KS, ++m) {
                const int buf = m & 1;
                const uint32_t u = static_cast<uint32_t>(m >> 1);
                if (!mbar_wait(&tempty[buf], (u & 1u) ^ 1u, abort_flag)) break;
                tc_fence_after();
                const uint32_t dt = tmem + static_cast<uint32_t>(buf * BN);
                const int kn = min(nk - c * chunk_stages, chunk_stages);
                for (int kk = 0; kk < kn; ++k, ++kk) {
                    const int s = k % STAGES;
                    if (!mbar_wait(&full[s], static_cast<uint32_t>(k / STAGES) & 1u, abort_flag)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a = smem_u32(smem + s * STAGE_BYTES);
                    const uint32_t b = a + A_BYTES;
#pragma unroll
                    for (int k16 = 0; k16 < BK / 16; ++k16) {
                        const uint64_t ad = smem_desc_sw128(a + k16 * 2048, LBO, SBO);
                        const uint64_t bd = smem_desc_sw128(b + k16 * 2048, LBO, SBO);
                        tc_mma_f16(dt, ad, bd, idesc, (kk > 0 || k16 > 0) ? 1u : 0u);
                    }
                    tc_commit(&empty[s]);
                }
                if (ok) tc_commit(&tfull[buf]);
            }
            // All MMAs must be complete before TMEM is released.
            tc_commit(mma_done);
            wait_noabort(mma_done, 0);
        }
    } else if constexpr (KS == 1) {
        // ------------------------------------------------------------ epilogue (8 warps)
        const int q = warp & 3;                 // TMEM lane quadrant this warp may access
        const int half = (warp - 2) >> 2;       // which 128 of the 256 columns
        const int row = i0 + q * 32 + lane;
        float acc[128];
#pragma unroll
        for (int i = 0; i < 128; ++i) acc[i] = 0.0f;
        bool ok = true;
        for (int c = 0; c < nchunks; ++c) {
            const int buf = c & 1;
            const uint32_t u = static_cast<uint32_t>(c >> 1);
            ok = mbar_wait(&tfull[buf], u & 1u, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint32_t base = tmem + (static_cast<uint32_t>(q * 32) << 16) +
                                  static_cast<uint32_t>(buf * BN + half * 128);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                float v[32];
                tmem_ld32(base + p * 32, v);
                tc_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) acc[p * 32 + i] += v[i];
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[buf]);
        }
        // Write-out through shared memory (the pipeline stages are idle now): each warp stages
        // its 32 rows x 128 columns, then updates the lower tile one 128-byte row segment at a
        // time (coalesced, also for the accumulate read) and writes the mirror from the staged
        // results (lanes on consecutive rows of H^T: coalesced too).
        ok = __all_sync(0xffffffffu, ok && !*abort_flag);
        if (ok) {
            constexpr int SLD = 129;
            float* st = reinterpret_cast<float*>(smem) + (warp - 2) * 32 * SLD;
#pragma unroll
            for (int i = 0; i < 128; ++i) st[lane * SLD + i] = acc[i];
            __syncwarp();
            const int cbase = j0 + half * 128;
            const int rbase = i0 + q * 32;
            // eight rows at a time, so 32 loads per lane are in flight (accumulate mode)
#pragma unroll 1
            for (int r8 = 0; r8 < 32; r8 += 8) {
                float old[8][4];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int rr = rbase + r8 + u;
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const int col = cbase + lane + 32 * m;
                        old[u][m] = (accumulate && rr < d && col < d && (CROSS || col <= rr))
                                        ? H[static_cast<int64_t>(rr) * d + col] : 0.0f;
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int rr = rbase + r8 + u;
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const int col = cbase + lane + 32 * m;
                        if (rr < d && col < d && (CROSS || col <= rr) &&
                            KQ_IN_RANGE(static_cast<int64_t>(rr) * d + col, static_cast<int64_t>(d) * d)) {
                            const float v = st[(r8 + u) * SLD + lane + 32 * m] + old[u][m];
                            H[static_cast<int64_t>(rr) * d + col] = v;
                            st[(r8 + u) * SLD + lane + 32 * m] = v;
                        }
                    }
                }
            }
            __syncwarp();
            if (!CROSS && row < d) {
#pragma unroll 4
                for (int i = 0; i < 128; ++i) {
                    const int col = cbase + i;
                    if (col < d && col < row && KQ_IN_RANGE(static_cast<int64_t>(col) * d + row, static_cast<int64_t>(d) * d))
                        H[static_cast<int64_t>(col) * d + row] = st[lane * SLD + i];
                }
            }
        }
    } else {
        // --------------------------------------------- epilogue of a shared tile (8 warps)
        // Round m: this CTA's chunk (c = KS m + rank) goes to the owners' inboxes, 128 columns at a
        // time, the warp's 32 TMEM lanes to the owner of those rows; then the owners' warps add the
        // round's chunks in order, each thread 16 / KS float4 of its CTA's rows. Inbox of a source:
        // [column quad 32][row 128 / KS] float4.
        constexpr int RO = BM / KS;             // rows owned
        constexpr int QN = RO / 32;             // quadrants (32-row groups) owned
        const int w = warp - 2;
        const int q = warp & 3;                 // TMEM lane quadrant this warp may access
        const int half = w >> 2;                // which 64 of a phase's 128 columns
        const int owner = q / QN;
        float4 acc[2][4 * QN];                  // [phase][quad of columns 4 w + .., row group]
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 4 * QN; ++i) acc[h][i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const uint32_t box = smem_u32(inbox) + static_cast<uint32_t>(rank * RO * 128 * 4);   // my part of any owner's inbox
        const uint32_t box_at = mapa_shared(box, static_cast<uint32_t>(owner)) +
                                static_cast<uint32_t>(((half * 16) * RO + (q % QN) * 32 + lane) * 16);
        const uint32_t full_at = mapa_shared(smem_u32(&in_full[rank]), static_cast<uint32_t>(owner));
        bool ok = true;
        const int rounds = (nchunks + KS - 1) / KS;
        for (int m = 0; m < rounds && ok; ++m) {
            const bool mine = m * KS + rank < nchunks;
            const int buf = m & 1;
            if (mine) {
                ok = mbar_wait(&tfull[buf], static_cast<uint32_t>(m >> 1) & 1u, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t ph = static_cast<uint32_t>(2 * m + h);
                if (mine) {
                    // the owner has added this CTA's previous part (the first wait passes at once)
                    ok = mbar_wait_cl(&in_free[owner], (ph & 1u) ^ 1u, abort_flag);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    const uint32_t base = tmem + (static_cast<uint32_t>(q * 32) << 16) +
                                          static_cast<uint32_t>(buf * BN + h * 128 + half * 64);
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        float v[32];
                        tmem_ld32(base + p * 32, v);
                        tc_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            st_cluster_f4(box_at + static_cast<uint32_t>((p * 8 + i) * RO * 16),
                                          make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
                    }
                    if (h == 1) tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive_remote(full_at);
                        if (h == 1) mbar_arrive(&tempty[buf]);
                    }
                }
                for (int src = 0; src < KS && ok; ++src) {
                    if (m * KS + src >= nchunks) break;
                    ok = mbar_wait_cl(&in_full[src], ph & 1u, abort_flag);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    const float4* in = reinterpret_cast<const float4*>(inbox) + src * RO * 32 + 4 * w * RO + lane;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int g = 0; g < QN; ++g) {
                            const float4 v = in[i * RO + 32 * g];
                            float4& a = acc[h][i * QN + g];
                            a.x += v.x;
                            a.y += v.y;
                            a.z += v.z;
                            a.w += v.w;
                        }
                    __syncwarp();
                    if (lane == 0) mbar_arrive_remote(mapa_shared(smem_u32(&in_free[rank]), static_cast<uint32_t>(src)));
                }
            }
        }
        // Write-out of the owned rows through shared memory (ring and inbox are idle: every chunk
        // sent here has been added), coalesced in both triangles as above.
        ok = named_bar_all(1, 256, ok && !*abort_flag);
        if (ok) {
            constexpr int SLD = BN + 1;
            float* st = reinterpret_cast<float*>(smem);
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int g = 0; g < QN; ++g) {
                        float* x = st + (32 * g + lane) * SLD + 128 * h + 16 * w + 4 * i;
                        const float4 v = acc[h][i * QN + g];
                        x[0] = v.x;
                        x[1] = v.y;
                        x[2] = v.z;
                        x[3] = v.w;
                    }
            named_bar_all(1, 256, true);
            const int rbase = i0 + rank * RO;
#pragma unroll 2
            for (int r = w; r < RO; r += 8) {
                const int rr = rbase + r;
                float old[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int col = j0 + lane + 32 * t;
                    old[t] = (accumulate && rr < d && col < d && (CROSS || col <= rr)) ? H[static_cast<int64_t>(rr) * d + col] : 0.0f;
                }
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int col = j0 + lane + 32 * t;
                    if (rr < d && col < d && (CROSS || col <= rr) &&
                        KQ_IN_RANGE(static_cast<int64_t>(rr) * d + col, static_cast<int64_t>(d) * d)) {
                        const float v = st[r * SLD + lane + 32 * t] + old[t];
                        H[static_cast<int64_t>(rr) * d + col] = v;
                        st[r * SLD + lane + 32 * t] = v;
                    }
                }
            }
            named_bar_all(1, 256, true);
            if (!CROSS) {
#pragma unroll 4
                for (int e = w; e < BN * QN; e += 8) {
                    const int col = j0 + e / QN, r = 32 * (e % QN) + lane, rr = rbase + r;
                    if (rr < d && col < d && col < rr && KQ_IN_RANGE(static_cast<int64_t>(col) * d + rr, static_cast<int64_t>(d) * d))
                        H[static_cast<int64_t>(col) * d + rr] = st[r * SLD + e / QN];
                }
            }
        }
    }

    // (of a cluster: no CTA leaves while another one may still write to it or signal it)
    if constexpr (KS > 1)
        cluster_barrier();
    else
        __syncthreads();
    if (*abort_flag && threadIdx.x == 0) record_error(info, -KQ_ERR_TIMEOUT);
    if (warp == 1) {
        __syncwarp();   // its lanes come from different roles, and the cluster's barrier is not a warp's
        tc_fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
}

template <int KS>
__global__ void __launch_bounds__(NUM_THREADS, 1)
syrk_tc_kernel(const __grid_constant__ CUtensorMap tmap, float* __restrict__ H, int d, int T,
               int n_row_tiles, int tile0, int chunk_stages, int accumulate, int* info) {
    gram_tc_body<false, KS>(&tmap, &tmap, &tmap, H, d, T, n_row_tiles, tile0, chunk_stages, accumulate, info);
}

template <int KS>
__global__ void __launch_bounds__(NUM_THREADS, 1)
drift_tc_kernel(const __grid_constant__ CUtensorMap a_hi, const __grid_constant__ CUtensorMap a_lo,
                const __grid_constant__ CUtensorMap b, float* __restrict__ D, int d, int T,
                int n_row_tiles, int chunk_stages, int accumulate, int* info) {
    gram_tc_body<true, KS>(&a_hi, &a_lo, &b, D, d, T, n_row_tiles, 0, chunk_stages, accumulate, info);
}

// CTAs that share a tile: four while all of them still run at once (one per SM) and each has a chunk.
// They keep four times the SMs for about three quarters of the time, so two such factors on two streams,
// which ran side by side with one CTA a tile, now run mostly one after the other: twice d = 1024 with
// 65536 tokens 361 -> 553 us (d = 512, 24 CTAs each, 359 -> 280). One factor alone is the usual case: two
// whole layers of 1024 x 1024 on two streams take 1328 -> 1275 us (65536 tokens), 3623 -> 3721 (262144).
int ks_of(int64_t tiles, int64_t chunks) { return 4 * tiles <= num_sms() && chunks >= 4 ? 4 : 1; }

// Round a finite fp32 value to the nearest bf16, ties to even; returns the 16 bf16 bits.
__device__ __forceinline__ uint32_t bf16_rn_bits(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u + 0x7fffu + ((u >> 16) & 1u)) >> 16;
}

// Exact split of the drift X~ - X into a bf16 pair: hi = bf16(x~ - x), lo = bf16((x~ - x) - hi).
// x~ - x of two bf16 values is exact in fp32 (their significands have 8 bits), and hi + lo
// carries 16 significant bits, which holds the difference exactly unless the two exponents
// are more than 8 apart (then the pair is within 2^-17 of it). Eight elements per thread.
__global__ void drift_split_kernel(const uint16_t* __restrict__ Xt, const uint16_t* __restrict__ X,
                                   int64_t T, int64_t d, int64_t ld, uint16_t* __restrict__ hi,
                                   uint16_t* __restrict__ lo) {
    const int64_t per_row = d >> 3;
    const int64_t total = T * per_row;
    for (int64_t v = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; v < total;
         v += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t t = v / per_row;
        const int64_t c = (v - t * per_row) << 3;
        const uint4 a = __ldg(reinterpret_cast<const uint4*>(Xt + t * ld + c));
        const uint4 b = __ldg(reinterpret_cast<const uint4*>(X + t * ld + c));
        const uint32_t aw[4] = {a.x, a.y, a.z, a.w};
        const uint32_t bw[4] = {b.x, b.y, b.z, b.w};
        uint32_t hw[4], lw[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t h2 = 0, l2 = 0;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float xa = __uint_as_float(((aw[q] >> (16 * e)) & 0xffffu) << 16);
                const float xb = __uint_as_float(((bw[q] >> (16 * e)) & 0xffffu) << 16);
                const float df = xa - xb;
                const uint32_t h = bf16_rn_bits(df);
                const uint32_t l = bf16_rn_bits(df - __uint_as_float(h << 16));
                h2 |= h << (16 * e);
                l2 |= l << (16 * e);
            }
            hw[q] = h2;
            lw[q] = l2;
        }
        *reinterpret_cast<uint4*>(hi + t * d + c) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
        *reinterpret_cast<uint4*>(lo + t * d + c) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
    }
}

// tr(H) in fp64 from the diagonal (one CTA).
__global__ void trace_kernel(const float* __restrict__ H, int64_t n, double* out) {
    __shared__ double part[32];
    double s = 0.0;
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) s += static_cast<double>(H[j * n + j]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = threadIdx.x < blockDim.x / 32 ? part[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) *out = s;
    }
}

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// 2D map over a [rows x d] bf16 matrix (row stride ld elements): 64-feature x BK-token
// boxes, 128-byte swizzle, zero fill past the last row.
kq_status make_bf16_map(CUtensorMap* m, const uint16_t* base, int64_t d, int64_t rows, int64_t ld,
                        const char* who) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) {
        set_error("%s: cuTensorMapEncodeTiled is unavailable", who);
        return KQ_ERR_CUDA;
    }
    std::memset(m, 0, sizeof(*m));
    cuuint64_t gdim[2] = {static_cast<cuuint64_t>(d), static_cast<cuuint64_t>(rows)};
    cuuint64_t gstride[1] = {static_cast<cuuint64_t>(ld) * 2};
    cuuint32_t box[2] = {64, static_cast<cuuint32_t>(BK)};
    cuuint32_t estride[2] = {1, 1};
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(base), gdim, gstride,
                     box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("%s: cuTensorMapEncodeTiled failed (%d)", who, static_cast<int>(r));
        return KQ_ERR_CUDA;
    }
    return KQ_OK;
}

// Stages (64 tokens each) between drains of the SYRK accumulator. Drains every 512 tokens
// keep the relative error of H_X at T = 262144 near 9e-7; every 1024 or 2048 tokens it grows
// to 2.4e-6 or 5.3e-6 (a downward bias of the tensor-core sums), for 2.5 % less time at 2048.
constexpr int syrk_chunk_stages() { return KQ_SYRK_CHUNK_TOKENS / BK; }

}  // namespace

kq_status launch_trace(const float* H, int64_t n, double* out, cudaStream_t stream) {
    trace_kernel<<<1, 1024, 0, stream>>>(H, n, out);
    KQ_LAUNCH_CHECK("trace_kernel");
    return KQ_OK;
}

KQ_DEBUG_UNIT(syrk)
}  // namespace kq

extern "C" kq_status kq_accum_factor(const uint16_t* A, int64_t T, int64_t d, int64_t lda,
                                     float* H, int accumulate, double* trace, int* info,
                                     kq_stream_t stream_) {
    return kq_accum_factor_beside(A, T, d, lda, H, accumulate, trace, info, 0, stream_);
}

extern "C" kq_status kq_accum_factor_beside(const uint16_t* A, int64_t T, int64_t d, int64_t lda,
                                            float* H, int accumulate, double* trace, int* info,
                                            int beside, kq_stream_t stream_) {
    using namespace kq;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (!H || d < 1 || d > 65536 || T < 0 || (T > 0 && !A) || lda < d) {
        set_error("kq_accum_factor: invalid arguments (d=%lld T=%lld lda=%lld)", (long long)d,
                  (long long)T, (long long)lda);
        return KQ_ERR_INVALID_ARG;
    }
    if (T > 0 && ((reinterpret_cast<uintptr_t>(A) & 15u) != 0 || (lda % 8) != 0 || T > (1ll << 31) - 64)) {
        set_error("kq_accum_factor: A must be 16-byte aligned with lda %% 8 == 0 and T < 2^31");
        return KQ_ERR_INVALID_ARG;
    }
    if (T == 0) {
        if (!accumulate) KQ_CUDA(cudaMemsetAsync(H, 0, sizeof(float) * d * d, stream));
    } else {
        CUtensorMap tmap;
        kq_status st = make_bf16_map(&tmap, A, d, T, lda, "kq_accum_factor");
        if (st != KQ_OK) return st;
        static std::atomic<uint64_t> attr_set{0};
        KQ_TRY(once_per_device(attr_set, [&]() -> kq_status {
            KQ_CUDA(cudaFuncSetAttribute(syrk_tc_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(1)));
            KQ_CUDA(cudaFuncSetAttribute(syrk_tc_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(4)));
            return KQ_OK;
        }));
        const int n_row = static_cast<int>(cdiv(d, BM));
        const int n_col = static_cast<int>(cdiv(d, BN));
        int64_t tiles = 0;
        for (int j = 0; j < n_col; ++j) tiles += (n_row - 2 * j > 0) ? n_row - 2 * j : 0;
        const int ks = ks_of(tiles, cdiv(T, KQ_SYRK_CHUNK_TOKENS));
        // Beside other work: a launch per wave, of equally many tiles, so that the SMs the last wave
        // would leave idle are free all the time (272 tiles on 152 SMs: twice 136; the inverse
        // Cholesky's chain beside them does not wait a tile's whole sum for an SM). Layers, us, one
        // launch and waves: 4096 x 4096 and 131072 tokens 5865 -> 5560 (twice 136), 3584 x 4096 5406 ->
        // 5005 (twice 105), 7168 x 4096 and 65536 6401 -> 5872 (six of 136). Only where 16 SMs or more
        // come free, in up to six waves: each wave's tiles end up to 0.1 ms apart, and 8192 x 4096 (seven
        // of 151, 65536 tokens) took 7128 -> 7199, 14336 x 4096 (21 of 152, 131072) 24103 -> 24723. 4096 x
        // 4096 with 16384 tokens 3419 -> 3432 (a tile takes 0.1 ms there) and with 262144 in one call
        // 8298 -> 8423, hence the range of T.
        const bool by_wave = beside && ks == 1 && T >= 32768 && T < 196608;
        const int64_t full = cdiv(tiles, num_sms());
        const int64_t waves = by_wave && full <= 6 && num_sms() - cdiv(tiles, full) >= 16 ? full : 1;
        const int64_t per = cdiv(tiles, waves);   // tiles per launch
        auto go = [&](auto* kern) -> kq_status {
            for (int64_t t0 = 0; t0 < tiles; t0 += per) {
                const int64_t nt = std::min(per, tiles - t0);
                KQ_CUDA(launch_dependent(kern, dim3(static_cast<unsigned>(nt * ks)), dim3(NUM_THREADS), smem_bytes(ks), stream,
                                         static_cast<unsigned>(ks), false, tmap, H, static_cast<int>(d), static_cast<int>(T),
                                         n_row, static_cast<int>(t0), syrk_chunk_stages(), accumulate, info));
                KQ_LAUNCH_CHECK("syrk_tc_kernel");
            }
            return KQ_OK;
        };
        KQ_TRY(ks == 4 ? go(syrk_tc_kernel<4>) : go(syrk_tc_kernel<1>));
    }
    if (trace) return launch_trace(H, d, trace, stream);
    return KQ_OK;
}

// ---------------------------------------------------------------------------- drift statistic
extern "C" size_t kq_accum_drift_workspace(int64_t T, int64_t d) {
    using namespace kq;
    if (T < 1 || d < 1) return 0;
    const int64_t Tr = cdiv(T, BK) * BK;
    return 2 * static_cast<size_t>(Tr) * static_cast<size_t>(d) * sizeof(uint16_t);
}

extern "C" kq_status kq_accum_drift(const uint16_t* Xt, const uint16_t* X, int64_t T, int64_t d, int64_t ld,
                                    float* D, int accumulate, int* info, void* ws, size_t ws_bytes,
                                    kq_stream_t stream_) {
    using namespace kq;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (!D || d < 1 || d > 65536 || T < 0 || (T > 0 && (!Xt || !X)) || ld < d) {
        set_error("kq_accum_drift: invalid arguments (d=%lld T=%lld ld=%lld)", (long long)d, (long long)T,
                  (long long)ld);
        return KQ_ERR_INVALID_ARG;
    }
    if (T > 0 && ((reinterpret_cast<uintptr_t>(Xt) & 15u) || (reinterpret_cast<uintptr_t>(X) & 15u) ||
                  (ld % 8) != 0 || (d % 8) != 0 || T > (1ll << 31) - 64)) {
        set_error("kq_accum_drift: X~ and X must be 16-byte aligned, d and ld multiples of 8, T < 2^31");
        return KQ_ERR_INVALID_ARG;
    }
    if (T == 0) {
        if (!accumulate) KQ_CUDA(cudaMemsetAsync(D, 0, sizeof(float) * d * d, stream));
        return KQ_OK;
    }
    // token chunk: what the workspace holds (a multiple of BK tokens), at most all of T
    const int64_t per_token = 2 * d * static_cast<int64_t>(sizeof(uint16_t));
    int64_t Tc = ws ? static_cast<int64_t>(ws_bytes / per_token) / BK * BK : 0;
    if (Tc > cdiv(T, BK) * BK) Tc = cdiv(T, BK) * BK;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || Tc < BK) {
        set_error("kq_accum_drift: workspace must be 256-byte aligned and hold at least %lld bytes "
                  "(%zu for one pass)", (long long)(per_token * BK), kq_accum_drift_workspace(T, d));
        return KQ_ERR_WORKSPACE;
    }
    uint16_t* hi = static_cast<uint16_t*>(ws);
    uint16_t* lo = hi + Tc * d;
    static std::atomic<uint64_t> attr_set{0};
    KQ_TRY(once_per_device(attr_set, [&]() -> kq_status {
        KQ_CUDA(cudaFuncSetAttribute(drift_tc_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(1)));
        KQ_CUDA(cudaFuncSetAttribute(drift_tc_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(4)));
        return KQ_OK;
    }));
    const int n_row = static_cast<int>(cdiv(d, BM));
    const int n_col = static_cast<int>(cdiv(d, BN));
    for (int64_t t0 = 0; t0 < T; t0 += Tc) {
        const int64_t tn = std::min<int64_t>(Tc, T - t0);
        const int64_t vecs = tn * (d / 8);
        const int64_t grid = std::min<int64_t>(cdiv(vecs, 256), static_cast<int64_t>(num_sms()) * 16);
        drift_split_kernel<<<static_cast<unsigned>(grid), 256, 0, stream>>>(Xt + t0 * ld, X + t0 * ld, tn, d, ld,
                                                                            hi, lo);
        KQ_LAUNCH_CHECK("drift_split_kernel");
        CUtensorMap mh, ml, mb;
        kq_status st = make_bf16_map(&mh, hi, d, tn, d, "kq_accum_drift");
        if (st == KQ_OK) st = make_bf16_map(&ml, lo, d, tn, d, "kq_accum_drift");
        if (st == KQ_OK) st = make_bf16_map(&mb, X + t0 * ld, d, tn, ld, "kq_accum_drift");
        if (st != KQ_OK) return st;
        const int ks = ks_of(static_cast<int64_t>(n_row) * n_col, cdiv(2 * cdiv(tn, BK), syrk_chunk_stages()));
        auto go = [&](auto* kern) -> kq_status {
            KQ_CUDA(launch_dependent(kern, dim3(static_cast<unsigned>(n_row * n_col * ks)), dim3(NUM_THREADS), smem_bytes(ks),
                                     stream, static_cast<unsigned>(ks), false, mh, ml, mb, D, static_cast<int>(d),
                                     static_cast<int>(tn), n_row, syrk_chunk_stages(), (accumulate || t0 > 0) ? 1 : 0, info));
            KQ_LAUNCH_CHECK("drift_tc_kernel");
            return KQ_OK;
        };
        KQ_TRY(ks == 4 ? go(drift_tc_kernel<4>) : go(drift_tc_kernel<1>));
    }
    return KQ_OK;
}
