// r x r factor kernel of the tensor-core engine: Cholesky factor of the Gram matrix and its explicit
// inverse, one CTA per matrix or one matrix per thread-block cluster (MULTI).
//
// Z L^T = [Gram; I] has the solution Z = [L; L^{-T}]: appending the identity below the Gram matrix
// turns the inverse into more rows of the factorisation.  Both are therefore ONE left-looking
// loop over 64-wide block columns k, in which every 64-row tile t takes the same two steps:
//     S = Z0[t, k] - sum_{c < k} Z[t, c] L[k, c]^T        (Z0: Gram rows for t > k, zero for L^{-T} rows t < k)
//     Z[t, k] = S X_k^T,     X_k = L[k, k]^{-1}
// and the block column has nb - 1 such tiles whatever k is.  L and L^{-T} are kept as split images
// (common.cuh), i.e. in the two bf16 terms that the products read anyway; the image of L^{-T} is the
// operand of the apply product, so nothing is converted afterwards.  Tile products run on the
// warp-level tensor path (mma.sync m16n8k16, hi*hi + hi*lo + lo*hi: about 2^-16), operand tiles of
// 64 x 64 come in by cp.async one step ahead.
//
// What bounds it: the chain of r / 64 diagonal blocks.  Four extra warps per CTA factor and invert a
// 64 x 64 block in fp32 (about 3 us: one warp eliminates 32 columns with the rows in registers and the
// next pivot computed ahead of its column) while the eight product warps do the S sums of
// the same block column, which do not depend on it; the tile below the diagonal goes first, together
// with the next diagonal block's own sum, so that the chain never waits for the rest.  64-wide
// blocks instead of 32: half the barriers, and a diagonal block still fits one warp pair's registers.
// Measured, factor stage of a step (six launches, ms), before (32-wide blocks, fp32 tiles split at every
// use, a pairwise inversion afterwards) -> now: one matrix r = 64 0.19 -> 0.09, r = 256 0.74 -> 0.26, r = 512
// 1.47 -> 0.37, r = 1024 3.68 -> 0.70; 56 matrices at r = 512 2.7 -> 0.7, 154 of them 5.0 -> 1.5.
//
// The later passes of a CholeskyQR see a Gram matrix I + E with E tiny; when a rigorous bound on
// |E|_2 is small enough, L^{-1} = I - Phi(E) (first order) replaces the factorisation.
//
// MULTI form: the row tiles are dealt out over the CTAs of the cluster (tile t to CTA t mod size); the
// matrix stays in global memory (L2), phases are separated by release/acquire cluster barriers, and
// what another CTA may have written is read past L1.  Per tile the arithmetic and its order are
// those of the single-CTA form: a matrix gets the same bits in either.  Decisions that steer control
// flow are taken from values that every CTA reads from memory after a barrier.
#pragma once
#include "common.cuh"
#include "factor_kernels.cuh"

namespace od {

constexpr int CT_MMA_WARPS = 8;
constexpr int CT_DIAG_WARPS = 4;
constexpr int CT_MMA_THREADS = 32 * CT_MMA_WARPS;
constexpr int CT_THREADS = 32 * (CT_MMA_WARPS + CT_DIAG_WARPS);
constexpr int CT_NB = 64;                     // block width, tile rows
constexpr int CT_TERM = CT_NB * 128;          // one bf16 term of a 64 x 64 tile: 64 image rows of 128 bytes
constexpr int CT_TILE = 2 * CT_TERM;
constexpr int CT_LDD = 68;                    // diagonal block, fp32 (rows 16-byte aligned, conflict-free by row)
constexpr int CT_LDT = 68;                    // transposed factor columns: 32 x 64 (the second half's in place of L11's)
constexpr int CT_LDS = 65;                    // transposing buffer of the first-order inverse
// dynamic shared memory: two stages of an A tile and a B tile, then the diagonal block's work area
constexpr int CT_OFF_D = 4 * CT_TILE;
constexpr int CT_DG_LT = CT_NB * CT_LDD * 4;                   // work area of a diagonal block: the block itself first
constexpr int CT_DG_RS = CT_DG_LT + 32 * CT_LDT * 4;
constexpr int CT_DG_BYTES = CT_DG_RS + 64 * 4;
constexpr int CT_OFF_D2 = CT_OFF_D + CT_DG_BYTES;              // the block of the odd columns (the even ones': CT_OFF_D)
constexpr int CT_SMEM_BYTES = CT_OFF_D2 + CT_NB * CT_LDD * 4 + 1024;     // + alignment of the tiles
static_assert(2 * (CT_SMEM_BYTES + 2048) <= 228 * 1024, "two CTAs per multiprocessor");
static_assert(3 * CT_NB * CT_LDS * 4 <= 4 * CT_TILE, "three transposing buffers fit the operand stages");
constexpr int CT_MAX_BLOCKS = 64;             // r <= 4096
constexpr int CT_STAT_FLOATS = 3 * CT_MAX_BLOCKS;   // per block: smallest and largest diagonal entry, row-sum bound
constexpr float CT_THIRD_PASS_LIMIT = 0.02f; // bound on |Gram - I|_2 of the second pass above which a third follows
constexpr float CT_SERIES_LIMIT = 1.4e-3f;   // bound on |Gram - I|_2 below which L^{-1} = I - Phi(E) is used

__device__ __forceinline__ void ct_bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void ct_bar_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// named barriers (0: the whole CTA); CT_BAR_XT: two, by the parity of the column
constexpr int CT_BAR_MMA = 1, CT_BAR_DIAG = 2, CT_BAR_READY = 3, CT_BAR_X = 4, CT_BAR_XT = 5;

__device__ __forceinline__ void ct_cp16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void ct_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void ct_cp_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void ct_prefetch(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

__device__ __forceinline__ void mma_bf16_16x8x16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ct_ldsm4(uint32_t (&v)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
}

// acc (this warp's 16 x 32 part of a 64 x 64 tile) += A B^T, both tiles K-major in shared memory (two
// terms each).  Warp w: rows 16 (w % 4) .., columns 32 (w / 4) ...
__device__ __forceinline__ void ct_tile_mma(float (&acc)[4][4], uint32_t a_tile, uint32_t b_tile, int warp, int lane) {
    const int l8 = lane & 7;
    const uint32_t a_row = a_tile + ((warp % 4) * 16 + l8 + ((lane >> 3) & 1) * 8) * 128;
    const uint32_t b_row = b_tile + ((warp / 4) * 32 + l8 + (lane >> 4) * 8) * 128;
    const int a_ch = lane >> 4, b_ch = (lane >> 3) & 1;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        const uint32_t ao = (uint32_t)(((2 * ks + a_ch) ^ l8) << 4), bo = (uint32_t)(((2 * ks + b_ch) ^ l8) << 4);
        uint32_t ah[4], al[4];
        ct_ldsm4(ah, a_row + ao);
        ct_ldsm4(al, a_row + CT_TERM + ao);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t bh[4], bl[4];
            ct_ldsm4(bh, b_row + h * 2048 + bo);
            ct_ldsm4(bl, b_row + CT_TERM + h * 2048 + bo);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                mma_bf16_16x8x16(acc[2 * h + u], ah, bh[2 * u], bh[2 * u + 1]);
                mma_bf16_16x8x16(acc[2 * h + u], ah, bl[2 * u], bl[2 * u + 1]);
                mma_bf16_16x8x16(acc[2 * h + u], al, bh[2 * u], bh[2 * u + 1]);
            }
        }
    }
}
// this warp's part of a tile, v -> the two bf16 terms of a K-major tile in shared memory
__device__ __forceinline__ void ct_store_tile(uint32_t tile, const float (&v)[4][4], int warp, int lane) {
    const int row = (warp % 4) * 16 + lane / 4;             // row & 7 == lane / 4 for both halves
#pragma unroll
    for (int nf = 0; nf < 4; ++nf) {
        const int ch = (warp / 4) * 4 + nf;
        const uint32_t o = (uint32_t)(row * 128 + ((ch ^ (row & 7)) << 4) + (lane % 4) * 4);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t hi = pack_bf16x2(v[nf][2 * h], v[nf][2 * h + 1]);
            const uint32_t lo = pack_bf16x2(v[nf][2 * h] - bf16lo_to_f32(hi), v[nf][2 * h + 1] - bf16hi_to_f32(hi));
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(tile + o + h * 1024), "r"(hi) : "memory");
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(tile + CT_TERM + o + h * 1024), "r"(lo) : "memory");
        }
    }
}

// ---- diagonal blocks (fp32, one warp) ------------------------------------------------------------
// Cholesky of the leading NC columns of the 32 x 32 block at `blk` (ld CT_LDD).  Lane i holds row i in registers.  LT[j][i] <- L(i, j),
// rs[j] <- 1 / L(j, j); the lane keeps its pivot in `piv`.  The pivot of column j + 1 is formed from two
// values fetched before column j was scaled, so that the chain per column is one reciprocal square root
// and two products; the next two columns get their multiplier by shuffle, the others from LT.
template <int NC>
__device__ __forceinline__ void ct_chol32(const float* blk, float* LT, float* rs, float& piv, int lane) {
    float a[NC];
#pragma unroll
    for (int c = 0; c < NC; c += 4) {
        const float4 v = *reinterpret_cast<const float4*>(blk + lane * CT_LDD + c);
        a[c] = v.x; a[c + 1] = v.y; a[c + 2] = v.z; a[c + 3] = v.w;
    }
    float d = __shfl_sync(0xffffffffu, a[0], 0);
    float q = __shfl_sync(0xffffffffu, a[0], 1), p = __shfl_sync(0xffffffffu, a[1], 1);
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const float inv = rsqrtf(d);
        if (lane == j) { piv = d; rs[j] = inv; }
        const float la = a[j] * inv;
        LT[j * CT_LDT + lane] = la;
        if (j + 1 < NC) { const float t = q * inv; d = fmaf(-t, t, p); }
#pragma unroll
        for (int c = j + 1; c < j + 3; ++c)
            if (c < NC) a[c] = fmaf(-la, __shfl_sync(0xffffffffu, la, c), a[c]);
        if (j + 2 < NC) { q = __shfl_sync(0xffffffffu, a[j + 1], j + 2); p = __shfl_sync(0xffffffffu, a[j + 2], j + 2); }
        __syncwarp();
#pragma unroll
        for (int c4 = (j + 3) / 4; c4 < NC / 4; ++c4) {
            const float4 v = *reinterpret_cast<const float4*>(LT + j * CT_LDT + 4 * c4);
            const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (4 * c4 + e >= j + 3) a[4 * c4 + e] = fmaf(-la, vv[e], a[4 * c4 + e]);
        }
    }
}
// s <- L^{-1} s for the NC x NC factor held in LT, rs; each lane has a right-hand side of its own
template <int NC>
__device__ __forceinline__ void ct_solve32(float (&s)[NC], const float* LT, const float* rs) {
#pragma unroll
    for (int p = 0; p < NC; ++p) {
        const float x = s[p] * rs[p];
        s[p] = x;
#pragma unroll
        for (int i4 = (p + 1) / 4; i4 < NC / 4; ++i4) {
            const float4 v = *reinterpret_cast<const float4*>(LT + p * CT_LDT + 4 * i4);
            const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (4 * i4 + e > p) s[4 * i4 + e] = fmaf(-vv[e], x, s[4 * i4 + e]);
        }
    }
}
// The four diagonal warps: sD (64 x 64, ld CT_LDD, identity beyond nbk) <- inverse of its Cholesky factor
// (lower triangle; what lies above it is not defined: the upper right quarter holds T).  piv[]: the lane's
// pivots of warp 0.  `area`: CT_DG_BYTES of shared memory, sD first.  NC < 32: nbk <= NC, only the leading NC
// columns are looked at.  (sD lies at the start of the area, or apart from its rest: `rest` is the area then.)
//   L11                                       warp 0
//   L21 = D21 L11^{-T}  (warp 1)              X11 = L11^{-1}  (warp 2)
//   D22 -= L21 L21^T                          all
//   L22  (warp 0)                             T = L21 X11  (warps 1-3, by rows)
//   X22 = L22^{-1}  (warp 0)                  X21 = -L22^{-1} T  (warp 1)
template <int NC>
__device__ __forceinline__ void ct_diag_block(float* sD, unsigned char* rest, int nbk, int dw, int lane, float (&piv)[2]) {
    float* LT = reinterpret_cast<float*>(rest + CT_DG_LT);
    float* sT = sD + 32;
    float* rs = reinterpret_cast<float*>(rest + CT_DG_RS);
    const bool two = NC == 32 && nbk > 32;
    if (dw == 0) ct_chol32<NC>(sD, LT, rs, piv[0], lane);
    ct_bar_sync(CT_BAR_DIAG, 32 * CT_DIAG_WARPS);
    float s[NC];
    if (dw == 2 || (dw == 1 && two)) {
#pragma unroll
        for (int i = 0; i < NC; i += 4) {
            float4 v = make_float4(i == lane ? 1.f : 0.f, i + 1 == lane ? 1.f : 0.f, i + 2 == lane ? 1.f : 0.f, i + 3 == lane ? 1.f : 0.f);
            if (dw == 1) v = *reinterpret_cast<const float4*>(sD + (32 + lane) * CT_LDD + i);
            s[i] = v.x; s[i + 1] = v.y; s[i + 2] = v.z; s[i + 3] = v.w;
        }
        ct_solve32<NC>(s, LT, rs);
        float* dst = dw == 1 ? LT + 32 + lane : sD + lane;
        const int ld = dw == 1 ? CT_LDT : CT_LDD;
#pragma unroll
        for (int i = 0; i < NC; ++i) dst[i * ld] = s[i];
    }
    ct_bar_sync(CT_BAR_DIAG, 32 * CT_DIAG_WARPS);
    if constexpr (NC == 32) {
    if (!two) return;
    {
        // D22(lane, 8 dw ..) -= sum_j L21(lane, j) L21(8 dw .., j)
        float o[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) o[e] = sD[(32 + lane) * CT_LDD + 32 + 8 * dw + e];
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const float l = LT[j * CT_LDT + 32 + lane];
            const float4 u = *reinterpret_cast<const float4*>(LT + j * CT_LDT + 32 + 8 * dw);
            const float4 v = *reinterpret_cast<const float4*>(LT + j * CT_LDT + 36 + 8 * dw);
            o[0] = fmaf(-l, u.x, o[0]); o[1] = fmaf(-l, u.y, o[1]); o[2] = fmaf(-l, u.z, o[2]); o[3] = fmaf(-l, u.w, o[3]);
            o[4] = fmaf(-l, v.x, o[4]); o[5] = fmaf(-l, v.y, o[5]); o[6] = fmaf(-l, v.z, o[6]); o[7] = fmaf(-l, v.w, o[7]);
        }
#pragma unroll
        for (int e = 0; e < 8; e += 4)
            *reinterpret_cast<float4*>(sD + (32 + lane) * CT_LDD + 32 + 8 * dw + e) = make_float4(o[e], o[e + 1], o[e + 2], o[e + 3]);
    }
    ct_bar_sync(CT_BAR_DIAG, 32 * CT_DIAG_WARPS);
    if (dw == 0) {
        ct_chol32<32>(sD + 32 * CT_LDD + 32, LT, rs + 32, piv[1], lane);
    } else {
        // rows 12 (dw - 1) .. + 11 of T (the last warp: 8 rows), a column per lane
        const int i0 = 12 * (dw - 1);
        float t[12];
#pragma unroll
        for (int e = 0; e < 12; ++e) t[e] = 0.f;
#pragma unroll 8
        for (int q = 0; q < 32; ++q) {
            const float x = sD[q * CT_LDD + lane];
#pragma unroll
            for (int e = 0; e < 12; e += 4) {
                if (e < 8 || dw < 3) {
                    const float4 v = *reinterpret_cast<const float4*>(LT + q * CT_LDT + 32 + i0 + e);
                    t[e] = fmaf(v.x, x, t[e]); t[e + 1] = fmaf(v.y, x, t[e + 1]);
                    t[e + 2] = fmaf(v.z, x, t[e + 2]); t[e + 3] = fmaf(v.w, x, t[e + 3]);
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 12; ++e)
            if (e < 8 || dw < 3) sT[(i0 + e) * CT_LDD + lane] = t[e];
    }
    ct_bar_sync(CT_BAR_DIAG, 32 * CT_DIAG_WARPS);
    if (dw < 2) {
#pragma unroll
        for (int i = 0; i < 32; ++i) s[i] = dw == 0 ? (i == lane ? 1.f : 0.f) : -sT[i * CT_LDD + lane];
        ct_solve32<32>(s, LT, rs + 32);
#pragma unroll
        for (int i = 0; i < 32; ++i) sD[(32 + i) * CT_LDD + (dw == 0 ? 32 : 0) + lane] = s[i];
    }
    ct_bar_sync(CT_BAR_DIAG, 32 * CT_DIAG_WARPS);
    }
}

// smallest and largest diagonal entry of the factor from the pivots of warp 0; smallest -1 after a breakdown
__device__ __forceinline__ void ct_pivot_range(const float (&piv)[2], int nbk, int lane, float& mn, float& mx) {
    mn = 3.0e38f; mx = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h * 32 + lane < nbk) {
            if (!(piv[h] > 0.f) || !(piv[h] <= 3.0e38f)) mn = -1.f;
            else { const float sq = sqrtf(piv[h]); mn = fminf(mn, sq); mx = fmaxf(mx, sq); }
        }
    }
    for (int o = 16; o; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
}
// v[e] over the value that its two bf16 terms hold
__device__ __forceinline__ float ct_diag_scale(const float (&v)[8], const uint4& t0, const uint4& t1, int e) {
    const uint32_t h[4] = {t0.x, t0.y, t0.z, t0.w}, l[4] = {t1.x, t1.y, t1.z, t1.w};
    float s = 1.f;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (i == e) {
            const uint32_t hp = h[i / 2], lp = l[i / 2];
            s = v[i] / ((i & 1) ? bf16hi_to_f32(hp) + bf16hi_to_f32(lp) : bf16lo_to_f32(hp) + bf16lo_to_f32(lp));
        }
    return s;
}

template <bool MULTI>
__global__ void __launch_bounds__(CT_THREADS, 2)
factor_kernel(const __grid_constant__ Batch batch, CholArgs a, int csize) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ float red[CT_THREADS / 32];
    __shared__ float s_row[64];
    __shared__ int s_status;
    unsigned char* smem = smem_raw;
    {
        const uint32_t raw = static_cast<uint32_t>(__cvta_generic_to_shared(smem_raw));
        smem += ((raw + 1023u) & ~1023u) - raw;
    }
    const uint32_t smem0 = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    auto diag_buf = [&](int k) { return reinterpret_cast<float*>(smem + ((k & 1) ? CT_OFF_D2 : CT_OFF_D)); };
    float* s_part = reinterpret_cast<float*>(smem);       // partial column sums, before the operand stages are in use

    // MULTI: the csize CTAs of a cluster (ranks 0 .. csize-1) share matrix blockIdx.x / csize
    const int crank = MULTI ? (int)(blockIdx.x % (unsigned)csize) : 0;
    const int nshare = MULTI ? csize : 1;
    const MatWork& w = batch.w[MULTI ? blockIdx.x / (unsigned)csize : blockIdx.x];
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const int r = a.r;
    const int nb = (r + CT_NB - 1) / CT_NB;
    const int shift_bit = a.which ? ST_SHIFT_R : ST_SHIFT_L;
    auto phase_sync = [&]() { if (MULTI) cluster_sync_all(); else __syncthreads(); };

    grid_dependency();
    if (tid == 0) s_status = *w.status;
    __syncthreads();
    // every CTA of the cluster has read the status word before any of them may change it
    if (MULTI) cluster_sync_all();
    const int st0 = s_status;
    if (st0 & ST_FAILED) return;
    if (a.pass == 3 && !(st0 & shift_bit)) return;

    const float* __restrict__ A = pick(w, a.gram);     // Gram matrix: never written here
    unsigned char* scr = reinterpret_cast<unsigned char*>(w.scratch);
    float* gdiag = reinterpret_cast<float*>(w.scratch + a.diag_off);      // r floats, then the block statistics
    float* gstat = reinterpret_cast<float*>(w.scratch + a.stat_off);
    float* gscale = reinterpret_cast<float*>(w.scratch + a.scale_off);
    const int64_t term = (int64_t)a.img.panels * a.img.rows_pad * 128;    // bytes between the terms of an image
    auto l_tile = [&](int t, int c) { return scr + a.limg_off + ((int64_t)c * a.img.rows_pad + (int64_t)t * CT_NB) * 128; };
    auto x_tile = [&](int t, int c) { return scr + a.img.off + ((int64_t)c * a.img.rows_pad + (int64_t)t * CT_NB) * 128; };

    // ---- Gram diagonal (from the fp32 column sums of squares), by row tile --------------------
    // Eight interleaved partial sums per column, added in order: the order depends on the number of
    // partials only.
    if (a.use_colsq) {
        const float* cs = pick(w, a.colsq);
        const int nparts = w.aux0;
        const int grp = tid / 128, g = (tid % 128) / 16, q4 = (tid % 16) * 4;     // three tiles at a time
        for (int t0 = crank; t0 < nb; t0 += 3 * nshare) {
            const int t = t0 + grp * nshare, col = t * CT_NB + q4;
            float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
            if (col < r) {
#pragma unroll 8
                for (int kb = g; kb < nparts; kb += 8) {
                    const float4 v = *reinterpret_cast<const float4*>(cs + (int64_t)kb * r + col);
                    d.x += v.x; d.y += v.y; d.z += v.z; d.w += v.w;
                }
            }
            *reinterpret_cast<float4*>(s_part + (grp * 8 + g) * 64 + q4) = d;
            __syncthreads();
            const int c = tid % 128, i = t * CT_NB + c;
            if (c < 64 && i < r) {
                float sum = 0.f;
                for (int q = 0; q < 8; ++q) sum += s_part[(grp * 8 + q) * 64 + c];
                gdiag[i] = sum;
                if (a.cnorm_off >= 0) reinterpret_cast<float*>(w.scratch + a.cnorm_off)[i] = sum;
            }
            __syncthreads();
        }
    } else {
        for (int t = crank; t < nb; t += nshare)
            if (tid < 64 && t * CT_NB + tid < r) {
                const int i = t * CT_NB + tid;
                const float d = A[(int64_t)i * r + i];
                gdiag[i] = d;
                if (a.cnorm_off >= 0) reinterpret_cast<float*>(w.scratch + a.cnorm_off)[i] = d;
            }
    }
    phase_sync();
    float trace = 0.f;
    {
        for (int i = tid; i < r; i += CT_THREADS) trace += __ldcg(gdiag + i);
        for (int o = 16; o; o >>= 1) trace += __shfl_xor_sync(0xffffffffu, trace, o);
        if (lane == 0) red[warp] = trace;
        __syncthreads();
        trace = 0.f;
        for (int i = 0; i < CT_THREADS / 32; ++i) trace += red[i];
        __syncthreads();
    }
    // (the same sum in the same order in every CTA of a cluster: all of them take this exit or none)
    if (!(fabsf(trace) <= 3.0e38f)) {   // Inf or NaN
        if (tid == 0 && crank == 0) atomicOr(w.status, ST_NONFINITE);
        return;
    }

    // Tiles of the L^{-T} image below its diagonal that the apply product reads as zeros: those inside the
    // same 256-column block
    for (int t = crank; t < nb; t += nshare)
        for (int c = t & ~3; c < t; ++c) {
            unsigned char* dst = x_tile(t, c);
            for (int q = tid; q < 1024; q += CT_THREADS)
                *reinterpret_cast<uint4*>(dst + (q >= 512 ? term : 0) + (q & 511) * 16) = make_uint4(0u, 0u, 0u, 0u);
        }

    // ---- later passes of the QR: the Gram matrix is I + E with E small ------------------------
    // L = I + X with X + X^T + X X^T = E, so L^{-1} = I - Phi(E) + O(|E|^2), Phi = strict lower part
    // plus half the diagonal.  |E|_2 <= max row sum of |E| (E is symmetric); when that bound is
    // below CT_SERIES_LIMIT the dropped terms are below 2e-6 and the factorisation is skipped.
    if (a.pass >= 2) {
        for (int t = crank; t < nb; t += nshare) {
            const int i0 = t * CT_NB;
            // left of the diagonal: a row per warp
            for (int i = i0 + warp; i < min(r, i0 + CT_NB); i += CT_THREADS / 32) {
                float s = 0.f;
                for (int j = lane * 4; j < i; j += 128) {
                    const float4 v = *reinterpret_cast<const float4*>(A + (int64_t)i * r + j);
                    s += fabsf(v.x) + (j + 1 < i ? fabsf(v.y) : 0.f) + (j + 2 < i ? fabsf(v.z) : 0.f) + (j + 3 < i ? fabsf(v.w) : 0.f);
                }
                for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) s_row[i - i0] = s;
            }
            // below the diagonal (the mirror of the row's right part): 24 row groups x 64 columns
            {
                const int g = tid / 16, j = i0 + (tid % 16) * 4;
                float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                if (j < r) {
#pragma unroll 4
                    for (int i = i0 + g; i < r; i += 24) {
                        const float4 v = *reinterpret_cast<const float4*>(A + (int64_t)i * r + j);
                        s.x += i > j ? fabsf(v.x) : 0.f; s.y += i > j + 1 ? fabsf(v.y) : 0.f;
                        s.z += i > j + 2 ? fabsf(v.z) : 0.f; s.w += i > j + 3 ? fabsf(v.w) : 0.f;
                    }
                }
                *reinterpret_cast<float4*>(s_part + g * 64 + (tid % 16) * 4) = s;
            }
            __syncthreads();
            if (warp == 0) {
                float mx = 0.f;
                for (int q = lane; q < 64 && i0 + q < r; q += 32) {
                    float s = fabsf(__ldcg(gdiag + i0 + q) - 1.f) + s_row[q];
                    for (int g = 0; g < 24; ++g) s += s_part[g * 64 + q];
                    mx = fmaxf(mx, s <= 3.0e38f ? s : 3.3e38f);
                }
                for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                if (lane == 0) gstat[2 * CT_MAX_BLOCKS + t] = mx;
            }
            __syncthreads();
        }
        phase_sync();
        float mx = 0.f;
        for (int t = 0; t < nb; ++t) mx = fmaxf(mx, __ldcg(gstat + 2 * CT_MAX_BLOCKS + t));
        // Second pass with Q1 far from orthonormal (cond(Y)^2 u was not small): its result will
        // not be orthonormal to working accuracy either, so ask for the third pass.
        if (a.pass == 2 && !(mx <= CT_THIRD_PASS_LIMIT) && tid == 0 && crank == 0) atomicOr(w.status, shift_bit);
        // (a diagonal this close to one is held by its two terms to 2^-20: no correction)
        if (tid == 0 && crank == 0) gscale[r] = mx <= CT_SERIES_LIMIT ? 0.f : 1.f;
        if (mx <= CT_SERIES_LIMIT) {
            // Image tiles (ta, tb), tb >= ta, of L^{-T}: entry (row, col) = -E(col, row) right of the
            // diagonal.  Three groups of four warps, each with a transposing buffer of its own.
            const int grp = tid / 128, gt = tid % 128;
            float* buf = reinterpret_cast<float*>(smem) + grp * CT_NB * CT_LDS;
            const int pairs = nb * (nb + 1) / 2;
            for (int q0 = crank * 3; q0 < pairs; q0 += 3 * nshare) {
                int tb = 0, q = q0 + grp;
                const bool on = q < pairs;
                while (on && q > tb) { q -= tb + 1; ++tb; }
                const int ta = q;
                if (on) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int i = gt / 16 + 8 * e, j = (gt % 16) * 4;
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (tb * CT_NB + i < r && ta * CT_NB + j < r)
                            v = *reinterpret_cast<const float4*>(A + (int64_t)(tb * CT_NB + i) * r + ta * CT_NB + j);
                        buf[i * CT_LDS + j] = v.x; buf[i * CT_LDS + j + 1] = v.y;
                        buf[i * CT_LDS + j + 2] = v.z; buf[i * CT_LDS + j + 3] = v.w;
                    }
                }
                __syncthreads();
                if (on) {
                    unsigned char* dst = x_tile(ta, tb);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int row = gt / 8 + 16 * e, ch = gt % 8;
                        const int gr = ta * CT_NB + row, gc = tb * CT_NB + ch * 8;
                        float v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] = gc + i > gr ? -buf[(ch * 8 + i) * CT_LDS + row] : 0.f;
                        if (gr >= gc && gr < gc + 8 && gr < r) {
                            const float dg = 0.5f * (3.f - __ldcg(gdiag + gr));
#pragma unroll
                            for (int i = 0; i < 8; ++i) v[i] = gc + i == gr ? dg : v[i];
                        }
                        uint4 t0, t1;
                        split8(v, t0, t1);
                        const int o = row * 128 + img_chunk_offset(row, ch);
                        *reinterpret_cast<uint4*>(dst + o) = t0;
                        *reinterpret_cast<uint4*>(dst + term + o) = t1;
                    }
                }
                __syncthreads();
            }
            return;
        }
    }

    // ---- factorisation and inverse ------------------------------------------------------------
    const bool mma_role = warp < CT_MMA_WARPS;
    const int mrow = (warp % 4) * 16 + lane / 4, mcol = (warp / 4) * 32 + (lane % 4) * 2;     // first element of acc
    int stage = 0;                     // operand stage that the next load goes to
    auto a_slot = [&](int s) { return smem0 + (uint32_t)s * 2 * CT_TILE; };
    auto b_slot = [&](int s) { return smem0 + (uint32_t)s * 2 * CT_TILE + CT_TILE; };
    auto load_tile = [&](uint32_t dst, const unsigned char* src) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int q = (tid + CT_MMA_THREADS * e) * 16;
            ct_cp16(dst + q, src + q);
            ct_cp16(dst + CT_TERM + q, src + term + q);
        }
    };
    // acc += sum_{c in [c0, k)} Z[t, c] L[k, c]^T; with `next` also accd += sum Z[t, c] Z[t, c]^T
    auto sum_products = [&](float (&acc)[4][4], float (&accd)[4][4], int t, int k, bool next) {
        const int c0 = t < k ? t : 0;
        auto load = [&](int c, int s) {
            load_tile(a_slot(s), t < k ? x_tile(t, c) : l_tile(t, c));
            load_tile(b_slot(s), l_tile(k, c));
            ct_cp_commit();
        };
        if (c0 < k) load(c0, stage);
        for (int c = c0; c < k; ++c) {
            ct_cp_wait_all();
            ct_bar_sync(CT_BAR_MMA, CT_MMA_THREADS);
            if (c + 1 < k) load(c + 1, stage ^ 1);
            ct_tile_mma(acc, a_slot(stage), b_slot(stage), warp, lane);
            if (next) ct_tile_mma(accd, a_slot(stage), a_slot(stage), warp, lane);
            stage ^= 1;
        }
    };
    auto prefetch_gram = [&](int t, int k) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = t * CT_NB + mrow + 8 * h, j = k * CT_NB + (warp / 4) * 32;
            if (i < r && j < r) ct_prefetch(A + (int64_t)i * r + j);
        }
    };
    // acc <- Gram[t, k] - acc (L rows) or -acc (L^{-T} rows)
    auto finish_sum = [&](float (&acc)[4][4], int t, int k) {
#pragma unroll
        for (int nf = 0; nf < 4; ++nf)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = t * CT_NB + mrow + 8 * h, j = k * CT_NB + mcol + nf * 8;
                float2 v = make_float2(0.f, 0.f);
                if (t > k && i < r && j < r) v = *reinterpret_cast<const float2*>(A + (int64_t)i * r + j);
                acc[nf][2 * h] = v.x - acc[nf][2 * h];
                acc[nf][2 * h + 1] = v.y - acc[nf][2 * h + 1];
            }
    };
    // Z[t, k] = acc X_k^T -> its image; leaves the tile in the A slot of stage ^ 1
    auto panel = [&](float (&acc)[4][4], int t, int k) {
        load_tile(b_slot(stage), l_tile(k, k));
        ct_cp_commit();
        ct_store_tile(a_slot(stage), acc, warp, lane);
        ct_cp_wait_all();
        ct_bar_sync(CT_BAR_MMA, CT_MMA_THREADS);
        float o[4][4] = {};
        ct_tile_mma(o, a_slot(stage), b_slot(stage), warp, lane);
        ct_store_tile(a_slot(stage ^ 1), o, warp, lane);
        ct_bar_sync(CT_BAR_MMA, CT_MMA_THREADS);
        unsigned char* dst = t < k ? x_tile(t, k) : l_tile(t, k);
        const unsigned char* src = smem + (size_t)(stage ^ 1) * 2 * CT_TILE;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int q = (tid + CT_MMA_THREADS * e) * 16;
            *reinterpret_cast<uint4*>(dst + q) = *reinterpret_cast<const uint4*>(src + q);
            *reinterpret_cast<uint4*>(dst + term + q) = *reinterpret_cast<const uint4*>(src + CT_TERM + q);
        }
    };
    // sD <- diagonal block k: Gram - accd, the diagonal itself from gdiag (+ shift), identity beyond r
    auto write_diag = [&](const float (&accd)[4][4], int k, float shift) {
        float* sD = diag_buf(k);
#pragma unroll
        for (int nf = 0; nf < 4; ++nf)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int il = mrow + 8 * (e / 2), jl = mcol + nf * 8 + (e % 2);
                const int i = k * CT_NB + il, j = k * CT_NB + jl;
                float v = il == jl ? 1.f : 0.f;
                if (i < r && j < r) v = (il == jl ? __ldcg(gdiag + i) + shift : A[(int64_t)i * r + j]) - accd[nf][e];
                sD[il * CT_LDD + jl] = v;
            }
    };

    bool ok = false;
    const int max_attempts = (a.pass == 1) ? 2 : 1;
    for (int attempt = 0; attempt < max_attempts && !ok; ++attempt) {
        const float shift = attempt ? a.shift_rel * trace : 0.f;
        if (mma_role) {
            if (crank == 0) {
                const float none[4][4] = {};
                write_diag(none, 0, shift);
                ct_bar_arrive(CT_BAR_READY, CT_THREADS);
            }
            for (int k = 0; k < nb; ++k) {
                const bool next = k + 1 < nb && (k + 1) % nshare == crank;      // this CTA has the next diagonal block
                // own tiles of this block column, the one below the diagonal first
                int t = next ? k + 1 : crank;
                auto seek = [&]() { while (t < nb && (t == k || (next && t == k + 1))) t += nshare; };
                if (!next) seek();
                float acc[4][4] = {}, accd[4][4] = {};
                const bool first = t < nb;
                if (first) {
                    if (t > k) prefetch_gram(t, k);
                    sum_products(acc, accd, t, k, next);
                    finish_sum(acc, t, k);
                }
                // X_k is in memory
                if (MULTI) cluster_sync_all();
                else ct_bar_sync(CT_BAR_X, CT_THREADS);
                if (first) {
                    panel(acc, t, k);
                    if (next) {
                        const uint32_t z = a_slot(stage ^ 1);
                        ct_tile_mma(accd, z, z, warp, lane);
                        write_diag(accd, k + 1, shift);
                        ct_bar_arrive(CT_BAR_READY, CT_THREADS);
                        t = crank;
                        seek();
                    } else {
                        t += nshare;
                        seek();
                    }
                    for (; t < nb;) {
                        if (t > k) prefetch_gram(t, k);
#pragma unroll
                        for (int nf = 0; nf < 4; ++nf)
#pragma unroll
                            for (int e = 0; e < 4; ++e) acc[nf][e] = 0.f;
                        sum_products(acc, accd, t, k, false);
                        finish_sum(acc, t, k);
                        panel(acc, t, k);
                        t += nshare;
                        seek();
                    }
                }
                // block column k is in memory
                if (MULTI) cluster_sync_all();
                else ct_bar_sync(CT_BAR_XT + (k & 1), CT_THREADS);
            }
        } else {
            // The four diagonal warps.  Block k + 1 is started as soon as the product warps have its sum, while they go
            // on with block column k: what they owe the barriers of column k is an arrival, not a wait.
            const int dw = warp - CT_MMA_WARPS, dt = tid - CT_MMA_THREADS;
            for (int k = 0; k < nb; ++k) {
                const bool mine = k % nshare == crank;
                const int nbk = min(CT_NB, r - k * CT_NB);
                const float* sD = diag_buf(k);
                if (mine) {
                    ct_bar_sync(CT_BAR_READY, CT_THREADS);
                    float piv[2] = {1.f, 1.f};
                    ct_diag_block<32>(diag_buf(k), smem + CT_OFF_D, nbk, dw, lane, piv);
                    if (dw == 0) {
                        float mn, mx;
                        ct_pivot_range(piv, nbk, lane, mn, mx);
                        if (lane == 0) { gstat[k] = mn; gstat[CT_MAX_BLOCKS + k] = mx; }
                    }
                    // X_k for the panels (in the unused diagonal tile of L's image)
                    unsigned char* xd = l_tile(k, k);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int q = dt + 128 * e, row = q / 8, ch = q % 8;
                        const float4 u = *reinterpret_cast<const float4*>(sD + row * CT_LDD + ch * 8);
                        const float4 w4 = *reinterpret_cast<const float4*>(sD + row * CT_LDD + ch * 8 + 4);
                        float v[8] = {u.x, u.y, u.z, u.w, w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (ch * 8 + i > row || row >= nbk) v[i] = 0.f;
                        uint4 t0, t1;
                        split8(v, t0, t1);
                        const int o = row * 128 + img_chunk_offset(row, ch);
                        *reinterpret_cast<uint4*>(xd + o) = t0;
                        *reinterpret_cast<uint4*>(xd + term + o) = t1;
                    }
                }
                if (MULTI) {
                    if (k) cluster_wait();                  // (the arrival of the column before)
                    cluster_sync_all();
                } else {
                    ct_bar_arrive(CT_BAR_X, CT_THREADS);
                }
                if (mine) {
                    // and X_k^T, the diagonal tile of the L^{-T} image
                    unsigned char* xt = x_tile(k, k);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int q = dt + 128 * e, row = q % 64, ch = q / 64;
                        float v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int col = ch * 8 + i;
                            v[i] = sD[col * CT_LDD + row];
                            if (row > col || col >= nbk) v[i] = 0.f;
                        }
                        uint4 t0, t1;
                        split8(v, t0, t1);
                        if (a.pass >= 2 && row / 8 == ch && row < nbk) gscale[k * CT_NB + row] = ct_diag_scale(v, t0, t1, row % 8);
                        const int o = row * 128 + img_chunk_offset(row, ch);
                        *reinterpret_cast<uint4*>(xt + o) = t0;
                        *reinterpret_cast<uint4*>(xt + term + o) = t1;
                    }
                }
                if (MULTI) cluster_arrive();
                else ct_bar_arrive(CT_BAR_XT + (k & 1), CT_THREADS);
            }
            if (MULTI) cluster_wait();
        }
        __syncthreads();
        // every CTA reads the same statistics and takes the same branch
        bool fail = false;
        float mn = 3.0e38f, mx = 0.f;
        for (int k = 0; k < nb; ++k) {
            const float lo = __ldcg(gstat + k);
            if (!(lo > 0.f)) fail = true;
            mn = fminf(mn, lo);
            mx = fmaxf(mx, __ldcg(gstat + CT_MAX_BLOCKS + k));
        }
        const bool ill = (a.pass == 1) && (mx > a.cond_limit * mn);
        if (!fail && !(ill && attempt == 0)) {
            ok = true;
        } else if (attempt == 0 && a.pass == 1) {
            if (tid == 0 && crank == 0) atomicOr(w.status, shift_bit);
            phase_sync();                          // all have read the statistics before they are written again
        }
    }
    if (!ok && tid == 0 && crank == 0) atomicOr(w.status, ST_RANKDEF);
}

}  // namespace od
