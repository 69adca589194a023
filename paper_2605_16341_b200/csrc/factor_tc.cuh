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
// 64 x 64 block in fp32 (below) while the eight product warps do the S sums of
// the same block column, which do not depend on it; the tile below the diagonal goes first, together
// with the next diagonal block's own sum, so that the chain never waits for the rest.  64-wide
// blocks instead of 32: half the barriers.
// Measured, factor stage of a step (six launches, ms), before (32-wide blocks, fp32 tiles split at every
// use, a pairwise inversion afterwards) -> now: one matrix r = 256 0.74 -> 0.21, r = 512
// 1.47 -> 0.32, r = 1024 3.68 -> 0.68; 56 matrices at r = 512 2.7 -> 0.7, 154 of them 5.0 -> 1.5.
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
constexpr int CT_LDS = 65;                    // transposing buffer of the first-order inverse
// dynamic shared memory: two stages of an A tile and a B tile, then the diagonal block's work area
constexpr int CT_OFF_D = 4 * CT_TILE;
constexpr int CT_DG_BLK = CT_NB * CT_LDD * 4;                  // work area of a diagonal block: the block itself, a panel's 8 x 8 block
constexpr int CT_DG_BYTES = CT_DG_BLK + 64 * 4;
constexpr int CT_OFF_D2 = CT_OFF_D + CT_DG_BYTES;              // the block of the odd columns (the even ones': CT_OFF_D)
constexpr int CT_SMEM_BYTES = CT_OFF_D2 + CT_NB * CT_LDD * 4 + 1024;     // + alignment of the tiles
static_assert(2 * (CT_SMEM_BYTES + 2048) <= 228 * 1024, "two CTAs per multiprocessor");
static_assert(3 * CT_NB * CT_LDS * 4 <= 4 * CT_TILE, "three transposing buffers fit the operand stages");
constexpr int CT_MAX_BLOCKS = 64;             // r <= 4096
constexpr int CT_STAT_FLOATS = 3 * CT_MAX_BLOCKS;   // per block: smallest and largest pivot, row-sum bound
constexpr float CT_THIRD_PASS_LIMIT = 0.02f; // bound on |Gram - I|_2 of the second pass above which a third follows
constexpr float CT_SERIES_LIMIT = 1.4e-3f;   // bound on |Gram - I|_2 below which L^{-1} = I - Phi(E) is used

__device__ __forceinline__ void ct_bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void ct_bar_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// named barriers (0: the whole CTA); CT_BAR_XT: two, by the parity of the column
constexpr int CT_BAR_MMA = 1, CT_BAR_DIAG = 2, CT_BAR_READY = 3, CT_BAR_X = 4, CT_BAR_XT = 5, CT_BAR_HAND = 7;

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
__device__ __forceinline__ void ct_ldsm4t(uint32_t (&v)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
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
// the same with B given transposed: acc += A B, B's rows (depth) in memory order
__device__ __forceinline__ void ct_tile_mma_nt(float (&acc)[4][4], uint32_t a_tile, uint32_t b_tile, int warp, int lane) {
    const int l8 = lane & 7;
    const uint32_t a_row = a_tile + ((warp % 4) * 16 + l8 + ((lane >> 3) & 1) * 8) * 128;
    const uint32_t b_row = b_tile + (l8 + ((lane >> 3) & 1) * 8) * 128;
    const int a_ch = lane >> 4;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        const uint32_t ao = (uint32_t)(((2 * ks + a_ch) ^ l8) << 4);
        uint32_t ah[4], al[4];
        ct_ldsm4(ah, a_row + ao);
        ct_ldsm4(al, a_row + CT_TERM + ao);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t bo = (uint32_t)(ks * 2048 + ((((warp / 4) * 4 + 2 * h + (lane >> 4)) ^ l8) << 4));
            uint32_t bh[4], bl[4];
            ct_ldsm4t(bh, b_row + bo);
            ct_ldsm4t(bl, b_row + CT_TERM + bo);
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

// ---- diagonal blocks (fp32, four warps) ----------------------------------------------------------
// sD (64 x 64 block, ld CT_LDD, beyond nbk a diagonal of the matrix's first pivot; row by row the lower part
// counts) -> X^T = L^{-T}, L its Cholesky factor, in the upper part of sD; out(row, chunk, z) gets the entries
// 8 chunk .. + 7 of every row as they are found (zeros left of the diagonal).
//
// As in the large, [D; I] L^{-T} = [L; L^{-T}]: rows of the block and of the identity go through the same
// elimination, in panels of eight columns.  Row i of the block is done with its own panel, and row i of the identity begins
// there: 64 row slots in place, a thread each.  Two warps form the chain: every lane factors the panel's 8 x 8 diagonal
// block for itself (eight reciprocal square roots one after the other, no shuffle), solves its row's eight
// entries and brings the next panel's columns of its row up to date.  Two warps follow with the columns behind those, and
// with the output.
// What bounds it is the chain and, no less, the instruction cache: a CTA of a cluster comes here once or twice in a
// factorisation, so the code is fetched as it is run.  Hence one loop over the panels, and one over the columns, of
// some 600 instructions together.  (Straight-line halves of 32 columns with every lane's row in registers: 9300 cycles alone
// and warm, but 23000 in the kernel and 42000 for the first block.)  Step, that form -> this, with the Gram entries
// of the next diagonal block fetched before the wait for the inverse: 4096 x 4096 r = 256 0.483 -> 0.423 ms, column shard 4096 x
// 3584 r = 512 0.845 -> 0.775, 11008 x 4096 r = 1024 1.885 -> 1.811, one-kernel QR 520 x 384 r = 64 0.1095 -> 0.1011, fp32
// engine 1023 x 777 r = 40 0.244 -> 0.229.
// Pivots are normal numbers here: the form of rsqrt that takes subnormal ones costs the chain three more
// dependent instructions per column.  A Gram matrix so small that its pivots may be subnormal (squared column
// norms of the factor below 2^-60) comes into sD times CT_TINY_UP, and `unit`, the root of that, in place of the
// identity's ones takes it out of the inverse again.  (Free: multiplying the entries of X^T as they leave cost 4 of
// 480 us at 4096 x 4096, r = 256.  A subnormal pivot in a Gram matrix of ordinary size means an
// ill-conditioned one, and fails.)
constexpr float CT_TINY_TRACE = 8.67361738e-19f;          // 2^-60
constexpr float CT_TINY_UP = 1.20892582e24f;              // 2^80
constexpr float CT_TINY_UP_ROOT = 1.09951163e12f;         // 2^40
__device__ __forceinline__ float ct_rsqrt(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void ct_ld8(float (&v)[8], const float* p) {
    const float4 x = *reinterpret_cast<const float4*>(p), y = *reinterpret_cast<const float4*>(p + 4);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
}
__device__ __forceinline__ void ct_st8(float* p, const float (&v)[8]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
// the lane's row entries z -> its entries of [L; L^{-T}]; blk: the panel's 8 x 8 diagonal block
__device__ __forceinline__ void ct_panel8(const float* blk, float (&z)[8], float& dmin, float& dmax) {
    float b[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c <= i; c += 4) {
            const float4 v = *reinterpret_cast<const float4*>(blk + i * 8 + c);
            b[i][c] = v.x; b[i][c + 1] = v.y; b[i][c + 2] = v.z; b[i][c + 3] = v.w;
        }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float d = b[j][j], inv = ct_rsqrt(d);
        dmin = d > 0.f ? fminf(dmin, d) : -1.f;              // (a breakdown stays: -1 is the smallest from then on)
        dmax = fmaxf(dmax, d);
        z[j] *= inv;
#pragma unroll
        for (int i = j + 1; i < 8; ++i) {
            const float l = b[i][j] * inv;
            b[i][j] = l;
            z[i] = fmaf(-z[j], l, z[i]);
        }
#pragma unroll
        for (int i = j + 1; i < 8; ++i)
#pragma unroll
            for (int c = j + 1; c <= i; ++c) b[i][c] = fmaf(-b[i][j], b[c][j], b[i][c]);
    }
}
// a[0 .. 3] -= sum_j z_j L(c .. c + 3, j), the rows of L eight entries each, CT_LDD apart
__device__ __forceinline__ void ct_rank8(float* a, const float (&z)[8], const float* L) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float l[8];
        ct_ld8(l, L + c * CT_LDD);
#pragma unroll
        for (int j = 0; j < 8; ++j) a[c] = fmaf(-z[j], l[j], a[c]);
    }
}
// `blk`: 64 floats of shared memory.  dmin, dmax: smallest (-1: breakdown) and largest pivot, in every lane of warps 0
// and 1.  unit: 1, or what ct_rsqrt says.  Called by four warps (dw).
template <class Out>
__device__ __forceinline__ void ct_diag_block(float* sD, float* blk, int nbk, float unit, int dw, int lane, float& dmin, float& dmax, Out out) {
    const int np = (nbk + 7) / 8, row = (dw & 1) * 32 + lane, own = row / 8;
    float* sR = sD + row * CT_LDD;
    dmin = 3.0e38f; dmax = 0.f;
    if (dw < 2) {
        float z[8];
        ct_ld8(z, sR);
        if (own == 0) ct_st8(blk + row * 8, z);
        ct_bar_sync(CT_BAR_DIAG, 64);
#pragma unroll 1
        for (int p = 0; p < np; ++p) {
            if (own == p) {                 // the identity's row begins
#pragma unroll
                for (int c = 0; c < 8; ++c) z[c] = row % 8 == c ? unit : 0.f;
            }
            ct_panel8(blk, z, dmin, dmax);
            ct_st8(sR + 8 * p, z);
            ct_bar_sync(CT_BAR_HAND, 128);
            if (p + 1 < np) {
                float a[8] = {};
                if (own != p) ct_ld8(a, sR + 8 * (p + 1));
                const float* L = sD + 8 * (p + 1) * CT_LDD + 8 * p;
                ct_rank8(a, z, L);
                ct_rank8(a + 4, z, L + 4 * CT_LDD);
                if (own == p + 1) ct_st8(blk + (row % 8) * 8, a);
#pragma unroll
                for (int c = 0; c < 8; ++c) z[c] = a[c];
                ct_bar_sync(CT_BAR_DIAG, 64);
            }
        }
    } else {
#pragma unroll 1
        for (int p = 0; p < np; ++p) {
            ct_bar_sync(CT_BAR_HAND, 128);
            float z[8];
            ct_ld8(z, sR + 8 * p);
#pragma unroll 1
            for (int c = 8 * (p + 2); c < 8 * np; c += 4) {
                const float4 v = own == p ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<const float4*>(sR + c);
                float a[4] = {v.x, v.y, v.z, v.w};
                ct_rank8(a, z, sD + c * CT_LDD + 8 * p);
                *reinterpret_cast<float4*>(sR + c) = make_float4(a[0], a[1], a[2], a[3]);
            }
            if (own > p) {
#pragma unroll
                for (int c = 0; c < 8; ++c) z[c] = 0.f;
            }
            out(row, p, z);
        }
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

// (Two CTAs per multiprocessor leave 80 registers a thread: ptxas reports 20 bytes of spill stores and 60 of loads,
// 104 and 96 in the MULTI form.)
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
    unsigned char* limg = scr + (int64_t)w.aux1 * 1024;
    auto l_tile = [&](int t, int c) { return limg + ((int64_t)c * a.img.rows_pad + (int64_t)t * CT_NB) * 128; };
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
    // same 256-column block; and a last diagonal tile that is written in part
    for (int t = crank; t < nb; t += nshare)
        for (int c = t & ~3; c < t + (t * CT_NB + CT_NB > r ? 1 : 0); ++c) {
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
    // Z[t, k] = acc X_k^T, left in the A slot of stage ^ 1
    auto panel = [&](float (&acc)[4][4], int k) {
        load_tile(b_slot(stage), x_tile(k, k));
        ct_cp_commit();
        ct_store_tile(a_slot(stage), acc, warp, lane);
        ct_cp_wait_all();
        ct_bar_sync(CT_BAR_MMA, CT_MMA_THREADS);
        float o[4][4] = {};
        ct_tile_mma_nt(o, a_slot(stage), b_slot(stage), warp, lane);
        ct_store_tile(a_slot(stage ^ 1), o, warp, lane);
        ct_bar_sync(CT_BAR_MMA, CT_MMA_THREADS);
    };
    // ... and from there to its image
    auto panel_out = [&](int t, int k) {
        unsigned char* dst = t < k ? x_tile(t, k) : l_tile(t, k);
        const unsigned char* src = smem + (size_t)(stage ^ 1) * 2 * CT_TILE;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int q = (tid + CT_MMA_THREADS * e) * 16;
            *reinterpret_cast<uint4*>(dst + q) = *reinterpret_cast<const uint4*>(src + q);
            *reinterpret_cast<uint4*>(dst + term + q) = *reinterpret_cast<const uint4*>(src + CT_TERM + q);
        }
    };
    // d <- diagonal block k of the Gram matrix less d, the diagonal itself from gdiag (+ shift); beyond r the matrix's first
    // pivot on the diagonal, which changes neither the smallest nor the largest (a one would: it is not of the matrix's scale)
    auto diag_base = [&](float (&d)[4][4], int k, float shift) {
        const float pad = __ldcg(gdiag) + shift;
#pragma unroll
        for (int nf = 0; nf < 4; ++nf)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int il = mrow + 8 * (e / 2), jl = mcol + nf * 8 + (e % 2);
                const int i = k * CT_NB + il, j = k * CT_NB + jl;
                float v = il == jl ? pad : 0.f;
                if (i < r && j < r) v = (il == jl ? __ldcg(gdiag + i) + shift : A[(int64_t)i * r + j]) - d[nf][e];
                d[nf][e] = v;
            }
    };
    // the work area of diagonal block k <- d - z
    auto diag_store = [&](const float (&d)[4][4], const float (&z)[4][4], int k) {
        float* sD = diag_buf(k);
        const float up = trace < CT_TINY_TRACE ? CT_TINY_UP : 1.f;         // see ct_rsqrt
#pragma unroll
        for (int nf = 0; nf < 4; ++nf)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2*>(sD + (mrow + 8 * h) * CT_LDD + mcol + nf * 8) =
                    make_float2((d[nf][2 * h] - z[nf][2 * h]) * up, (d[nf][2 * h + 1] - z[nf][2 * h + 1]) * up);
    };

    bool ok = false;
    const int max_attempts = (a.pass == 1) ? 2 : 1;
    for (int attempt = 0; attempt < max_attempts && !ok; ++attempt) {
        const float shift = attempt ? a.shift_rel * trace : 0.f;
        if (mma_role) {
            if (crank == 0) {
                const float none[4][4] = {};
                float d[4][4] = {};
                diag_base(d, 0, shift);
                diag_store(d, none, 0);
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
                    if (next) diag_base(accd, k + 1, shift);
                }
                // X_k is in memory
                if (MULTI) cluster_sync_all();
                else ct_bar_sync(CT_BAR_X, CT_THREADS);
                if (first) {
                    panel(acc, k);
                    if (next) {
                        // the chain goes on before anything else
                        const uint32_t z = a_slot(stage ^ 1);
                        float dz[4][4] = {};
                        ct_tile_mma(dz, z, z, warp, lane);
                        diag_store(accd, dz, k + 1);
                        ct_bar_arrive(CT_BAR_READY, CT_THREADS);
                    }
                    panel_out(t, k);
                    t = next ? crank : t + nshare;
                    seek();
                    for (; t < nb;) {
                        if (t > k) prefetch_gram(t, k);
#pragma unroll
                        for (int nf = 0; nf < 4; ++nf)
#pragma unroll
                            for (int e = 0; e < 4; ++e) acc[nf][e] = 0.f;
                        sum_products(acc, accd, t, k, false);
                        finish_sum(acc, t, k);
                        panel(acc, k);
                        panel_out(t, k);
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
            const int dw = warp - CT_MMA_WARPS;
            for (int k = 0; k < nb; ++k) {
                const bool mine = k % nshare == crank;
                const int nbk = min(CT_NB, r - k * CT_NB);
                if (mine) {
                    ct_bar_sync(CT_BAR_READY, CT_THREADS);
                    // X_k^T goes to the diagonal tile of the L^{-T} image, chunk by chunk, while it is being found
                    unsigned char* xt = x_tile(k, k);
                    auto out = [&](int row, int ch, const float (&z)[8]) {
                        float v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] = row < nbk && ch * 8 + i < nbk ? z[i] : 0.f;
                        uint4 t0, t1;
                        split8(v, t0, t1);
                        if (a.pass >= 2 && row / 8 == ch && row < nbk) gscale[k * CT_NB + row] = ct_diag_scale(v, t0, t1, row % 8);
                        const int o = row * 128 + img_chunk_offset(row, ch);
                        *reinterpret_cast<uint4*>(xt + o) = t0;
                        *reinterpret_cast<uint4*>(xt + term + o) = t1;
                    };
                    float mn, mx;
                    ct_diag_block(diag_buf(k), reinterpret_cast<float*>(smem + CT_OFF_D + CT_DG_BLK), nbk,
                                  trace < CT_TINY_TRACE ? CT_TINY_UP_ROOT : 1.f, dw, lane, mn, mx, out);
                    // statistics: squared diagonal entries of L
                    if (lane == 0 && dw == 0) {
                        if (!(mx <= 3.0e38f)) mn = -1.f;
                        gstat[k] = mn;
                        gstat[CT_MAX_BLOCKS + k] = mx;
                    }
                }
                if (MULTI) {
                    if (k) cluster_wait();                  // (the arrival of the column before)
                    cluster_sync_all();
                } else {
                    ct_bar_arrive(CT_BAR_X, CT_THREADS);
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
        const bool ill = (a.pass == 1) && (sqrtf(mx) > a.cond_limit * sqrtf(mn));
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
