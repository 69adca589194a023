// r x r factor kernel of the tensor-core engine: Cholesky factor of the Gram matrix and its explicit
// inverse, one matrix per thread-block cluster (of one CTA in calls with many matrices).
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
// 64 x 64 come in by cp.async up to three steps ahead (one in the two-stage form).
//
// What bounds it: the chain of r / 64 diagonal blocks.  Four extra warps per CTA factor and invert a
// 64 x 64 block in fp32 (below) while the eight product warps do the S sums of the same block column, which do not
// depend on it.  The tile below the diagonal goes first, and the next diagonal block's own sum is kept up column by
// column, so that the chain (block 10000 cycles, barrier 1000, panel 2400, next block's last product 1300)
// never waits for the rest.  One CTA per multiprocessor: 164 registers a thread without spills and four operand stages (two
// CTAs with 80 registers and two stages: 25000 cycles a block column at r = 1024, where a sum of 15 tiles took
// longer than the chain).  Step, before all this -> now: 4096 x 4096 r = 256 0.423 -> 0.412 ms, column shard 4096 x 3584 r = 512
// 0.775 -> 0.730, 11008 x 4096 r = 1024 1.811 -> 1.687, 28 matrices 1000 wide at r = 272 1.65 -> 1.61; the 1.1B and 8B
// groups (one CTA per matrix) as before.
//
// The later passes of a CholeskyQR see a Gram matrix I + E with E tiny; when a rigorous bound on
// |E|_2 is small enough, L^{-1} = I - Phi(E) (first order) replaces the factorisation.
//
// The row tiles are dealt out over the CTAs of the cluster (tile t to CTA t mod size); the
// matrix stays in global memory (L2), phases are separated by release/acquire cluster barriers, and
// what another CTA may have written is read past L1.  Per tile the arithmetic and its order do not depend on the size of
// the cluster: a matrix gets the same bits with any.  Decisions that steer control
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
// dynamic shared memory: the operand stages, then the diagonal block's work area
constexpr int CT_STAGES = 4;                  // operand stages, an A tile and a B tile each (a power of two)
constexpr int CT_DG_BLK = CT_NB * CT_LDD * 4;                  // work area of a diagonal block: the block itself, a panel's 8 x 8 block
constexpr int CT_DG_BYTES = CT_DG_BLK + 64 * 4;
// the block of the even columns after the stages, that of the odd ones after its work area; + alignment of the tiles
__host__ __device__ constexpr int ct_smem_bytes(int stages) { return stages * 2 * CT_TILE + CT_DG_BYTES + CT_NB * CT_LDD * 4 + 1024; }
static_assert(2 * (ct_smem_bytes(2) + 2048) <= 228 * 1024, "two CTAs per multiprocessor with two stages");
static_assert(6 * CT_NB * CT_LDS * 4 <= CT_STAGES * 2 * CT_TILE, "six transposing buffers fit the operand stages");
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
// named barriers (0: the whole CTA; CT_BAR_MMA + 1 and + 2 also serve the thread groups of the first-order inverse)
constexpr int CT_BAR_MMA = 1, CT_BAR_DIAG = 2, CT_BAR_READY = 3, CT_BAR_HAND = 4;

__device__ __forceinline__ void ct_cp16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void ct_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void ct_cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
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
// counts) -> X^T = L^{-T}, L its Cholesky factor, in the upper part of sD and, with xt, as the two terms (`term` bytes
// apart) of an image tile, row chunk by row chunk as the entries are found.
//
// As in the large, [D; I] L^{-T} = [L; L^{-T}]: rows of the block and of the identity go through the same
// elimination, in panels of eight columns.  Row i of the block is done with its own panel, and row i of the identity begins
// there: 64 row slots in place, a thread each.  Two warps form the chain: every lane factors the panel's 8 x 8 diagonal
// block for itself (eight reciprocal square roots one after the other, no shuffle), solves its row's eight
// entries and brings the next panel's columns of its row up to date.  Two warps follow with the columns behind those, and
// with the output.
// What bounds it is the chain and, no less, the instruction cache: a CTA of a cluster comes here once or twice in a
// factorisation, so the code is fetched as it is run.  Hence one loop over the panels, and one over the columns, of
// some 600 instructions together, and the trial run ahead of time in factor_kernel.  (Straight-line halves of 32 columns with every lane's row in registers: 9300 cycles alone
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

// d_off, blk_off: byte offsets of sD and of 64 more floats in dynamic shared memory.  gscale: corrections of the rounded
// diagonal, or null.  Returns the smallest (-1: breakdown) and the largest pivot in every lane of warps 0 and 1.  unit: 1,
// or what ct_rsqrt says.  Called by four warps (dw).  (Not inlined, 16500 cycles a block in place of 13000.)
__device__ __forceinline__ float2 ct_diag_block(uint32_t d_off, uint32_t blk_off, int nbk, float unit, int dw, int lane,
                                             unsigned char* xt, int64_t term, float* gscale) {
    extern __shared__ __align__(16) unsigned char ct_dyn_smem[];
    float* sD = reinterpret_cast<float*>(ct_dyn_smem + d_off);
    float* blk = reinterpret_cast<float*>(ct_dyn_smem + blk_off);
    const int np = (nbk + 7) / 8, row = (dw & 1) * 32 + lane, own = row / 8;
    float* sR = sD + row * CT_LDD;
    float dmin = 3.0e38f, dmax = 0.f;
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
            for (int c = 8 * (p + 2); c < 8 * np; c += 8) {
                float a[8] = {};
                if (own != p) ct_ld8(a, sR + c);
                ct_rank8(a, z, sD + c * CT_LDD + 8 * p);
                ct_rank8(a + 4, z, sD + (c + 4) * CT_LDD + 8 * p);
                ct_st8(sR + c, a);
            }
            if (!xt) continue;
            // (beyond nbk the elimination has left the padding's part)
#pragma unroll
            for (int c = 0; c < 8; ++c) z[c] = own <= p && row < nbk && 8 * p + c < nbk ? z[c] : 0.f;
            uint4 t0, t1;
            split8(z, t0, t1);
            if (gscale && own == p && row < nbk) gscale[row] = ct_diag_scale(z, t0, t1, row % 8);
            const int o = row * 128 + img_chunk_offset(row, p);
            *reinterpret_cast<uint4*>(xt + o) = t0;
            *reinterpret_cast<uint4*>(xt + term + o) = t1;
        }
    }
    return make_float2(dmin, dmax);
}

// STAGES 4: one CTA per multiprocessor.  2: two, for one launch over more matrices than there are multiprocessors (154 at
// r = 512, factorisations of a step 1.71 -> 1.56 ms, 168 at r = 192 0.287 -> 0.226).  Not below that: 140 at r = 512 0.888 with one
// and 1.036 with two, 129 at r = 192 0.167 and 0.184, 148 at r = 272 0.316 and 0.358.
template <class BATCH, int STAGES>
__global__ void __launch_bounds__(CT_THREADS, STAGES == 4 ? 1 : 2)
factor_kernel(const __grid_constant__ BATCH batch, CholArgs a, int csize) {
    constexpr int CT_OFF_D = STAGES * 2 * CT_TILE, CT_OFF_D2 = CT_OFF_D + CT_DG_BYTES;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float red[CT_THREADS / 32];
    __shared__ int s_status;
    unsigned char* smem = smem_raw;
    {
        const uint32_t raw = static_cast<uint32_t>(__cvta_generic_to_shared(smem_raw));
        smem += ((raw + 1023u) & ~1023u) - raw;
    }
    const uint32_t smem0 = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    float* s_part = reinterpret_cast<float*>(smem);       // partial sums, before the operand stages are in use

    // the csize CTAs of a cluster (ranks 0 .. csize-1) share matrix blockIdx.x / csize
    const int crank = (int)(blockIdx.x % (unsigned)csize);
    const MatWork& w = batch.w[blockIdx.x / (unsigned)csize];
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const int r = a.r;
    const int nb = (r + CT_NB - 1) / CT_NB;
    const int shift_bit = a.which ? ST_SHIFT_R : ST_SHIFT_L;
    const bool mma_role = warp < CT_MMA_WARPS;

    const float* __restrict__ A = pick(w, a.gram);     // Gram matrix: never written here
    unsigned char* scr = reinterpret_cast<unsigned char*>(w.scratch);
    float* gdiag = reinterpret_cast<float*>(w.scratch + a.diag_off);      // r floats, then the block statistics
    float* gstat = reinterpret_cast<float*>(w.scratch + a.stat_off);
    float* gscale = reinterpret_cast<float*>(w.scratch + a.scale_off);
    const int64_t term = (int64_t)a.img.panels * a.img.rows_pad * 128;    // bytes between the terms of an image
    unsigned char* limg = scr + (int64_t)w.aux1 * 1024;
    auto l_tile = [&](int t, int c) { return limg + ((int64_t)c * a.img.rows_pad + (int64_t)t * CT_NB) * 128; };
    auto x_tile = [&](int t, int c) { return scr + a.img.off + ((int64_t)c * a.img.rows_pad + (int64_t)t * CT_NB) * 128; };
    float trace = 0.f;

    // All that comes before the factorisation.  False: there is nothing (more) to do.
    auto prepare = [&]() -> bool {
        if (tid == 0) s_status = *w.status;
        __syncthreads();
        // every CTA of the cluster has read the status word before any of them may change it
        cluster_sync_all();
        const int st0 = s_status;
        if (st0 & ST_FAILED) return false;
        if (a.pass == 3 && !(st0 & shift_bit)) return false;

        // ---- Gram diagonal (from the fp32 column sums of squares), by row tile --------------------
        // 24 interleaved partial sums per column, added in order: the order depends on the number of
        // partials only.  Loads go out eight at a time, whatever the remainder (one matrix of 11008 rows, r = 1024, with
        // a loop for the rest and a third of the threads per tile: 13300 cycles).
        if (a.use_colsq) {
            const float* cs = pick(w, a.colsq);
            const int nparts = w.aux0;
            const int g = tid / 16, q4 = (tid % 16) * 4;
            for (int t = crank; t < nb; t += csize) {
                const int col = t * CT_NB + q4;
                float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
                if (col < r) {
#pragma unroll 1
                    for (int kb = g; kb < nparts; kb += 8 * (CT_THREADS / 16)) {
                        float4 v[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const int k = kb + e * (CT_THREADS / 16);
                            v[e] = k < nparts ? *reinterpret_cast<const float4*>(cs + (int64_t)k * r + col) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
#pragma unroll
                        for (int e = 0; e < 8; ++e) { d.x += v[e].x; d.y += v[e].y; d.z += v[e].z; d.w += v[e].w; }
                    }
                }
                *reinterpret_cast<float4*>(s_part + g * 64 + q4) = d;
                __syncthreads();
                const int i = t * CT_NB + tid;
                if (tid < 64 && i < r) {
                    float sum = 0.f;
#pragma unroll
                    for (int q = 0; q < CT_THREADS / 16; ++q) sum += s_part[q * 64 + tid];
                    gdiag[i] = sum;
                    if (a.cnorm_off >= 0) reinterpret_cast<float*>(w.scratch + a.cnorm_off)[i] = sum;
                }
                __syncthreads();
            }
        } else {
            for (int t = crank; t < nb; t += csize)
                if (tid < 64 && t * CT_NB + tid < r) {
                    const int i = t * CT_NB + tid;
                    const float d = A[(int64_t)i * r + i];
                    gdiag[i] = d;
                    if (a.cnorm_off >= 0) reinterpret_cast<float*>(w.scratch + a.cnorm_off)[i] = d;
                }
        }
        cluster_sync_all();
        for (int i = tid; i < r; i += CT_THREADS) trace += __ldcg(gdiag + i);
        for (int o = 16; o; o >>= 1) trace += __shfl_xor_sync(0xffffffffu, trace, o);
        if (lane == 0) red[warp] = trace;
        __syncthreads();
        trace = 0.f;
        for (int i = 0; i < CT_THREADS / 32; ++i) trace += red[i];
        __syncthreads();
        // (the same sum in the same order in every CTA of a cluster: all of them take this exit or none)
        if (!(fabsf(trace) <= 3.0e38f)) {   // Inf or NaN
            if (tid == 0 && crank == 0) atomicOr(w.status, ST_NONFINITE);
            return false;
        }

        // Tiles of the L^{-T} image below its diagonal that the apply product reads as zeros: those inside the
        // same 256-column block; and a last diagonal tile that is written in part
        for (int t = crank; t < nb; t += csize)
            for (int c = t & ~3; c < t + (t * CT_NB + CT_NB > r ? 1 : 0); ++c) {
                unsigned char* dst = x_tile(t, c);
                for (int q = tid; q < 1024; q += CT_THREADS)
                    *reinterpret_cast<uint4*>(dst + (q >= 512 ? term : 0) + (q & 511) * 16) = make_uint4(0u, 0u, 0u, 0u);
            }
        if (a.pass < 2) return true;

        // ---- later passes of the QR: the Gram matrix is I + E with E small ------------------------
        // L = I + X with X + X^T + X X^T = E, so L^{-1} = I - Phi(E) + O(|E|^2), Phi = strict lower part
        // plus half the diagonal.  |E|_2 <= max row sum of |E| (E is symmetric); when that bound is
        // below CT_SERIES_LIMIT the dropped terms are below 2e-6 and the factorisation is skipped.
        for (int t = crank; t < nb; t += csize) {
            const int i0 = t * CT_NB, g = tid / 16, j4 = (tid % 16) * 4;
            float* s_row = s_part + 24 * 64;
            // left of the diagonal: 24 rows at a time, 16 threads along each, four loads under way
            for (int i = i0 + g; i < i0 + CT_NB; i += 24) {
                float s = 0.f;
                if (i < r)
#pragma unroll 1
                    for (int j0 = j4; j0 < i; j0 += 256) {
                        float4 v[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            v[e] = j0 + 64 * e < i ? *reinterpret_cast<const float4*>(A + (int64_t)i * r + j0 + 64 * e) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int j = j0 + 64 * e;
                            s += (j < i ? fabsf(v[e].x) : 0.f) + (j + 1 < i ? fabsf(v[e].y) : 0.f) + (j + 2 < i ? fabsf(v[e].z) : 0.f) +
                                 (j + 3 < i ? fabsf(v[e].w) : 0.f);
                        }
                    }
                const unsigned mask = 0xffffu << (lane & 16);
                for (int o = 8; o; o >>= 1) s += __shfl_xor_sync(mask, s, o);
                if (tid % 16 == 0) s_row[i - i0] = s;
            }
            // below the diagonal (the mirror of the row's right part): 24 row groups x 64 columns
            {
                const int j = i0 + j4;
                float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                if (j < r)
#pragma unroll 1
                    for (int ib = i0 + g; ib < r; ib += 24 * 8) {
                        float4 v[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            v[e] = ib + 24 * e < r ? *reinterpret_cast<const float4*>(A + (int64_t)(ib + 24 * e) * r + j) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const int i = ib + 24 * e;
                            s.x += i > j ? fabsf(v[e].x) : 0.f; s.y += i > j + 1 ? fabsf(v[e].y) : 0.f;
                            s.z += i > j + 2 ? fabsf(v[e].z) : 0.f; s.w += i > j + 3 ? fabsf(v[e].w) : 0.f;
                        }
                    }
                *reinterpret_cast<float4*>(s_part + g * 64 + j4) = s;
            }
            __syncthreads();
            if (warp == 0) {
                float mx = 0.f;
                for (int q = lane; q < 64 && i0 + q < r; q += 32) {
                    float s = fabsf(__ldcg(gdiag + i0 + q) - 1.f) + s_row[q];
#pragma unroll
                    for (int e = 0; e < 24; ++e) s += s_part[e * 64 + q];
                    mx = fmaxf(mx, s <= 3.0e38f ? s : 3.3e38f);
                }
                for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                if (lane == 0) gstat[2 * CT_MAX_BLOCKS + t] = mx;
            }
            __syncthreads();
        }
        cluster_sync_all();
        float mx = 0.f;
        for (int t = 0; t < nb; ++t) mx = fmaxf(mx, __ldcg(gstat + 2 * CT_MAX_BLOCKS + t));
        // Second pass with Q1 far from orthonormal (cond(Y)^2 u was not small): its result will
        // not be orthonormal to working accuracy either, so ask for the third pass.
        if (a.pass == 2 && !(mx <= CT_THIRD_PASS_LIMIT) && tid == 0 && crank == 0) atomicOr(w.status, shift_bit);
        // (a diagonal this close to one is held by its two terms to 2^-20: no correction)
        if (tid == 0 && crank == 0) gscale[r] = mx <= CT_SERIES_LIMIT ? 0.f : 1.f;
        if (!(mx <= CT_SERIES_LIMIT)) return true;
        // Image tiles (ta, tb), tb >= ta, of L^{-T}: entry (row, col) = -E(col, row) right of the
        // diagonal.  Three groups of four warps, each with two transposing buffers of its own (one where there is no room) and
        // the next tile's entries under way while it writes one.
        constexpr int NBUF = STAGES == 4 ? 2 : 1;
        const int grp = tid / 128, gt = tid % 128;
        float* bufs = reinterpret_cast<float*>(smem) + grp * NBUF * CT_NB * CT_LDS;
        const int pairs = nb * (nb + 1) / 2, step = 3 * csize;
        int ta = 0, tb = 0;
        float4 v[8];
        auto fetch = [&](int q) {                // tile q of the list, if there is one
            tb = 0;
            while (q > tb) { q -= tb + 1; ++tb; }
            ta = q;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int i = tb * CT_NB + gt / 16 + 8 * e, j = ta * CT_NB + (gt % 16) * 4;
                v[e] = i < r && j < r ? *reinterpret_cast<const float4*>(A + (int64_t)i * r + j) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        };
        int q = crank * 3 + grp, b = 0;
        if (q < pairs) fetch(q);
        for (; q < pairs; q += step, b ^= NBUF - 1) {
            if (NBUF == 1) ct_bar_sync(CT_BAR_MMA + grp, 128);       // (the one buffer has been read)
            float* buf = bufs + b * CT_NB * CT_LDS;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float* o = buf + (gt / 16 + 8 * e) * CT_LDS + (gt % 16) * 4;
                o[0] = v[e].x; o[1] = v[e].y; o[2] = v[e].z; o[3] = v[e].w;
            }
            const int ca = ta, cb = tb;
            ct_bar_sync(CT_BAR_MMA + grp, 128);
            if (q + step < pairs) fetch(q + step);
            unsigned char* dst = x_tile(ca, cb);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int row = gt / 8 + 16 * e, ch = gt % 8;
                const int gr = ca * CT_NB + row, gc = cb * CT_NB + ch * 8;
                float x[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) x[i] = gc + i > gr ? -buf[(ch * 8 + i) * CT_LDS + row] : 0.f;
                if (gr >= gc && gr < gc + 8 && gr < r) {
                    const float dg = 0.5f * (3.f - __ldcg(gdiag + gr));
#pragma unroll
                    for (int i = 0; i < 8; ++i) x[i] = gc + i == gr ? dg : x[i];
                }
                uint4 t0, t1;
                split8(x, t0, t1);
                const int o = row * 128 + img_chunk_offset(row, ch);
                *reinterpret_cast<uint4*>(dst + o) = t0;
                *reinterpret_cast<uint4*>(dst + term + o) = t1;
            }
        }
        return false;
    };

    // ---- factorisation and inverse ------------------------------------------------------------
    const int mrow = (warp % 4) * 16 + lane / 4, mcol = (warp / 4) * 32 + (lane % 4) * 2;     // first element of acc
    const uint32_t dyn0 = static_cast<uint32_t>(smem - smem_raw);
    auto diag_off = [&](int k) { return dyn0 + ((k & 1) ? CT_OFF_D2 : CT_OFF_D); };
    int stage = 0;                     // operand stage that the next load goes to
    auto slot = [&](int s) { return (s & (STAGES - 1)) * 2 * CT_TILE; };      // A tile, then B tile
    auto load_tile = [&](uint32_t dst, const unsigned char* src) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int q = (tid + CT_MMA_THREADS * e) * 16;
            ct_cp16(dst + q, src + q);
            ct_cp16(dst + CT_TERM + q, src + term + q);
        }
    };
    // acc += sum_{c < k} Z[t, c] L[k, c]^T, accd += sum_{d0 <= c < k} Z[t, c] Z[t, c]^T
    auto sum_products = [&](float (&acc)[4][4], float (&accd)[4][4], int t, int k, int d0) {
        const int c0 = t < k ? t : 0;
        auto load = [&](int c, int s) {
            if (c < k) {
                load_tile(smem0 + slot(s), t < k ? x_tile(t, c) : l_tile(t, c));
                load_tile(smem0 + slot(s) + CT_TILE, l_tile(k, c));
            }
            ct_cp_commit();
        };
        if (c0 >= k) return;
#pragma unroll
        for (int e = 0; e < STAGES - 1; ++e) load(c0 + e, stage + e);
#pragma unroll 1
        for (int c = c0; c < k; ++c) {
            ct_cp_wait<STAGES - 2>();
            ct_bar_sync(CT_BAR_MMA, CT_MMA_THREADS);
            load(c + STAGES - 1, stage + STAGES - 1);
            const uint32_t at = smem0 + slot(stage);
            ct_tile_mma(acc, at, at + CT_TILE, warp, lane);
            if (c >= d0) ct_tile_mma(accd, at, at, warp, lane);
            ++stage;
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
    // Z[t, k] = acc X_k^T, left in the A slot of the stage that is loaded last
    auto panel = [&](float (&acc)[4][4], int k) {
        const uint32_t at = smem0 + slot(stage);
        load_tile(at + CT_TILE, x_tile(k, k));
        ct_cp_commit();
        ct_store_tile(at, acc, warp, lane);
        ct_cp_wait<0>();
        ct_bar_sync(CT_BAR_MMA, CT_MMA_THREADS);
        float o[4][4] = {};
        ct_tile_mma_nt(o, at, at + CT_TILE, warp, lane);
        ct_store_tile(smem0 + slot(stage + STAGES - 1), o, warp, lane);
        ct_bar_sync(CT_BAR_MMA, CT_MMA_THREADS);
    };
    // ... and from there to its image
    auto panel_out = [&](int t, int k) {
        unsigned char* dst = t < k ? x_tile(t, k) : l_tile(t, k);
        const unsigned char* src = smem + slot(stage + STAGES - 1);
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
        float* sD = reinterpret_cast<float*>(smem_raw + diag_off(k));
        const float up = trace < CT_TINY_TRACE ? CT_TINY_UP : 1.f;         // see ct_rsqrt
#pragma unroll
        for (int nf = 0; nf < 4; ++nf)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2*>(sD + (mrow + 8 * h) * CT_LDD + mcol + nf * 8) =
                    make_float2((d[nf][2 * h] - z[nf][2 * h]) * up, (d[nf][2 * h + 1] - z[nf][2 * h + 1]) * up);
    };
    auto clear = [&](float (&d)[4][4]) {
#pragma unroll
        for (int nf = 0; nf < 4; ++nf)
#pragma unroll
            for (int e = 0; e < 4; ++e) d[nf][e] = 0.f;
    };

    grid_dependency_launch();
    bool ok = false, prepared = false;
    // The diagonal warps first run a block of three panels on whatever shared memory holds, while the kernel before is still
    // at work (where launches overlap) or while the first CTA of the cluster has the first block: their code then is in
    // the instruction cache (a block in the chain of one matrix: 19000 cycles the first and 13000 the others, 10000 either way so).
#pragma unroll 1
    for (int dry = a.pass == 1 && (a.ahead || crank) ? 1 : 0; dry >= 0; --dry) {
        if (!prepared && !(dry && a.ahead)) {
            grid_dependency_wait();
            if (!prepare()) return;
            prepared = true;
        }
        if (dry && mma_role) continue;
        const int max_attempts = (a.pass == 1 && !dry) ? 2 : 1;
        for (int attempt = 0; attempt < max_attempts && !ok; ++attempt) {
            const float shift = attempt ? a.shift_rel * trace : 0.f;
            if (mma_role) {
                // The next diagonal block of this CTA, dt: its sum is kept up with column by column, as the tiles of its
                // row are found (columns below dc are in accd), so that it does not lengthen the column that it is wanted in.
                float accd[4][4] = {};
                int dt = crank ? crank : csize, dc = 0;
                if (crank == 0) {
                    const float none[4][4] = {};
                    diag_base(accd, 0, shift);
                    diag_store(accd, none, 0);
                    ct_bar_arrive(CT_BAR_READY, CT_THREADS);
                    clear(accd);
                }
                for (int k = 0; k < nb; ++k) {
                    const bool next = k + 1 < nb && dt == k + 1;
                    // own tiles of this block column, the one below the diagonal first
                    int t = next ? k + 1 : crank;
                    auto seek = [&]() { while (t < nb && (t == k || (next && t == k + 1))) t += csize; };
                    if (!next) seek();
                    bool first = true;
                    do {
                        float acc[4][4] = {};
                        const bool on = t < nb, lead = first && next;
                        if (on) {
                            if (t > k) prefetch_gram(t, k);
                            sum_products(acc, accd, t, k, t == dt ? dc : k);
                            finish_sum(acc, t, k);
                            if (lead) diag_base(accd, k + 1, shift);
                        }
                        if (first) cluster_sync_all();                  // X_k is in memory
                        if (on) {
                            panel(acc, k);
                            const uint32_t z = smem0 + slot(stage + STAGES - 1);
                            if (lead) {
                                // the chain goes on before anything else
                                float dz[4][4] = {};
                                ct_tile_mma(dz, z, z, warp, lane);
                                diag_store(accd, dz, k + 1);
                                ct_bar_arrive(CT_BAR_READY, CT_THREADS);
                                clear(accd);
                                dt += csize; dc = 0;
                            } else if (t == dt) {
                                ct_tile_mma(accd, z, z, warp, lane);
                                dc = k + 1;
                            }
                            panel_out(t, k);
                            t = lead ? crank : t + csize;
                            seek();
                        }
                        first = false;
                    } while (t < nb);
                    cluster_sync_all();                                 // block column k is in memory
                }
            } else {
                // The four diagonal warps.  Block k + 1 is started as soon as the product warps have its sum, while they go
                // on with block column k: what they owe the barriers of column k is an arrival, not a wait.
                const int dw = warp - CT_MMA_WARPS;
                for (int k = 0; k < nb; ++k) {
                    if (dry || k % csize == crank) {
                        const int nbk = dry ? 24 : min(CT_NB, r - k * CT_NB);
                        if (!dry) ct_bar_sync(CT_BAR_READY, CT_THREADS);
                        // X_k^T goes to the diagonal tile of the L^{-T} image while it is being found
                        const float2 mm = ct_diag_block(diag_off(k), dyn0 + CT_OFF_D + CT_DG_BLK, nbk,
                                                        trace < CT_TINY_TRACE ? CT_TINY_UP_ROOT : 1.f, dw, lane, dry ? smem : x_tile(k, k),
                                                        dry ? CT_TERM : term, a.pass >= 2 ? gscale + k * CT_NB : nullptr);
                        if (dry) break;
                        // statistics: squared diagonal entries of L
                        if (lane == 0 && dw == 0) {
                            gstat[k] = mm.y <= 3.0e38f ? mm.x : -1.f;
                            gstat[CT_MAX_BLOCKS + k] = mm.y;
                        }
                    }
                    if (k) cluster_wait();                  // (the arrival of the column before)
                    cluster_sync_all();
                    cluster_arrive();
                }
                if (dry) break;
                cluster_wait();
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
                cluster_sync_all();                        // all have read the statistics before they are written again
            }
        }
    }
    if (!ok && tid == 0 && crank == 0) atomicOr(w.status, ST_RANKDEF);
}

}  // namespace od
