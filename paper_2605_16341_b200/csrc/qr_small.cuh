// QR of a tall-skinny factor at rank <= 64 in ONE kernel (both engines): one matrix per cluster, its rows
// dealt out over the CTAs and kept in shared memory.
//
//   load the rows (adding up the partial results of a depth-split product)
//   Gram matrix, Cholesky + inverse, rows <- rows * L^{-T}, twice (CholeskyQR2), a third time when flagged
//   write the factor and its operand images; for the right factor also R's images
// or, for column-normalised Dion, the column norms and one scaling.
//
// What bounds it: the chain Gram -> factor -> apply.  As kernels of their own (three per pass, three passes
// of which the last mostly finds nothing to do) each link cost 5 to 10 us of launch, set-up and
// first-load latency for less than 1 us of arithmetic at r <= 64.  Here a link is a cluster barrier.  All
// arithmetic is fp32 FMA: at r <= 64 the products are 2 % of the step's, and the operands are neither split
// nor packed on the way.  Every CTA factors the Gram matrix for itself (one diagonal block, the routine of
// factor_tc.cuh).
// The rows are cut into 1 to 16 parts by row count and rank only, the parts' Gram matrices are added as a
// balanced binary tree, and a CTA takes one part or a run of them: a call with many matrices uses fewer CTAs
// for each (they would all factor the same matrix again) and a matrix still gets the same bits alone and in any group.
// The diagonal block takes all of the 128 registers and puts 4 to 15 others away meanwhile (ptxas: 16 to 58 bytes of spill stores, none
// without the block); the batched loads of the rows spill nothing.
// Measured, both QRs of a step with their launches (23 -> 6 per step): one 256 x 512 fp32 matrix, r = 16: step
// 198 -> 67 us; 520 x 384, r = 64: 235 -> 115 us; 4096 x 4096, r = 32: 442 -> 240 us.
#pragma once
#include "factor_tc.cuh"

namespace od {

constexpr int QS_MAX_RANK = 64;
constexpr int QS_MAX_ROWS_64 = 640;
constexpr int QS_SMEM_LIMIT = 227 * 1024 - 256;      // less the static variables
constexpr int QS_SMEM_TWO = 228 * 1024 / 2 - 1024 - 256;     // up to here two CTAs of 256 threads share a multiprocessor
// Bound on |Gram - I|_2 below which L^{-1} = I - Phi(E) is used on the fp32 engine: the dropped terms, of order |E|^2, are
// then below 2^-26, a quarter of what rounding a 1 to fp32 loses.  (Below the tensor engine's CT_SERIES_LIMIT they reach 2e-6:
// nothing beside products good to 2^-16, several roundings here.)
constexpr float QS_SERIES_LIMIT_F32 = 1.22070312e-4f;      // 2^-13

struct QrSmallArgs {
    Sel src;                // rows x r fp32, or `splits` partial results split_stride floats apart
    int64_t split_stride;
    int32_t splits;
    int32_t rows, r, csize, parts_per_cta, rows_per_part;
    int32_t which;          // 0: left QR (P), 1: right factor (Q)
    int32_t colnorm;        // 1: column normalisation instead of the QR
    float shift_rel, cond_limit, series_limit;
    Sel dst;                // the factor, fp32
    ImgRef img;             // and its image
    int32_t img_planes;     // bit mask of the planes to write: 1 | 2 bf16 terms, 4 fp16
    // right factor: R itself, when `src` holds partial results (copy_r), and its image
    int32_t copy_r, r_planes;
    Sel r_dst;
    ImgRef r_img;
    int64_t rscale_off;     // r_planes & 4: where the inverse of the plane's scale goes
};

inline int qs_width(int r) { return r <= 16 ? 16 : (r <= 32 ? 32 : 64); }
inline int qs_row_bytes(int r) { return 4 * (r <= 16 ? 20 : (r <= 32 ? 32 : 68)); }
// partial Gram matrices of the thread groups, or a diagonal block
__host__ __device__ constexpr int qs_part_bytes(int threads) { return 64 * threads > CT_DG_BYTES ? 64 * threads : CT_DG_BYTES; }
inline int qs_fixed(int r, int threads) { return qs_part_bytes(threads) + qs_width(r) * qs_width(r) * 4; }

// Parts of a factor: 4096 row entries each (64 rows at r = 64, 256 at r = 16) while that gives at most max_ctas.
inline int qs_parts(int64_t rows, int r, int max_ctas) {
    const int64_t per = 4096 / qs_width(r);
    int c = 1;
    while (c < max_ctas && rows > per * c) c *= 2;
    return c;
}
inline int qs_rows_per_part(int64_t rows, int parts) { return (int)((rows + parts * 32 - 1) / (parts * 32) * 32); }
inline int64_t qs_smem(int64_t rows_per_cta, int r, int threads) { return rows_per_cta * qs_row_bytes(r) + qs_fixed(r, threads); }
// Threads of a CTA, by the plan only (they decide how a Gram matrix is summed): 512, one CTA per multiprocessor, for parts
// of 256 rows and more and for the fp32 engine above rank 32; else 256 and two.  Step with 256 and with 512 threads: 11008 x 4096 r = 32, Dion
// 0.324 and 0.315 ms, 14336 x 4096 r = 16 0.365 and 0.361; 360 x 360 r = 32 0.0629 and 0.0640; 1023 x 777 r = 40, fp32 engine, 0.103 and
// 0.099; 24 layers 640 wide at r = 64 1.21 and 1.28.  And 256 where the work area of 512 leaves the rows no room, up to 26112
// rows at r = 32 and 41984 at r = 16: against separate kernels, 39700 x 512 r = 16 0.350 -> 0.274 ms, 41984 x 2048 0.620 -> 0.533,
// 24320 x 512 r = 32 0.254 -> 0.239 (eight 25800 x 512 0.741 -> 0.759), 26112 x 512 r = 17 on the fp32 engine 0.868 -> 0.549.
inline int qs_threads(int64_t rows, int r, int max_ctas, bool fp32_engine) {
    const int per = qs_rows_per_part(rows, qs_parts(rows, r, max_ctas));
    return (r > 32 ? fp32_engine : per >= 256) && qs_smem(per, r, 512) <= QS_SMEM_LIMIT ? 512 : 256;
}
// Whether the kernel takes a rows x r factor.  From r = 33 up only short ones: the fp32 products and the repeated
// factorisations cost a call with many matrices more than the separate tensor-core kernels do, and the choice cannot
// depend on the call (a matrix gets the same bits alone and in a group).  Step with separate kernels and with this one
// at r = 64: 512 x 512 one 0.204 and 0.106 ms, 72 of them 0.383 and 0.321; 640 x 640 one 0.214 and 0.101, 24 0.285 and
// 0.189, 72 0.491 and 0.547; 768 x 768 one 0.220 and 0.100, 24 0.331 and 0.207, 72 0.556 and 0.612; 24 layers of a
// 768-wide model (168 matrices) 1.39 and 1.61; 4096 x 4096 one 0.336 and 0.263.
// The fp32 engine's separate kernels have no such side, at any number of matrices: 767 x 767 r = 40 one 0.217 and 0.091 ms, 24 0.702 and
// 0.494, 72 1.82 and 1.39, 168 3.98 and 2.99; r = 64 24 0.722 and 0.499, 168 4.00 and 3.02; 72 of 1400 x 1100 r = 40 4.57 and 3.31.  It
// takes whatever shared memory holds.
inline bool qs_fits(int64_t rows, int r, int max_ctas, bool fp32_engine) {
    if (r > QS_MAX_RANK || (r > 32 && rows > QS_MAX_ROWS_64 && !fp32_engine)) return false;
    const int c = qs_parts(rows, r, max_ctas);
    return qs_smem(qs_rows_per_part(rows, c), r, qs_threads(rows, r, max_ctas, fp32_engine)) <= QS_SMEM_LIMIT;
}
// CTAs per matrix in a call of `matrices`: the largest cluster of which all run at once.  room(size, per_sm): such clusters that
// the device holds.  (Counted in CTAs, 128 of 148 multiprocessors for eight matrices in clusters of 16, of which seven
// run at once: eight 4096 x 4096 at r = 32 104 us for both QRs, with two CTAs per multiprocessor 81.)
template <class Room>
inline int qs_ctas(int64_t rows, int r, int max_ctas, int matrices, int threads, Room room) {
    const int parts = qs_parts(rows, r, max_ctas), per = qs_rows_per_part(rows, parts);
    const int max_run = r > 32 ? 4 : 16;            // (tree levels held in registers)
    int c = parts;
    auto smem = [&](int ctas) { return qs_smem((int64_t)per * (parts / ctas), r, threads); };
    while (c > 1 && matrices > room(c, threads == 256 && smem(c) <= QS_SMEM_TWO ? 2 : 1) && parts / c < max_run && smem(c / 2) <= QS_SMEM_LIMIT)
        c /= 2;
    return c;
}

__device__ __forceinline__ float4 qs_ld_remote4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void qs_st_remote4(uint32_t addr, const float4& v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

template <class BATCH, int R, int QS_THREADS>
__global__ void __launch_bounds__(QS_THREADS, 512 / QS_THREADS)
qr_small_kernel(const __grid_constant__ BATCH batch, const __grid_constant__ QrSmallArgs a) {
    constexpr int LD = R == 32 ? 32 : R + 4;         // row stride: no bank conflicts in either product
    constexpr int TX = R / 4;                        // threads along the columns of a 4 x 4-blocked product
    constexpr int GROUPS = QS_THREADS / (TX * TX);   // Gram product: thread groups that share the rows
    constexpr int RT = QS_THREADS / TX * 4;          // apply product: rows of a step
    constexpr int ENT = R * R / 4 > QS_THREADS ? R * R / 4 / QS_THREADS : 1;             // Gram entries (in fours) per thread
    constexpr int LEVELS = R == 64 ? 3 : 5;
    extern __shared__ __align__(16) unsigned char smem[];
    float* sD = reinterpret_cast<float*>(smem);      // diagonal block's area; partial Gram matrices before it
    float* part = sD;
    float* G = reinterpret_cast<float*>(smem + qs_part_bytes(QS_THREADS));     // Gram matrix, then L^{-T}
    float* Y = G + R * R;                            // this CTA's rows
    __shared__ float s_min, s_max, s_bound;
    static_assert(GROUPS * R * R * 4 <= qs_part_bytes(QS_THREADS), "partial Gram matrices fit the diagonal block's area");

    grid_dependency();
    const int C = a.csize, crank = (int)(blockIdx.x % (unsigned)C);
    const MatWork& w = batch.w[blockIdx.x / (unsigned)C];
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const int r = a.r, r4 = r / 4;
    const int shift_bit = a.which ? ST_SHIFT_R : ST_SHIFT_L;
    const int st0 = *w.status;
    cluster_sync_all();          // every CTA has read the status word before one of them may change it
    if (st0 & ST_FAILED) return;

    const int rows_per_cta = a.rows_per_part * a.parts_per_cta;
    const int row0 = crank * rows_per_cta;
    const int nrows = max(0, min(rows_per_cta, a.rows - row0));

    // ---- rows -> shared memory ----
    {
        const float* S = pick(w, a.src) + (int64_t)row0 * r;
        float* Rd = a.copy_r ? pick(w, a.r_dst) + (int64_t)row0 * r : nullptr;
        const int total = nrows * (R / 4);
        if (r % 4) {                // (fp32 engine)
            for (int q = tid; q < nrows * R; q += QS_THREADS) Y[q / R * LD + q % R] = q % R < r ? S[q / R * r + q % R] : 0.f;
        } else {
            // four chunks of four columns, two partial results of each under way (one after the other, 11008 rows at r = 32
            // in five parts took 40 us)
            for (int q0 = tid; q0 < total; q0 += 4 * QS_THREADS) {
                float4 v[4];
#pragma unroll 1
                for (int p = 0; p < a.splits; p += 2) {
                    float4 u[4][2];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int q = q0 + e * QS_THREADS, i = q / (R / 4), c = q % (R / 4);
                        const bool in = q < total && c < r4;
                        const float* s = S + p * a.split_stride + i * r + c * 4;
                        u[e][0] = in ? *reinterpret_cast<const float4*>(s) : make_float4(0.f, 0.f, 0.f, 0.f);
                        u[e][1] = in && p + 1 < a.splits ? *reinterpret_cast<const float4*>(s + a.split_stride) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (p == 0) v[e] = u[e][0];
                        else { v[e].x += u[e][0].x; v[e].y += u[e][0].y; v[e].z += u[e][0].z; v[e].w += u[e][0].w; }
                        v[e].x += u[e][1].x; v[e].y += u[e][1].y; v[e].z += u[e][1].z; v[e].w += u[e][1].w;
                    }
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int q = q0 + e * QS_THREADS, i = q / (R / 4), c = q % (R / 4);
                    if (q >= total) continue;
                    if (Rd && c < r4) *reinterpret_cast<float4*>(Rd + i * r + c * 4) = v[e];
                    *reinterpret_cast<float4*>(Y + i * LD + c * 4) = v[e];
                }
            }
        }
    }
    __syncthreads();

    // G <- Gram matrix of all rows, the same bits in every CTA
    auto gram = [&]() {
        const int g = tid / (TX * TX), t = tid % (TX * TX), ty = t / TX, tx = t % TX;
        float4 level[LEVELS][ENT];                   // binary counter of part sums: level l holds 2^l parts
        for (int v = 0; v < a.parts_per_cta; ++v) {
            float acc[4][4] = {};
            const int end = min(nrows, (v + 1) * a.rows_per_part);
#pragma unroll 4
            for (int k = v * a.rows_per_part + g; k < end; k += GROUPS) {
                const float4 x = *reinterpret_cast<const float4*>(Y + k * LD + ty * 4);
                const float4 y = *reinterpret_cast<const float4*>(Y + k * LD + tx * 4);
                const float xa[4] = {x.x, x.y, x.z, x.w}, yb[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int f = 0; f < 4; ++f) acc[e][f] = fmaf(xa[e], yb[f], acc[e][f]);
            }
            if (v) __syncthreads();                  // the previous part's sums have been taken
#pragma unroll
            for (int e = 0; e < 4; ++e)
                *reinterpret_cast<float4*>(part + (g * R + ty * 4 + e) * R + tx * 4) = make_float4(acc[e][0], acc[e][1], acc[e][2], acc[e][3]);
            __syncthreads();
            float4 cur[ENT];
#pragma unroll
            for (int n = 0; n < ENT; ++n) {
                const int q = tid + n * QS_THREADS;
                cur[n] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (q < R * R / 4) {
#pragma unroll
                    for (int gg = 0; gg < GROUPS; ++gg) {
                        const float4 u = *reinterpret_cast<const float4*>(part + gg * R * R + q * 4);
                        cur[n].x += u.x; cur[n].y += u.y; cur[n].z += u.z; cur[n].w += u.w;
                    }
                }
            }
            bool carry = true;
#pragma unroll
            for (int l = 0; l < LEVELS; ++l) {
                if (!carry) continue;
                if ((v >> l) & 1) {
#pragma unroll
                    for (int n = 0; n < ENT; ++n) {
                        cur[n].x = level[l][n].x + cur[n].x; cur[n].y = level[l][n].y + cur[n].y;
                        cur[n].z = level[l][n].z + cur[n].z; cur[n].w = level[l][n].w + cur[n].w;
                    }
                } else {
#pragma unroll
                    for (int n = 0; n < ENT; ++n) level[l][n] = cur[n];
                    carry = false;
                }
            }
        }
        // parts_per_cta is a power of two: its sum sits at that level
        __syncthreads();
#pragma unroll
        for (int l = 0; l < LEVELS; ++l)
            if (a.parts_per_cta == (1 << l)) {
#pragma unroll
                for (int n = 0; n < ENT; ++n) {
                    const int q = tid + n * QS_THREADS;
                    if (q < R * R / 4) *reinterpret_cast<float4*>(part + q * 4) = level[l][n];
                }
            }
        cluster_sync_all();
        // this CTA's share of the entries: the rest of the tree over the CTAs; the sum goes to every CTA.  Four
        // threads per four entries: thread u adds up C / 4 neighbouring CTAs, then the four sums meet
        const uint32_t p0 = static_cast<uint32_t>(__cvta_generic_to_shared(part));
        const uint32_t g0 = static_cast<uint32_t>(__cvta_generic_to_shared(G));
        const int share = R * R / 4 / C;             // (C <= 16 divides R R / 4)
        const int run = max(1, C / 4);               // 1, 2 or 4
        for (int e = tid; e < share * 4; e += QS_THREADS) {
            const int q = crank * share + e / 4, u = e % 4;
            float4 s[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                s[c] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (c < run && u * run + c < C) s[c] = qs_ld_remote4(map_to_rank(p0, u * run + c) + q * 16);
            }
            float4 t;
            t.x = (s[0].x + s[1].x) + (s[2].x + s[3].x); t.y = (s[0].y + s[1].y) + (s[2].y + s[3].y);
            t.z = (s[0].z + s[1].z) + (s[2].z + s[3].z); t.w = (s[0].w + s[1].w) + (s[2].w + s[3].w);
            const unsigned mask = 0xfu << (lane & 28);
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                t.x += __shfl_xor_sync(mask, t.x, o); t.y += __shfl_xor_sync(mask, t.y, o);
                t.z += __shfl_xor_sync(mask, t.z, o); t.w += __shfl_xor_sync(mask, t.w, o);
            }
            for (int c = u; c < C; c += 4) qs_st_remote4(map_to_rank(g0, c) + q * 16, t);
        }
        cluster_sync_all();
    };
    // rows <- rows * G, G holding L^{-T} (row k, column j)
    auto apply = [&]() {
        if constexpr (R == 64) {
            // L^{-T} is upper triangular: column c needs the first c + 1 entries of a row only.  Warp w takes the
            // columns 4 w .. and 60 - 4 w .. (17 depth steps of four together, for every warp; w of each eight), a lane two rows.
            const int ca = 4 * (warp % 8), cb = 60 - ca;
            constexpr int NR = 4 * 256 / QS_THREADS;            // rows of a lane
            for (int i0 = 32 * NR * (warp / 8); i0 - 32 * NR * (warp / 8) < nrows; i0 += 128) {
                float xa[NR][4] = {}, xb[NR][4] = {};
                const float* yr = Y + (i0 + lane) * LD;
                auto step = [&](float (&acc)[NR][4], int k0, int col) {
                    float4 x[NR];
#pragma unroll
                    for (int e = 0; e < NR; ++e)
                        x[e] = i0 + lane + 32 * e < nrows ? *reinterpret_cast<const float4*>(yr + 32 * e * LD + k0) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const float4 b = *reinterpret_cast<const float4*>(G + (k0 + kk) * R + col);
#pragma unroll
                        for (int e = 0; e < NR; ++e) {
                            const float xv = kk == 0 ? x[e].x : (kk == 1 ? x[e].y : (kk == 2 ? x[e].z : x[e].w));
                            acc[e][0] = fmaf(xv, b.x, acc[e][0]); acc[e][1] = fmaf(xv, b.y, acc[e][1]);
                            acc[e][2] = fmaf(xv, b.z, acc[e][2]); acc[e][3] = fmaf(xv, b.w, acc[e][3]);
                        }
                    }
                };
#pragma unroll 2
                for (int k0 = 0; k0 <= ca; k0 += 4) step(xa, k0, ca);
#pragma unroll 2
                for (int k0 = 0; k0 <= cb; k0 += 4) step(xb, k0, cb);
                __syncthreads();
#pragma unroll
                for (int e = 0; e < NR; ++e)
                    if (i0 + lane + 32 * e < nrows) {
                        float* o = Y + (i0 + lane + 32 * e) * LD;
                        *reinterpret_cast<float4*>(o + ca) = make_float4(xa[e][0], xa[e][1], xa[e][2], xa[e][3]);
                        *reinterpret_cast<float4*>(o + cb) = make_float4(xb[e][0], xb[e][1], xb[e][2], xb[e][3]);
                    }
            }
            __syncthreads();
            return;
        }
        const int tx = tid % TX, ty = tid / TX;
        for (int i0 = 0; i0 < nrows; i0 += RT) {
            float acc[4][4] = {};
            const float* yr = Y + (i0 + ty * 4) * LD;
            const bool in = i0 + ty * 4 < nrows;         // rows come in fours: a part has a multiple of 32
            if (in) {
#pragma unroll 2
                for (int k0 = 0; k0 < R; k0 += 4) {
                    float4 x[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) x[e] = *reinterpret_cast<const float4*>(yr + e * LD + k0);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const float4 b = *reinterpret_cast<const float4*>(G + (k0 + kk) * R + tx * 4);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float xv = kk == 0 ? x[e].x : (kk == 1 ? x[e].y : (kk == 2 ? x[e].z : x[e].w));
                            acc[e][0] = fmaf(xv, b.x, acc[e][0]); acc[e][1] = fmaf(xv, b.y, acc[e][1]);
                            acc[e][2] = fmaf(xv, b.z, acc[e][2]); acc[e][3] = fmaf(xv, b.w, acc[e][3]);
                        }
                    }
                }
            }
            __syncthreads();
            if (in) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (i0 + ty * 4 + e < nrows)
                        *reinterpret_cast<float4*>(Y + (i0 + ty * 4 + e) * LD + tx * 4) =
                            make_float4(acc[e][0], acc[e][1], acc[e][2], acc[e][3]);
            }
        }
        __syncthreads();
    };
    // image rows of this CTA from Y (times scale); the last CTA also writes the padding rows as zeros
    auto write_image = [&](const ImgRef& im, int planes, float scale) {
        unsigned char* scr = reinterpret_cast<unsigned char*>(w.scratch);
        const int end = crank == C - 1 ? im.rows_pad : min(im.rows_pad, row0 + rows_per_cta);
        const int total = (end - row0) * 8;              // eight 16-byte chunks per row of the one panel
        for (int q = tid; q < total; q += QS_THREADS) {
            const int i = q / 8, c = q % 8;
            float v[8] = {};
            if (i < nrows && c * 8 < R) {
                const float4 x = *reinterpret_cast<const float4*>(Y + i * LD + c * 8);
                const float4 y = *reinterpret_cast<const float4*>(Y + i * LD + c * 8 + 4);
                v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
            }
            const int row = row0 + i, o = img_chunk_offset(row & 7, c);
            if (planes & 3) {
                uint4 t0, t1;
                split8(v, t0, t1);
                *reinterpret_cast<uint4*>(scr + img_row_offset(im, 0, 0, row) + o) = t0;
                *reinterpret_cast<uint4*>(scr + img_row_offset(im, 1, 0, row) + o) = t1;
            }
            if (planes & 4) *reinterpret_cast<uint4*>(scr + img_row_offset(im, 2, 0, row) + o) = half8(v, scale);
        }
    };

    // (one place for the Gram product: its code is fetched as it is run, and again from the cache)
    bool third = false;
    float trace = 0.f;
    for (int pass = 1; pass <= 3; ++pass) {
        gram();
        if (pass == 1) {
            // R's images for the fused pass (the fp16 plane scaled by the power of two that brings the largest
            // column norm to about 2^10)
            if (a.r_planes) {
                float scale = 1.f;
                if (a.r_planes & 4) {
                    float mx = 0.f;
                    for (int j = 0; j < r; ++j) mx = fmaxf(mx, G[j * R + j]);
                    int e = 0;
                    const float nrm = sqrtf(mx);
                    if (nrm > 0.f && nrm <= 3.0e38f) frexpf(nrm, &e);      // nrm = f * 2^e, 0.5 <= f < 1
                    scale = ldexpf(1.f, 10 - e);
                    if (crank == 0 && tid == 0) *reinterpret_cast<float*>(w.scratch + a.rscale_off) = ldexpf(1.f, e - 10);
                }
                write_image(a.r_img, a.r_planes, scale);
                __syncthreads();
            }
            if (a.colnorm) {
                float inv = 0.f;
                if (tid < r) {
                    const float nrm = sqrtf(G[tid * R + tid]);
                    if (!(nrm > 0.f) && crank == 0) atomicOr(w.status, ST_ZEROCOL);
                    inv = nrm > 0.f ? 1.f / nrm : 0.f;
                }
                __syncthreads();
                if (tid < R) G[tid] = inv;
                __syncthreads();
                for (int q = tid; q < nrows * R; q += QS_THREADS) Y[q / R * LD + q % R] *= G[q % R];
                __syncthreads();
                break;
            }
            for (int j = 0; j < r; ++j) trace += G[j * R + j];
            if (!(fabsf(trace) <= 3.0e38f)) {   // Inf or NaN
                if (tid == 0 && crank == 0) atomicOr(w.status, ST_NONFINITE);
                return;
            }
        }
        bool series = false;
        if (pass > 1) {
            // |G - I|_2 <= largest absolute row sum (see factor_tc.cuh: first-order inverse, third pass)
            constexpr int HS = QS_THREADS / R < R ? QS_THREADS / R : R;      // threads per row
            {
                const int i = tid % R, h = tid / R;
                float s = 0.f;
#pragma unroll
                for (int jj = 0; jj < R / HS; ++jj) {
                    const int j = min(h, HS - 1) * (R / HS) + jj;
                    s += j < r && i < r ? fabsf(G[j * R + i] - (i == j ? 1.f : 0.f)) : 0.f;
                }
                if (h < HS) part[tid] = s;
            }
            __syncthreads();
            if (warp == 0) {
                float mx = 0.f;
                for (int i = lane; i < R; i += 32) {
                    float s = 0.f;
#pragma unroll
                    for (int h = 0; h < HS; ++h) s += part[h * R + i];
                    mx = fmaxf(mx, s <= 3.0e38f ? s : 3.3e38f);
                }
                for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                if (lane == 0) s_bound = mx;
            }
            __syncthreads();
            if (pass == 2 && !(s_bound <= CT_THIRD_PASS_LIMIT)) third = true;
            series = s_bound <= a.series_limit;
            __syncthreads();
        }
        if (series) {
            for (int q = tid; q < R * R; q += QS_THREADS) {
                const int k = q / R, j = q % R;
                const float v = G[q];
                G[q] = k < j ? -v : (k == j ? 0.5f * (3.f - v) : 0.f);
            }
        } else {
            const bool tiny = pass == 1 && trace < CT_TINY_TRACE;          // see ct_rsqrt
            auto scale_block = [&](float f) {
                for (int q = tid; q < R * R; q += QS_THREADS) sD[q / R * CT_LDD + q % R] *= f;
                __syncthreads();
            };
            bool ok = false;
            for (int attempt = 0; attempt < (pass == 1 ? 2 : 1) && !ok; ++attempt) {
                const float shift = attempt ? a.shift_rel * trace : 0.f;
                const float pad = G[0] + shift;      // diagonal of the padding: the first pivot (see factor_tc.cuh)
                constexpr int DN = R <= 32 ? 32 : 64;
                for (int q = tid; q < DN * DN; q += QS_THREADS) {
                    const int i = q / DN, j = q % DN;
                    float v = i == j ? pad : 0.f;
                    if (i < r && j < r) v = G[i * R + j] + (i == j ? shift : 0.f);
                    sD[i * CT_LDD + j] = v;
                }
                __syncthreads();
                if (tiny) scale_block(CT_TINY_UP);
                if (warp < CT_DIAG_WARPS) {
                    const float2 mm = ct_diag_block(0, CT_DG_BLK, r, 1.f, warp, lane, nullptr, 0, nullptr);
                    if (tid == 0) { s_min = mm.y <= 3.0e38f ? mm.x : -1.f; s_max = mm.y; }
                }
                __syncthreads();
                const float mn = s_min, mx = s_max;
                const bool fail = !(mn > 0.f);
                const bool ill = pass == 1 && sqrtf(mx) > a.cond_limit * sqrtf(mn);
                if (!fail && !(ill && attempt == 0)) ok = true;
                else if (attempt == 0 && pass == 1) third = true;
                __syncthreads();
            }
            if (!ok) {
                if (tid == 0 && crank == 0) atomicOr(w.status, ST_RANKDEF | (third ? shift_bit : 0));
                return;
            }
            if (tiny) scale_block(CT_TINY_UP_ROOT);
            for (int q = tid; q < R * R; q += QS_THREADS) {
                const int k = q / R, j = q % R;
                G[q] = (k <= j && j < r) ? sD[k * CT_LDD + j] : 0.f;
            }
        }
        __syncthreads();
        apply();
        if (pass == 2 && !third) break;
    }
    if (third && tid == 0 && crank == 0) atomicOr(w.status, shift_bit);

    // ---- the factor and its image ----
    {
        float* D = pick(w, a.dst) + (int64_t)row0 * r;
        if (r % 4)
            for (int q = tid; q < nrows * r; q += QS_THREADS) D[q] = Y[q / r * LD + q % r];
        else
            for (int q = tid; q < nrows * r4; q += QS_THREADS) {
                const int i = q / r4, c = q % r4;
                *reinterpret_cast<float4*>(D + i * r + c * 4) = *reinterpret_cast<const float4*>(Y + i * LD + c * 4);
            }
    }
    if (a.img_planes) write_image(a.img, a.img_planes, 1.f);
}

}  // namespace od
