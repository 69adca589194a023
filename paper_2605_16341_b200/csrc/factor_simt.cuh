// r x r factor kernel of the SIMT engine: Cholesky factor of the Gram matrix and its explicit inverse in
// fp32, one CTA per matrix.
//
// The same loop as the tensor engine's kernel (factor_tc.cuh: [Gram; I] as one left-looking
// factorisation over 64-wide block columns, diagonal blocks by four warps), with fp32 tile products.
// `work` holds L below its diagonal tiles, L^{-T} above them and, in each of them, X_k = L(k,k)^{-1} on
// and below the diagonal and its transpose above: row i of L^{-T} is row i of `work` from column i on.  At
// the end the upper part is transposed into the lower one and cleared.
//
// What bounds it: one diagonal block (about 6 us) per 64 columns and, from r = 256 up, the fp32
// products of a single CTA.  Measured, one factorisation (before: 32-wide blocks, right-looking, pairwise
// inversion): r = 40 87 -> 26 us.
#pragma once
#include "factor_tc.cuh"
#include "simt_kernels.cuh"

namespace od {

constexpr int FS_THREADS = 256;
constexpr int FS_OFF_X = 4 * SIMT_KC * SIMT_LD * 4;      // X_k transposed, after the two operand stages
constexpr int FS_OFF_D = FS_OFF_X + CT_NB * SIMT_LD * 4;     // the diagonal block's area
constexpr int FS_SMEM_BYTES = FS_OFF_D + CT_DG_BYTES;

template <class BATCH>
__global__ void __launch_bounds__(FS_THREADS, 2)
factor_simt_kernel(const __grid_constant__ BATCH batch, CholArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    SimtStage* As = reinterpret_cast<SimtStage*>(smem);
    SimtStage* Bs = As + 2;
    float* Xs = reinterpret_cast<float*>(smem + FS_OFF_X);
    float* sD = reinterpret_cast<float*>(smem + FS_OFF_D);
    __shared__ float red[FS_THREADS / 32];
    __shared__ float s_up[2];                 // scales of a tiny matrix (see ct_rsqrt)
    __shared__ float s_min, s_max;            // smallest and largest pivot

    const MatWork& w = batch.w[blockIdx.x];
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const int tx = tid % 16, ty = tid / 16;
    const int r = a.r, nb = (r + CT_NB - 1) / CT_NB;
    const int shift_bit = a.which ? ST_SHIFT_R : ST_SHIFT_L;
    grid_dependency();
    const int st0 = *w.status;
    if (st0 & ST_FAILED) return;
    if (a.pass == 3 && !(st0 & shift_bit)) return;
    __syncthreads();            // the status word may change below
    const float* __restrict__ A = pick(w, a.gram);     // Gram matrix: never written here
    float* W = pick(w, a.work);

    // trace and finiteness of the Gram diagonal
    float trace = 0.f;
    for (int i = tid; i < r; i += FS_THREADS) trace += A[(int64_t)i * r + i];
    for (int o = 16; o; o >>= 1) trace += __shfl_xor_sync(0xffffffffu, trace, o);
    if (lane == 0) red[warp] = trace;
    __syncthreads();
    trace = 0.f;
    for (int i = 0; i < FS_THREADS / 32; ++i) trace += red[i];
    if (!(fabsf(trace) <= 3.0e38f)) {   // Inf or NaN
        if (tid == 0) atomicOr(w.status, ST_NONFINITE);
        return;
    }

    // acc(i, j) = sum_{c in [c0, c1)} W[ri + i][c] W[rj + j][c]; upper: row ri + i counts from column ri + i on
    // only (a row of L^{-T})
    auto row_products = [&](float (&acc)[4][4], int ri, int rj, int c0, int c1, bool upper) {
        float va[8], vb[8];
        auto load = [&](int k0) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                int ii, kk;
                simt_pos(true, e, ii, kk);
                const int c = k0 + kk;
                va[e] = (ri + ii < r && c < c1 && (!upper || c >= ri + ii)) ? W[(int64_t)(ri + ii) * r + c] : 0.f;
                vb[e] = (rj + ii < r && c < c1) ? W[(int64_t)(rj + ii) * r + c] : 0.f;
            }
        };
        if (c0 < c1) load(c0);
        int s = 0;
        for (int k0 = c0; k0 < c1; k0 += SIMT_KC) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                int ii, kk;
                simt_pos(true, e, ii, kk);
                As[s][kk][ii] = va[e];
                Bs[s][kk][ii] = vb[e];
            }
            __syncthreads();
            if (k0 + SIMT_KC < c1) load(k0 + SIMT_KC);
            simt_fma(acc, As[s], Bs[s], ty, tx);
            s ^= 1;
        }
        __syncthreads();
    };

    if (tid == 0) { s_up[0] = trace < CT_TINY_TRACE ? CT_TINY_UP : 1.f; s_up[1] = trace < CT_TINY_TRACE ? CT_TINY_UP_ROOT : 1.f; }

    bool ok = false;
    const int max_attempts = (a.pass == 1) ? 2 : 1;
    for (int attempt = 0; attempt < max_attempts && !ok; ++attempt) {
        const float shift = attempt ? a.shift_rel * trace : 0.f;
        const float pad = A[0] + shift;         // diagonal of the padding: the first pivot (see factor_tc.cuh)
        if (tid == 0) { s_min = 3.0e38f; s_max = 0.f; }
        for (int k = 0; k < nb; ++k) {
            const int k0 = k * CT_NB, nbk = min(CT_NB, r - k0);
            // diagonal block
            {
                float acc[4][4] = {};
                row_products(acc, k0, k0, 0, k0, false);
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int f = 0; f < 4; ++f) {
                        const int i = ty * 4 + e, j = tx * 4 + f;
                        float v = i == j ? pad : 0.f;
                        if (i < nbk && j < nbk) v = A[(int64_t)(k0 + max(i, j)) * r + k0 + min(i, j)] + (i == j ? shift : 0.f) - acc[e][f];
                        sD[i * CT_LDD + j] = v * s_up[0];
                    }
            }
            __syncthreads();
            if (warp < CT_DIAG_WARPS) {
                const float2 mm = ct_diag_block(FS_OFF_D, FS_OFF_D + CT_DG_BLK, nbk, 1.f, warp, lane, nullptr, 0, nullptr);
                if (tid == 0) { s_min = mm.y <= 3.0e38f ? fminf(s_min, mm.x) : -1.f; s_max = fmaxf(s_max, mm.y); }
            }
            __syncthreads();
            for (int q = tid; q < CT_NB * CT_NB; q += FS_THREADS) {
                const int i = q / CT_NB, j = q % CT_NB;
                const float v = sD[min(i, j) * CT_LDD + max(i, j)] * s_up[1];
                if (i < nbk && j < nbk) W[(int64_t)(k0 + i) * r + k0 + j] = v;
                Xs[i * SIMT_LD + j] = (i <= j && j < nbk) ? v : 0.f;         // X_k(j, i)
            }
            // the other tiles of the block column
            for (int t = 0; t < nb; ++t) {
                if (t == k) continue;
                const int i0 = t * CT_NB;
                float acc[4][4] = {};
                row_products(acc, i0, k0, t < k ? i0 : 0, k0, t < k);
                float* S = &As[0][0][0];                 // S transposed, 64 deep
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    const int j = k0 + tx * 4 + f;
                    float v[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int i = i0 + ty * 4 + e;
                        v[e] = ((t > k && i < r && j < r) ? A[(int64_t)i * r + j] : 0.f) - acc[e][f];
                    }
                    *reinterpret_cast<float4*>(S + (tx * 4 + f) * SIMT_LD + ty * 4) = make_float4(v[0], v[1], v[2], v[3]);
                }
                __syncthreads();
                float o[4][4] = {};
                simt_fma(o, As[0], reinterpret_cast<const SimtStage*>(Xs)[0], ty, tx);
                simt_fma(o, As[1], reinterpret_cast<const SimtStage*>(Xs)[1], ty, tx);
                __syncthreads();
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int f = 0; f < 4; ++f) {
                        const int i = i0 + ty * 4 + e, j = k0 + tx * 4 + f;
                        if (i < r && j < r) W[(int64_t)i * r + j] = o[e][f];
                    }
            }
            __syncthreads();
        }
        const float mn = s_min, mx = s_max;
        const bool fail = !(mn > 0.f);
        const bool ill = (a.pass == 1) && (sqrtf(mx) > a.cond_limit * sqrtf(mn));
        if (!fail && !(ill && attempt == 0)) {
            ok = true;
        } else if (attempt == 0 && a.pass == 1) {
            if (tid == 0) atomicOr(w.status, shift_bit);
        }
        __syncthreads();
    }
    if (!ok) {
        if (tid == 0) atomicOr(w.status, ST_RANKDEF);
        return;
    }

    // upper part (L^{-T}) -> lower part, upper part <- 0
    float* buf = reinterpret_cast<float*>(smem);         // 64 x 65
    for (int tb = 0; tb < nb; ++tb)
        for (int ta = 0; ta <= tb; ++ta) {
            for (int q = tid; q < CT_NB * CT_NB; q += FS_THREADS) {
                const int i = ta * CT_NB + q / CT_NB, j = tb * CT_NB + q % CT_NB;
                if (i < r && j < r && i <= j) {
                    buf[(q / CT_NB) * 65 + q % CT_NB] = W[(int64_t)i * r + j];
                    if (i < j) W[(int64_t)i * r + j] = 0.f;
                }
            }
            __syncthreads();
            for (int q = tid; q < CT_NB * CT_NB; q += FS_THREADS) {
                const int i = tb * CT_NB + q / CT_NB, j = ta * CT_NB + q % CT_NB;
                if (i < r && j <= i) W[(int64_t)i * r + j] = buf[(q % CT_NB) * 65 + q / CT_NB];
            }
            __syncthreads();
        }
}

}  // namespace od
