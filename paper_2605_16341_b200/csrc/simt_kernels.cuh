// Plain fp32 FMA kernels: the SIMT engine's matrix products (any shape, any r >= 1).
// Used for tiny matrices, sizes that fit no tile, and as an on-device cross-check of the tensor-core
// engine.
//
// What bounds them: latency.  The results are a few 64 x 64 tiles (one for the Gram matrix at
// r <= 64), each a sum over a thousand rows or columns.  The depth is therefore cut into up to eight
// chunks that the CTAs of a cluster take side by side; the partial tiles are added in chunk order
// through distributed shared memory, so no extra launch and no workspace.  Loads run along the contiguous
// direction, one 32-deep step ahead of the products.  Measured on one 1023 x 777 fp32 matrix, r = 40 (one
// CTA per tile, 16-deep steps, no loads ahead -> now): Gram product 149 -> 19 us, Y = B Q_prev 187 ->
// 31, R = B^T P 217 -> 31, the two products of the update 19.5 + 19.0 -> 21.5 in one kernel.
#pragma once
#include "common.cuh"
#include "launch.cuh"

namespace od {

// ---- operand readers: values of the logical operand at (row i, depth k) ----------------------
// fetch() sends eight loads out and waits for none; value() is what comes of them.  (With the sum of M and G formed element
// by element as they were read, a 32-deep step of B Q_prev took 9500 cycles, one load after the other.)
struct RdPlain {            // fp32 matrix with arbitrary strides: elem(i,k) = p[i*rs + k*cs]
    Sel sel; int64_t rs, cs;
    struct Raw { float v[8]; };
    __device__ __forceinline__ bool depth_contiguous() const { return cs == 1; }
    __device__ __forceinline__ void fetch(const MatWork& w, const int64_t (&i)[8], const int64_t (&k)[8], const bool (&in)[8], Raw& r) const {
        const float* p = pick(w, sel);
#pragma unroll
        for (int e = 0; e < 8; ++e) r.v[e] = in[e] ? p[i[e] * rs + k[e] * cs] : 0.f;
    }
    __device__ __forceinline__ float value(const Raw& r, int e) const { return r.v[e]; }
};
struct RdBuffer {           // B = M + G formed on the fly (Alg. 1, buffer step); trans: elem(i,k)=B[k][i]
    int64_t ld; int32_t g_bf16; int32_t trans;
    struct Raw { float m[8]; uint32_t g[8]; };
    __device__ __forceinline__ bool depth_contiguous() const { return !trans; }
    __device__ __forceinline__ void fetch(const MatWork& w, const int64_t (&i)[8], const int64_t (&k)[8], const bool (&in)[8], Raw& r) const {
        int64_t idx[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            idx[e] = trans ? k[e] * ld + i[e] : i[e] * ld + k[e];
            r.m[e] = in[e] ? w.M[idx[e]] : 0.f;
        }
        if (g_bf16) {
#pragma unroll
            for (int e = 0; e < 8; ++e) r.g[e] = in[e] ? (uint32_t)reinterpret_cast<const uint16_t*>(w.G)[idx[e]] << 16 : 0u;
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) r.g[e] = in[e] ? reinterpret_cast<const uint32_t*>(w.G)[idx[e]] : 0u;
        }
    }
    __device__ __forceinline__ float value(const Raw& r, int e) const { return r.m[e] + __uint_as_float(r.g[e]); }
};

struct SimtOut {            // C[i*ld + j] = acc ; destination may depend on the shift flag
    Sel dst, dst_if_shifted; int32_t shift_bit; int32_t skip_if_failed; int64_t ld;
    int32_t only_if_shifted;
    int32_t lower_only;     // symmetric result: tiles above the diagonal are not computed
    __device__ __forceinline__ bool active(int st) const {
        if (skip_if_failed && (st & ST_FAILED)) return false;
        if (only_if_shifted && !(st & shift_bit)) return false;
        return true;
    }
};

constexpr int SIMT_KC = 32;         // depth of one staged step
constexpr int SIMT_LD = 68;         // staged rows: 64 + 4 floats (16-byte aligned, few bank conflicts)
constexpr int SIMT_MAX_PARTS = 8;
using SimtStage = float[SIMT_KC][SIMT_LD];

// Number of depth chunks (CTAs of a cluster) of a product: at least 64 deep each.  A function of the
// depth only, so that a matrix gets the same bits alone and in any group.
inline int simt_parts(int64_t depth) {
    int parts = 1;
    while (parts < SIMT_MAX_PARTS && depth >= 128 * parts) parts *= 2;
    return parts;
}

// This thread's eight elements of a 64 x SIMT_KC operand step: element e at (row, depth) below.
__device__ __forceinline__ void simt_pos(bool depth_fast, int e, int& ii, int& kk) {
    const int idx = threadIdx.x + 256 * e;
    if (depth_fast) { kk = idx % SIMT_KC; ii = idx / SIMT_KC; }
    else { ii = idx % 64; kk = idx / 64; }
}
template <class RD>
__device__ __forceinline__ void simt_load(const RD& rd, const MatWork& w, int64_t i0, int64_t k0, int64_t rows, int64_t kend,
                                          typename RD::Raw& raw) {
    const bool fast = rd.depth_contiguous();
    int64_t i[8], k[8];
    bool in[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        int ii, kk;
        simt_pos(fast, e, ii, kk);
        i[e] = i0 + ii; k[e] = k0 + kk;
        in[e] = i[e] < rows && k[e] < kend;
    }
    rd.fetch(w, i, k, in, raw);
}
template <class RD>
__device__ __forceinline__ void simt_store(const RD& rd, SimtStage& s, const typename RD::Raw& raw) {
    const bool fast = rd.depth_contiguous();
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        int ii, kk;
        simt_pos(fast, e, ii, kk);
        s[kk][ii] = rd.value(raw, e);
    }
}
__device__ __forceinline__ void simt_fma(float (&acc)[4][4], const SimtStage& a, const SimtStage& b, int ty, int tx) {
#pragma unroll 8
    for (int kk = 0; kk < SIMT_KC; ++kk) {
        const float4 x = *reinterpret_cast<const float4*>(&a[kk][ty * 4]);
        const float4 y = *reinterpret_cast<const float4*>(&b[kk][tx * 4]);
        const float xa[4] = {x.x, x.y, x.z, x.w}, yb[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int f = 0; f < 4; ++f) acc[e][f] = fmaf(xa[e], yb[f], acc[e][f]);
    }
}

// C(i,j) = sum_k A(i,k) * Bm(j,k): both operands are read as (row, depth).
// 64 x 64 tile per cluster of `parts` CTAs (chunk `rank` of the depth each), 256 threads, 4 x 4
// results per thread.
template <class BATCH, class RA, class RB>
__global__ void __launch_bounds__(256)
simt_gemm_kernel(const __grid_constant__ BATCH batch, int64_t Md, int64_t Nd, int64_t Kd, int parts, RA ra, RB rb, SimtOut out) {
    grid_dependency();
    const MatWork& w = batch.w[blockIdx.z];
    const int st = *w.status;
    if (!out.active(st)) return;
    __shared__ SimtStage As[2], Bs[2];
    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const int rank = (int)(blockIdx.x % (unsigned)parts);
    const int64_t i0 = (int64_t)blockIdx.y * 64, j0 = (int64_t)(blockIdx.x / (unsigned)parts) * 64;
    if (out.lower_only && j0 > i0) return;
    const int64_t per = (Kd + (int64_t)parts * SIMT_KC - 1) / ((int64_t)parts * SIMT_KC) * SIMT_KC;
    const int64_t kbeg = rank * per, kend = min(Kd, kbeg + per);
    float acc[4][4] = {};
    typename RA::Raw va;
    typename RB::Raw vb;
    if (kbeg < kend) {
        simt_load(ra, w, i0, kbeg, Md, kend, va);
        simt_load(rb, w, j0, kbeg, Nd, kend, vb);
    }
    int s = 0;
    for (int64_t k0 = kbeg; k0 < kend; k0 += SIMT_KC) {
        simt_store(ra, As[s], va);
        simt_store(rb, Bs[s], vb);
        __syncthreads();
        if (k0 + SIMT_KC < kend) {
            simt_load(ra, w, i0, k0 + SIMT_KC, Md, kend, va);
            simt_load(rb, w, j0, k0 + SIMT_KC, Nd, kend, vb);
        }
        simt_fma(acc, As[s], Bs[s], ty, tx);
        s ^= 1;
    }
    float* C = pick(w, (out.shift_bit && (st & out.shift_bit)) ? out.dst_if_shifted : out.dst);
    if (parts == 1) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                const int64_t gi = i0 + ty * 4 + e, gj = j0 + tx * 4 + f;
                if (gi < Md && gj < Nd) C[gi * out.ld + gj] = acc[e][f];
            }
        return;
    }
    // partial tiles meet in shared memory; CTA `rank` adds its share of the tile, in chunk order
    __syncthreads();
    float* tile = &As[0][0][0];
#pragma unroll
    for (int e = 0; e < 4; ++e)
        *reinterpret_cast<float4*>(tile + (ty * 4 + e) * 64 + tx * 4) = make_float4(acc[e][0], acc[e][1], acc[e][2], acc[e][3]);
    cluster_sync_all();
    const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(tile));
    const int share = 4096 / parts;
    for (int q = rank * share + tid; q < (rank + 1) * share; q += 256) {
        float v[SIMT_MAX_PARTS];
#pragma unroll
        for (int p = 0; p < SIMT_MAX_PARTS; ++p) {
            v[p] = 0.f;
            if (p < parts)
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v[p]) : "r"(map_to_rank(local + q * 4, p)) : "memory");
        }
        float sum = v[0];
#pragma unroll
        for (int p = 1; p < SIMT_MAX_PARTS; ++p) sum += v[p];
        const int64_t gi = i0 + q / 64, gj = j0 + q % 64;
        if (gi < Md && gj < Nd) C[gi * out.ld + gj] = sum;
    }
    cluster_sync_all();         // nobody leaves while its tile may still be read
}

// M <- a (M + G) - b P R^T,  X <- c X - d P Q^T  (Alg. 1, update and error-feedback steps): both products
// in one pass, P read once.  64 x 64 tile per CTA.
template <class BATCH>
__global__ void __launch_bounds__(256)
simt_update_kernel(const __grid_constant__ BATCH batch, int64_t m, int64_t n, int r, float a, float b, float c, float d,
                   int g_bf16, int x_bf16) {
    grid_dependency();
    const MatWork& w = batch.w[blockIdx.z];
    if (*w.status & ST_FAILED) return;
    // the operand steps, then the two products by rows (65 floats apart: both ways without bank conflicts)
    __shared__ __align__(16) float buf[2 * 64 * 65];
    static_assert(3 * SIMT_KC * SIMT_LD <= 2 * 64 * 65, "three operand steps fit");
    SimtStage* st = reinterpret_cast<SimtStage*>(buf);
    SimtStage &Ps = st[0], &Rs = st[1], &Qs = st[2];
    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const int64_t i0 = (int64_t)blockIdx.y * 64, j0 = (int64_t)blockIdx.x * 64;
    const RdPlain rp{Sel{W_P, 0, 0}, r, 1}, rr{Sel{W_R, 0, 0}, r, 1}, rq{Sel{W_Q, 0, 0}, r, 1};
    float accm[4][4] = {}, accx[4][4] = {};
    RdPlain::Raw vp, vr, vq;
    simt_load(rp, w, i0, 0, m, r, vp);
    simt_load(rr, w, j0, 0, n, r, vr);
    simt_load(rq, w, j0, 0, n, r, vq);
    for (int64_t k0 = 0; k0 < r; k0 += SIMT_KC) {
        simt_store(rp, Ps, vp);
        simt_store(rr, Rs, vr);
        simt_store(rq, Qs, vq);
        __syncthreads();
        if (k0 + SIMT_KC < r) {
            simt_load(rp, w, i0, k0 + SIMT_KC, m, r, vp);
            simt_load(rr, w, j0, k0 + SIMT_KC, n, r, vr);
            simt_load(rq, w, j0, k0 + SIMT_KC, n, r, vq);
        }
        simt_fma(accm, Ps, Rs, ty, tx);
        simt_fma(accx, Ps, Qs, ty, tx);
        __syncthreads();
    }
    float *dm = buf, *dx = buf + 64 * 65;
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            dm[(ty * 4 + e) * 65 + tx * 4 + f] = accm[e][f];
            dx[(ty * 4 + e) * 65 + tx * 4 + f] = accx[e][f];
        }
    __syncthreads();
    // rows of the tile, lanes along them; eight elements of M, G and X under way (read where they were wanted, one after the
    // other, this took most of 20 us for 1023 x 777)
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        float mv[8];
        uint32_t gv[8], xv[8];
        int64_t idx[8];
        bool in[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int64_t gi = i0 + h * 32 + e * 4 + tid / 64, gj = j0 + tid % 64;
            in[e] = gi < m && gj < n;
            idx[e] = gi * n + gj;
            mv[e] = in[e] ? w.M[idx[e]] : 0.f;
        }
        auto raw = [&](const void* p, int bf16, uint32_t (&v)[8]) {
            if (bf16) {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = in[e] ? (uint32_t)reinterpret_cast<const uint16_t*>(p)[idx[e]] << 16 : 0u;
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = in[e] ? reinterpret_cast<const uint32_t*>(p)[idx[e]] : 0u;
            }
        };
        raw(w.G, g_bf16, gv);
        raw(w.X, x_bf16, xv);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int q = (h * 32 + e * 4 + tid / 64) * 65 + tid % 64;
            if (!in[e]) continue;
            w.M[idx[e]] = a * (mv[e] + __uint_as_float(gv[e])) - b * dm[q];
            const float x = c * __uint_as_float(xv[e]) - d * dx[q];
            if (x_bf16) reinterpret_cast<__nv_bfloat16*>(w.X)[idx[e]] = __float2bfloat16_rn(x);
            else reinterpret_cast<float*>(w.X)[idx[e]] = x;
        }
    }
}

}  // namespace od
