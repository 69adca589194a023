// Arguments of the r x r factor kernels; ColNorm; status initialisation.
#pragma once
#include "common.cuh"
#include "launch.cuh"

namespace od {

struct CholArgs {
    Sel gram;        // r x r Gram matrix (input, left intact)
    Sel work;        // SIMT engine: r x r, receives L^{-1} (lower triangular, strict upper part zero)
    int32_t r;
    int32_t which;   // 0: left QR (P), 1: right QR (Q)
    int32_t pass;    // 1, 2 or 3
    float shift_rel; // shift = shift_rel * trace(Gram) on the retry of pass 1
    float cond_limit;// take the shifted path when max diag(L) / min diag(L) exceeds this (pass 1)
    // Optional fp32 column sums of squares, colsq[p * r + i] for p < MatWork::aux0 partial rows: when
    // use_colsq is set they replace the Gram diagonal.  (The tensor core truncates when it adds
    // into its fp32 accumulator, which biases long sums of squares low; the off-diagonal sums have
    // no such bias.)
    Sel colsq;
    int32_t use_colsq;
    int32_t ahead;       // launches overlap: run the code of the diagonal blocks once while the kernel before is still at work
    // tensor engine: split image of L^{-T} (the result there, operand of the apply product; the image of L has the
    // same geometry and lies at MatWork::aux1), the Gram diagonal (fp32 [r]), the statistics of the
    // diagonal blocks, and later passes: L^{-1}(j, j) over the value that its two image terms hold (fp32 [r], then
    // one more float: not zero when these factors are to be used)
    ImgRef img;
    int64_t diag_off, stat_off, scale_off;
    int64_t cnorm_off;   // >= 0: also leave the Gram diagonal (squared column norms) there, fp32 [r]
};

// ---- ColNorm of the SIMT engine (Alg. 1, normalisation step, Dion branch): Q[:,j] = R[:,j] / ||R[:,j]||_2 ---
// One CTA per 32 columns: 32 x 32 threads, lanes along columns (coalesced rows).
template <class BATCH>
__global__ void __launch_bounds__(1024)
colnorm_kernel(const __grid_constant__ BATCH batch, int64_t n, int r) {
    grid_dependency();
    const MatWork& w = batch.w[blockIdx.z];
    if (*w.status & ST_FAILED) return;
    __shared__ float part[32][33];
    __shared__ float inv[32];
    const int lane = threadIdx.x % 32, ry = threadIdx.x / 32;
    const int j = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (j < r)
        for (int64_t i = ry; i < n; i += 32) { float v = w.R[i * r + j]; s = fmaf(v, v, s); }
    part[ry][lane] = s;
    __syncthreads();
    if (ry == 0) {
        float t = 0.f;
        for (int k = 0; k < 32; ++k) t += part[k][lane];
        float nrm = sqrtf(t);
        if (j < r && !(nrm > 0.f)) atomicOr(w.status, ST_ZEROCOL);
        inv[lane] = (nrm > 0.f) ? 1.f / nrm : 0.f;
    }
    __syncthreads();
    if (j < r) {
        const float sc = inv[lane];
        for (int64_t i = ry; i < n; i += 32) w.Q[i * r + j] = w.R[i * r + j] * sc;
    }
}

// ---- squared column norms -----------------------------------------------------------------------
// dst[j * stride] <- sum over the blocks of the column sums of squares that a product kernel has left per 32 rows
// (colsq[block * r + j]).  stride 1: the squared column norms; r + 1: the diagonal of a Gram matrix (fp32 sums: the tensor
// core's truncating accumulation would bias it low), so that a sum of it over shards carries the exact diagonal along.
// One CTA per 64 columns: 16 interleaved sums per column, eight loads of each under way (latency is all there is: a serial
// loop took 11.5 us for 3584 rows at r = 512).
template <class BATCH>
__global__ void __launch_bounds__(256)
colsum_kernel(const __grid_constant__ BATCH batch, int64_t colsq_off, int blocks, int r, Sel dst, int64_t stride) {
    grid_dependency();
    const MatWork& w = batch.w[blockIdx.z];
    if (*w.status & ST_FAILED) return;
    __shared__ float part[16][64];
    const float* cs = reinterpret_cast<const float*>(w.scratch + colsq_off);
    const int g = threadIdx.x / 16, q4 = threadIdx.x % 16 * 4, col = blockIdx.x * 64 + q4;
    float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
    if (col < r)
#pragma unroll 1
        for (int kb = g; kb < blocks; kb += 128) {
            float4 v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                v[e] = kb + 16 * e < blocks ? *reinterpret_cast<const float4*>(cs + (int64_t)(kb + 16 * e) * r + col) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int e = 0; e < 8; ++e) { d.x += v[e].x; d.y += v[e].y; d.z += v[e].z; d.w += v[e].w; }
        }
    *reinterpret_cast<float4*>(&part[g][q4]) = d;
    __syncthreads();
    const int j = blockIdx.x * 64 + threadIdx.x;
    if (threadIdx.x < 64 && j < r) {
        float sum = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) sum += part[k][threadIdx.x];
        pick(w, dst)[j * stride] = sum;
    }
}

// ---- helpers of the column-sharded step ---------------------------------------------------------
// Column sums of squares of an fp32 matrix S (rows x r) per block of 32 rows, in the layout the
// product kernels write next to their results: out[blk * r + j], blk < 4 * ceil(rows / 128)
// (blocks beyond the matrix hold zeros).  One CTA per (32-row block, 256 columns).
__global__ void __launch_bounds__(256)
colsq_blocks_kernel(const __grid_constant__ SmallBatch batch, Sel src, int64_t rows, int r, int64_t colsq_off) {
    grid_dependency();
    const MatWork& w = batch.w[blockIdx.z];
    if (*w.status & ST_FAILED) return;
    const float* S = pick(w, src);
    float* out = reinterpret_cast<float*>(w.scratch + colsq_off);
    const int j = blockIdx.y * 256 + threadIdx.x;
    if (j >= r) return;
    const int64_t i0 = (int64_t)blockIdx.x * 32;
    float s = 0.f;
    for (int k = 0; k < 32; ++k)
        if (i0 + k < rows) { const float v = S[(i0 + k) * r + j]; s = fmaf(v, v, s); }
    out[(int64_t)blockIdx.x * r + j] = s;
}

template <class BATCH>
__global__ void init_status_kernel(const __grid_constant__ BATCH batch) {
    grid_dependency();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < batch.count) *batch.w[i].status = 0;
}

}  // namespace od
