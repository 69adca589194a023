// Tensor-core engine: tcgen05 (5th-generation tensor core) kernels with accumulators in tensor
// memory.  Every matrix product of the step is a sum of bf16 products with fp32 accumulation:
// an fp32 operand v is split as v = t0 + t1 with t0 = bf16(v), t1 = bf16(v - t0), and "3 passes"
// means t0*u0 + t0*u1 + t1*u0 (relative error about 2^-16), "1 pass" t0*u0.
//
// Operands.  Every small operand (Q, Y, P, R, L^{-1} and the QR intermediates) lives in global
// memory as a split image (common.cuh): ready-made swizzled shared-memory tiles that one tiled
// TMA load (cp.async.bulk.tensor over a 5-d tensor map: 64 elements, rows, panels, terms,
// matrices of the launch batch) drops into an operand ring, usable both K-major and MN-major,
// so no kernel ever transposes.  Images are written by the epilogue of the kernel
// that produces the matrix; only Q_prev (caller-owned fp32) is packed by a kernel of its own.
// The big operand B = M + G (Alg. 1, buffer step) is never stored: transform warps read M and G from
// HBM, add, split and write the A tile directly.
//
// One CTA per SM walks a tile list.  Two rings in shared memory: A tiles of 128 x 64 (both terms,
// 32 KB) and N-side pieces (a slice of the other operand, at most 48 KB), each with full/empty
// mbarriers; accumulators (up to 128 x 512 fp32) sit in tensor memory.
#pragma once
#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <cstdio>

#include "common.cuh"
#include "factor_tc.cuh"
#include "launch.cuh"
#include "qr_small.cuh"
#include "simt_kernels.cuh"

namespace od {
namespace tc {

constexpr int BM = 128;                      // tile rows (MMA M)
constexpr int BK = 64;                       // depth of one A tile: 64 bf16 = one 128-byte row
constexpr int A_TERM_BYTES = 128 * 128;      // one 128 x 64 bf16 tile
constexpr int A_RING_BYTES = 4 * A_TERM_BYTES;   // two slots of two terms, or four slots of one
constexpr int MAX_A_SLOTS = 4;
constexpr int MAX_N_SLOTS = 6;
constexpr int NUM_XF_WARPS = 16;             // transform warps of the kernels that form B = M + G
constexpr int STORE_STAGING_BYTES = 4096;    // epilogue staging of the products: one 32 x 32 fp32 block per warp
// ... of the fused pass: 32 x 32 slabs of M, G and X per warp (xg bit 0: G is bf16, bit 1: X is)
__host__ __device__ constexpr int slab_bytes(int xg) { return 4096 + ((xg & 1) ? 2048 : 4096) + ((xg & 2) ? 2048 : 4096); }
constexpr int SMEM_LIMIT = 227 * 1024;
constexpr long long WAIT_LIMIT_CYCLES = 4000000000LL;   // about two seconds

enum AMode : int { A_IMG_K = 0, A_IMG_MN = 1, A_BUF_ROW = 2, A_BUF_COL = 3 };
enum NMode : int { N_IMG_K = 0, N_IMG_MN = 1 };
enum EpiMode : int { EPI_STORE = 0, EPI_K5 = 1 };

__host__ __device__ constexpr bool a_is_buf(int amode) { return amode == A_BUF_ROW || amode == A_BUF_COL; }
// Eight epilogue warps (two per tensor-memory lane quarter, splitting the columns): the epilogue is most of a tile's time
// in the fused pass, and a third of it in launches of one tile of an image product (one 4096 x 4096 matrix at r = 256, four ->
// eight: step 406 -> 402 us; their staging is 32 KB, which leaves room for the third A slot).  Four in the products that
// form B, which have sixteen transform warps already.
__host__ __device__ constexpr int epi_warps(int amode, int epi) { return epi == EPI_K5 || !a_is_buf(amode) ? 8 : 4; }
__host__ __device__ constexpr int gemm_threads(int amode, int epi) {
    return 32 * (2 + epi_warps(amode, epi) + (a_is_buf(amode) ? NUM_XF_WARPS : 0));
}

// Where the result of an EPI_STORE product goes.
struct Dest {
    Sel f32;            // fp32 row-major copy (leading dimension OutSpec::ld) when has_f32
    ImgRef img;         // split image when img.off >= 0
    int32_t has_f32;
    int32_t colsq;      // also write per-(32-row block) column sums of squares (fp32)
};
struct OutSpec {
    Dest normal, shifted;      // `shifted` is used when the matrix's status has shift_bit set
    int32_t shift_bit;
    int32_t only_if_shifted;   // skip the matrix unless shift_bit is set
    int64_t ld;
};

struct GemmArgs {
    int32_t Mrows, Ncols, Kdim, BN;          // BN: nominal tile width (multiple of 16, <= 512)
    int32_t m_tiles, n_tiles, k_blocks, total_tiles;
    int32_t tri;                             // N-side is lower triangular (apply): skip depth beyond the tile
    int32_t lower_only;                      // symmetric result (Gram): skip tiles above the diagonal
    int32_t one_operand;                     // ... whose tiles on the diagonal have the same columns on either side
    int32_t passes, passes2;                 // 1 or 3; passes2: second product of the fused pass
    int32_t ks;                              // N_IMG_MN: depth of one N-side piece (16, 32 or 64)
    int32_t n_slots, n_piece_bytes;          // N ring
    int32_t n_split;                         // fused pass: the R piece and the Q piece of a depth block in slots of their own
    int32_t acc_bufs;                        // accumulator buffers in tensor memory (1 or 2)
    int32_t tmem_cols;                       // allocation (power of two >= 32)
    int32_t fp16;                            // single-pass fp16 products from plane 2 of the images
    int32_t a_slots, a_slot_bytes;           // A ring
    int32_t epi_bufs;                        // fused pass: 8 KB epilogue buffers per warp (1 or 2)
    int32_t pair;                            // launched as CTA pairs (clusters of two, M = 256 instructions)
    int32_t chunks, kb_per_chunk;            // depth chunks whose sums are added up in order, and their depth blocks
    int32_t acc_chunks;                      // chunks within one tile: accumulators side by side in tensor memory,
                                             // added up by the epilogue (products with B)
    int32_t ksplit, kb_per_tile;             // tiles of such chunks that a result tile is computed as, their depth
    int64_t split_stride;                    // blocks; stored split_stride floats apart
    int32_t ahead;                           // depth blocks of M and G to prefetch while the kernel before is at work (0: launches do not overlap)
    int32_t run;                             // ksplit or 1: so many consecutive tiles (those of one result tile) go to the
                                             // same CTA, which adds each to what it has stored
    int64_t rscale_off;                      // fp16 fused pass: scratch offset of 1 / (scale of R's plane)
    int64_t ld;                              // leading dimension of M, G, X
    ImgRef a, n1, n2;
    int64_t colsq_off;                       // scratch offset of the column-square partials
    int64_t cscale_off;                      // apply: scratch offset of a factor per result column (fp32), or -1
    float ef_a, ef_b, wc, wd;
    OutSpec out;
    // tensor maps of the images a, n1, n2 over the whole launch batch; the box of each map is the
    // tile or piece this launch loads with one instruction
    alignas(64) CUtensorMap map_a;
    alignas(64) CUtensorMap map_n1;
    alignas(64) CUtensorMap map_n2;
};

// ------------------------------------------------------------------------------------------
// PTX wrappers
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait: gives up after WAIT_LIMIT_CYCLES or as soon as another role of the CTA gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    int spins = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++spins & 63) == 0) {
            if (*abort_flag) return false;
            if (clock64() - t0 > WAIT_LIMIT_CYCLES) { *abort_flag = 1; return false; }
        }
    }
    return true;
}
// One tiled TMA load: the box of `map` at (0, row, panel, plane, matrix) -> shared memory, laid
// out [term][panel][row][128 bytes]; completes on the mbarrier with the full box size.
__device__ __forceinline__ void tma_load_box(uint32_t dst, const CUtensorMap* map, int row, int panel, int plane,
                                             int matrix, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(panel), "r"(plane), "r"(matrix), "r"(bar)
        : "memory");
}
// ---- CTA pairs (clusters of two CTAs on neighbouring SMs, tcgen05 cta_group::2) ----------------
// One MMA instruction of the pair's leader (cluster rank 0) multiplies M = 256 rows: each CTA
// supplies its own 128 rows of A and HALF of the N-side operand, and receives its 128 rows of the
// result in its own tensor memory.  Per CTA that halves the N-side bytes that are fetched from L2
// and read from shared memory by the tensor core.  Barriers that gather both CTAs (operand
// "full", accumulator "empty") live in the leader and are reached by remote arrives; barriers
// that release (operand "empty", accumulator "full") live in each CTA and are reached by the
// leader's multicast commit.  All of them keep the default (CTA-scope) semantics of the single-CTA
// barriers: with release/acquire at cluster scope on every arrive and wait the same kernels ran up
// to twice as long (the producer thread then pays a cluster-wide fence per load).
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx_remote(uint32_t cluster_addr, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%0], %1;"
                 ::"r"(cluster_addr), "r"(bytes) : "memory");
}
// Tiled TMA load of a CTA of a pair: the data lands in this CTA's shared memory, the bytes are
// counted on the mbarrier at cluster address `bar` (the leader's).
__device__ __forceinline__ void tma_load_box_pair(uint32_t dst, const CUtensorMap* map, int row, int panel, int plane,
                                                  int matrix, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(panel), "r"(plane), "r"(matrix), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t slot_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// D[tmem of both CTAs] (+)= A * B^T with M = 256; issued by one thread of the leader.
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// the mbarrier at offset `bar` of BOTH CTAs arrives once every MMA issued so far has completed
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(bar), "h"((uint16_t)3) : "memory");
}

__device__ __forceinline__ void prefetch_tensor_map(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
// Asynchronous 16-byte copy global -> shared (no register staging), grouped per thread.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void fence_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T, bf16 inputs, fp32 accumulation; issued by one thread.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// mbarrier arrives once every MMA issued so far by this thread has completed
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle.  K-major: rows of 128 bytes, 8-row groups
// 1024 bytes apart (stride offset), leading offset unused.  MN-major: lbo = distance between
// 64-element groups along M/N, sbo = distance between 8-deep groups along K.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;     // descriptor version of this architecture
    d |= (uint64_t)2 << 61;     // 128-byte swizzle
    return d;
}
// Instruction descriptor: fp32 accumulate, bf16 A and B, M = 128, N = n; a_mn / b_mn = 1 for an
// MN-major A / B operand (0: K-major).
// fmt: operand format, 1 = bf16, 0 = fp16 (both operands alike).
// m: rows of the instruction, 128, or 256 for an instruction of a CTA pair.
__device__ __forceinline__ uint32_t instr_desc(uint32_t n, uint32_t a_mn, uint32_t b_mn, uint32_t fmt = 1u,
                                               uint32_t m = (uint32_t)BM) {
    return (1u << 4) | (fmt << 7) | (fmt << 10) | (a_mn << 15) | (b_mn << 16) | ((n >> 3) << 17) |
           ((m >> 4) << 24);
}
template <bool PAIR>
__device__ __forceinline__ void umma_any(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    if (PAIR) umma_bf16_pair(d_tmem, adesc, bdesc, idesc, accumulate);
    else umma_bf16(d_tmem, adesc, bdesc, idesc, accumulate);
}
// The same with the descriptors given as halves (the high one is constant), always adding to D.
template <bool PAIR>
__device__ __forceinline__ void umma_add(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                         uint32_t idesc) {
    if (PAIR)
        asm volatile("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
                     "tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %5, 1;\n\t}"
                     ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc) : "memory");
    else
        asm volatile("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, 1;\n\t}"
                     ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc) : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void umma_halves(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                            uint32_t idesc, uint32_t accumulate) {
    umma_any<PAIR>(d_tmem, ((uint64_t)a_hi << 32) | a_lo, ((uint64_t)b_hi << 32) | b_lo, idesc, accumulate);
}
// NS 16-deep slices in one straight line: descriptors by additions, nothing else between the instructions.
template <bool PAIR, int NS, bool THREE>
__device__ __forceinline__ void umma_slices(uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi, uint32_t a_step,
                                            uint32_t b_step, uint32_t a_term, uint32_t b_term, uint32_t idesc, uint32_t accum) {
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        const uint32_t aj = a + j * a_step, bj = b + j * b_step;
        if (j == 0) umma_halves<PAIR>(d, aj, a_hi, bj, b_hi, idesc, accum);
        else umma_add<PAIR>(d, aj, a_hi, bj, b_hi, idesc);
        if (THREE) {
            umma_add<PAIR>(d, aj, a_hi, bj + b_term, b_hi, idesc);
            umma_add<PAIR>(d, aj + a_term, a_hi, bj, b_hi, idesc);
        }
    }
}
template <bool PAIR>
__device__ __forceinline__ void commit_any(uint32_t bar) {
    if (PAIR) umma_commit_pair(bar);
    else umma_commit(bar);
}

__device__ __forceinline__ void load8(const void* base, int64_t idx, int is_bf16, float (&v)[8]) {
    if (is_bf16) {
        uint4 u = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(base) + idx);
        v[0] = bf16lo_to_f32(u.x); v[1] = bf16hi_to_f32(u.x);
        v[2] = bf16lo_to_f32(u.y); v[3] = bf16hi_to_f32(u.y);
        v[4] = bf16lo_to_f32(u.z); v[5] = bf16hi_to_f32(u.z);
        v[6] = bf16lo_to_f32(u.w); v[7] = bf16hi_to_f32(u.w);
    } else {
        const float4* p = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(base) + idx);
        float4 x = p[0], y = p[1];
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
    }
}

// ------------------------------------------------------------------------------------------
// Pack kernel: fp32 matrix S (rows x cols, row-major, cols % 8 == 0) -> split image.
// One CTA per (panel, 128-row block), 256 threads; rows beyond `rows` are written as zeros.
// ------------------------------------------------------------------------------------------
struct PackArgs {
    Sel src;
    int32_t rows, cols;
    ImgRef dst;
    int32_t init, pad;      // first kernel of a step: clears the status word instead of reading it
};

template <class BATCH>
__global__ void __launch_bounds__(256)
pack_kernel(const __grid_constant__ BATCH batch, PackArgs a) {
    // (the first product, which follows, prefetches M and G before it waits: not while the step before is still writing M)
    grid_dependency_wait();
    grid_dependency_launch();
    const MatWork& w = batch.w[blockIdx.z];
    if (a.init) {
        if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *w.status = 0;
    } else if (*w.status & ST_FAILED) {
        return;
    }
    const float* S = pick(w, a.src);
    const int panel = blockIdx.x, rb = blockIdx.y;
    unsigned char* out0 = reinterpret_cast<unsigned char*>(w.scratch) + img_row_offset(a.dst, 0, panel, (int64_t)rb * 128);
    unsigned char* out1 = reinterpret_cast<unsigned char*>(w.scratch) + img_row_offset(a.dst, 1, panel, (int64_t)rb * 128);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int q = threadIdx.x + 256 * e;
        const int rho = q / 8, c = q % 8;
        const int64_t gr = (int64_t)rb * 128 + rho, gk = (int64_t)panel * 64 + c * 8;
        float v[8];
        if (gr < a.rows && gk < a.cols) {
            load8(S, gr * a.cols + gk, 0, v);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = 0.f;
        }
        uint4 t0, t1;
        split8(v, t0, t1);
        const int o = rho * 128 + img_chunk_offset(rho, c);
        *reinterpret_cast<uint4*>(out0 + o) = t0;
        *reinterpret_cast<uint4*>(out1 + o) = t1;
    }
}

// Power of two that brings the largest of `cols` squared column norms (cn) to a norm of about 2^10, for the fp16 plane of R
// in the single-pass fused feedback/update product (no entry can then overflow fp16, and typical entries stay far from the
// subnormal range); its inverse is left at *inverse, if there is such a place.  Called by 256 threads.
__device__ __forceinline__ float half_scale(const float* cn, int cols, float* inverse) {
    __shared__ float red[8];
    float mx = 0.f;
    for (int j = threadIdx.x; j < cols; j += 256) mx = fmaxf(mx, cn[j]);
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = mx;
    __syncthreads();
    mx = red[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) mx = fmaxf(mx, red[i]);
    int e = 0;
    const float nrm = sqrtf(mx);
    if (nrm > 0.f && nrm <= 3.0e38f) frexpf(nrm, &e);      // nrm = f * 2^e, 0.5 <= f < 1
    if (inverse && threadIdx.x == 0) *inverse = ldexpf(1.f, e - 10);
    return ldexpf(1.f, 10 - e);
}

// The fp16 plane of R; with `normalise` also column-normalised Dion's Q = R / column norms, fp32 and image planes, in the
// same pass over R (before: a normalisation that read R twice with one CTA per 32 columns, a pack of Q and one of R; the
// stages of a 1.1B model at r = 128 0.50 -> 0.24 ms, its step 7.23 -> 6.92; one 4096 x 4096 matrix at r = 256 0.314 -> 0.283).  cnorm holds the squared column norms of R.  One CTA
// per (panel, 128-row block), 256 threads.
struct PackRightArgs {
    int32_t rows, cols;
    ImgRef r_img, q_img;
    int32_t r_half;           // write R's fp16 plane
    int32_t normalise;        // bit mask of Q's image planes (1 | 2 bf16 terms, 4 fp16), 0: Q is not asked for
    int64_t cnorm_off, rscale_off;
};

template <class BATCH>
__global__ void __launch_bounds__(256)
pack_right_kernel(const __grid_constant__ BATCH batch, PackRightArgs a) {
    grid_dependency();
    const MatWork& w = batch.w[blockIdx.z];
    if (*w.status & ST_FAILED) return;
    const int panel = blockIdx.x, rb = blockIdx.y;
    const float* cn = reinterpret_cast<const float*>(w.scratch + a.cnorm_off);
    float scale = 1.f;
    if (a.r_half) scale = half_scale(cn, a.cols, panel == 0 && rb == 0 ? reinterpret_cast<float*>(w.scratch + a.rscale_off) : nullptr);
    unsigned char* scr = reinterpret_cast<unsigned char*>(w.scratch);
    const int c = threadIdx.x % 8;
    const int64_t gk = (int64_t)panel * 64 + c * 8;
    float inv[8] = {};
    if (a.normalise && gk < a.cols) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float nrm = sqrtf(cn[gk + i]);
            if (!(nrm > 0.f) && rb == 0 && threadIdx.x < 8) atomicOr(w.status, ST_ZEROCOL);
            inv[i] = nrm > 0.f ? 1.f / nrm : 0.f;
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int rho = threadIdx.x / 8 + 32 * e;
        const int64_t gr = (int64_t)rb * 128 + rho;
        const int o = img_chunk_offset(rho, c);
        float v[8] = {};
        const bool in = gr < a.rows && gk < a.cols;
        if (in) load8(w.R, gr * a.cols + gk, 0, v);
        if (a.r_half) *reinterpret_cast<uint4*>(scr + img_row_offset(a.r_img, 2, panel, gr) + o) = half8(v, scale);
        if (a.normalise) {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] *= inv[i];
            if (in) {
                float4* q = reinterpret_cast<float4*>(w.Q + gr * a.cols + gk);
                q[0] = make_float4(v[0], v[1], v[2], v[3]);
                q[1] = make_float4(v[4], v[5], v[6], v[7]);
            }
            if (a.normalise & 3) {
                uint4 t0, t1;
                split8(v, t0, t1);
                *reinterpret_cast<uint4*>(scr + img_row_offset(a.q_img, 0, panel, gr) + o) = t0;
                *reinterpret_cast<uint4*>(scr + img_row_offset(a.q_img, 1, panel, gr) + o) = t1;
            }
            if (a.normalise & 4) *reinterpret_cast<uint4*>(scr + img_row_offset(a.q_img, 2, panel, gr) + o) = half8(v, 1.f);
        }
    }
}

// ------------------------------------------------------------------------------------------
// Tile bookkeeping shared by all roles of the GEMM kernel
// ------------------------------------------------------------------------------------------
struct TileCoord { int b, mt, nt, n0, bn, kb_begin, kb_end, chunk; bool active, self; };    // self: the A tiles are the N side as well
// Each role remembers the status word of the matrix it is working on (nothing changes it while
// the kernel runs), so that only the first tile of a matrix pays for the global load.
struct StatusCache { int b = -1; int st = 0; };

// Pair launches (g.pair): a scheduled row tile is 256 rows, CTA `rank` of the pair owns its
// rows 128 * rank .. ; c.mt stays the 128-row tile index (it may lie one past the last tile when
// the number of tiles is odd: that CTA multiplies zeros and stores nothing).
template <bool V> struct BoolConst { static constexpr bool value = V; };

template <int EPI, class BATCH>
__device__ __forceinline__ TileCoord decode_tile(const BATCH& batch, const GemmArgs& g, int t, StatusCache& sc,
                                                 int rank, bool look = true) {         // look: at the status word (`active` counts)
    TileCoord c;
    const int per = g.m_tiles * g.n_tiles * g.ksplit;
    c.b = t / per;
    int rem = t - c.b * per;
    c.chunk = 0;
    if (g.ksplit > 1) { const int tl = rem / g.ksplit; c.chunk = rem - tl * g.ksplit; rem = tl; }
    const int mts = rem / g.n_tiles;
    c.nt = rem - mts * g.n_tiles;
    c.mt = g.pair ? 2 * mts + rank : mts;
    c.n0 = c.nt * g.BN;
    c.bn = min(g.BN, g.Ncols - c.n0);
    c.kb_begin = 0;
    c.kb_end = g.k_blocks;
    if (g.tri) c.kb_end = min(g.k_blocks, (c.n0 + c.bn + BK - 1) / BK);
    if (g.ksplit > 1) { c.kb_begin = c.chunk * g.kb_per_tile; c.kb_end = min(g.k_blocks, c.kb_begin + g.kb_per_tile); }
    if (look && c.b != sc.b) { sc.b = c.b; sc.st = *batch.w[c.b].status; }
    const int st = sc.st;
    c.active = !(st & ST_FAILED);
    if (EPI != EPI_K5 && g.out.only_if_shifted && !(st & g.out.shift_bit)) c.active = false;
    c.self = g.one_operand && c.n0 == (g.pair ? 2 * mts : mts) * BM;
    if (g.lower_only && c.n0 > (g.pair ? 2 * mts + 1 : c.mt) * BM + BM - 1) c.active = false;
    if (c.kb_begin >= c.kb_end) c.active = false;
    return c;
}

// N_IMG_MN: the pieces of depth block kb are its ks-deep slices that start below Kdim.
__device__ __forceinline__ int mn_pieces(const GemmArgs& g, int kb) {
    const int left = g.Kdim - kb * BK;
    return (min(left, BK) + g.ks - 1) / g.ks;
}
// ------------------------------------------------------------------------------------------
// The GEMM kernel.  D (128 x bn, fp32 in tensor memory) = A (128 x K) * N^T (bn x K).
//   warp 0        producer: bulk copies of image tiles into the A ring and the N ring
//   warp 1        MMA issuer, owns the tensor-memory allocation
//   next 4 or 8   epilogue warps (tensor memory -> registers -> global)
//   last 16       transform warps (A_BUF_* only): form B = M + G, split, write the A tile
// AMODE  where the A tile comes from and how it lies in shared memory
//          A_IMG_K / A_IMG_MN   image tile, K-major / MN-major
//          A_BUF_ROW            rows of B = M + G      (K-major;  Y = B Q_prev, Alg. 1, left-factor step)
//          A_BUF_COL            columns of B = M + G   (MN-major; R = B^T P,    Alg. 1, right-factor step)
// NMODE  N_IMG_K   pieces = 128-row chunks of the N range, 64 deep (image K-major; the fused pass)
//        N_IMG_MN  pieces = ks-deep slices of the whole N range (image MN-major)
// EPI    EPI_STORE  fp32 copy and/or split image (+ column-square partials) of D
//        EPI_K5     M <- a (M+G) - b D1,  X <- c X - d D2     (Alg. 1, update and error-feedback steps), D1 = P R^T, D2 = P Q^T
// XG     bit 0: G is bf16, bit 1: X is bf16
// ------------------------------------------------------------------------------------------
// RUN    the tiles come in runs (GemmArgs::run): the Gram product, and products with B that have more chunks than
//        accumulators.  (Instantiations of their own for the latter: the test for a run alone cost the other
//        products with B up to 1 % of a step, in registers that the transform warps then lack.)
template <class BATCH, int AMODE, int NMODE, int EPI, int XG, bool PAIR, bool RUN>
__global__ void __launch_bounds__(gemm_threads(AMODE, EPI), 1)
gemm_kernel(const __grid_constant__ BATCH batch, const __grid_constant__ GemmArgs g) {
    constexpr int NE = epi_warps(AMODE, EPI);
    // PAIR: launched in clusters of two; rank 0 (the leader) issues every MMA for both CTAs
    const int crank = PAIR ? (int)cluster_ctarank() : 0;
    constexpr bool A_BUF = a_is_buf(AMODE);
    const int tile0 = (PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x) * (RUN ? g.run : 1);
    const int tstride = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
    // the next tile of this CTA after tile t
    auto next = [&](int t) {
        if constexpr (!RUN) return t + tstride;
        else return (t + 1) % g.run ? t + 1 : t + 1 + (tstride - 1) * g.run;
    };
    constexpr bool A_MN = (AMODE == A_IMG_MN || AMODE == A_BUF_COL);
    constexpr bool SYM = AMODE == A_IMG_MN;          // Gram product
    constexpr bool G_BF16 = (XG & 1) != 0;
    constexpr bool X_BF16 = (XG & 2) != 0;

    if constexpr (EPI == EPI_STORE && !A_BUF) {
        // Third pass of a QR: mostly there is nothing to do, and a look at the status words is all (before: every tile's, with
        // barriers and tensor memory set up; 5 to 20 us a launch, now 4 to 6 cold).
        if (g.out.only_if_shifted) {
            grid_dependency();
            int any = 0;
            for (int i = threadIdx.x; i < batch.count; i += blockDim.x) {
                const int st = *batch.w[i].status;
                any |= !(st & ST_FAILED) && (st & g.out.shift_bit);
            }
            if (!__syncthreads_or(any)) return;          // (both CTAs of a pair alike)
        }
    }
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    unsigned char* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    unsigned char* a_ring = smem;
    unsigned char* n_ring = smem + g.a_slots * g.a_slot_bytes;
    unsigned char* staging = n_ring + (size_t)g.n_slots * g.n_piece_bytes;
    unsigned char* tail = staging + NE * (EPI == EPI_STORE ? STORE_STAGING_BYTES : g.epi_bufs * slab_bytes(XG));
    uint64_t* bars = reinterpret_cast<uint64_t*>(tail);
    const uint32_t a_full0 = smem_u32(bars), a_empty0 = a_full0 + 8 * MAX_A_SLOTS;
    const uint32_t n_full0 = a_empty0 + 8 * MAX_A_SLOTS, n_empty0 = n_full0 + 8 * MAX_N_SLOTS;
    const uint32_t tfull0 = n_empty0 + 8 * MAX_N_SLOTS, tempty0 = tfull0 + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * MAX_A_SLOTS + 2 * MAX_N_SLOTS + 4);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

    // Pairs: the "full" barriers of the operand rings and the "empty" barriers of the accumulators
    // that are used are the leader's; they count the arrivals of both CTAs.
    constexpr uint32_t NCTA = PAIR ? 2u : 1u;
    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_A_SLOTS; ++s) {
            mbar_init(a_full0 + 8 * s, NCTA * (A_BUF ? NUM_XF_WARPS : 1));
            mbar_init(a_empty0 + 8 * s, 1);
        }
        for (int s = 0; s < MAX_N_SLOTS; ++s) {
            mbar_init(n_full0 + 8 * s, NCTA);
            mbar_init(n_empty0 + 8 * s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(tfull0 + 8 * a, 1);
            mbar_init(tempty0 + 8 * a, NCTA * NE);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    if (warp == 0 && lane == 0) {
        if (!A_BUF) prefetch_tensor_map(&g.map_a);
        prefetch_tensor_map(&g.map_n1);
        if (EPI == EPI_K5) prefetch_tensor_map(&g.map_n2);
    }
    grid_dependency_launch();
    if (warp == 1) {
        if (PAIR) tmem_alloc_pair(smem_u32(tmem_slot), (uint32_t)g.tmem_cols);
        else tmem_alloc(smem_u32(tmem_slot), (uint32_t)g.tmem_cols);
    }
    tc_fence_before();
    StatusCache scache;
    if constexpr (!A_BUF) {
        grid_dependency_wait();
        // (most often the matrix of the first tile: on its way while the CTA gathers)
        scache.b = 0; scache.st = *batch.w[0].status;
    }
    __syncthreads();
    if (PAIR) cluster_sync_all();       // the peer's barriers are initialised before anything reaches them
    tc_fence_after();
    if constexpr (A_BUF) {
        // (the transform warps have something to do first, see there)
        if (warp < 2 + NE) grid_dependency_wait();
    }
    // cluster addresses of the leader's gathering barriers (slot s: + 8 s)
    const uint32_t a_full_ld = PAIR ? map_to_rank(a_full0, 0) : a_full0;
    const uint32_t n_full_ld = PAIR ? map_to_rank(n_full0, 0) : n_full0;
    const uint32_t tempty_ld = PAIR ? map_to_rank(tempty0, 0) : tempty0;
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t acc_stride = (uint32_t)(g.tmem_cols / g.acc_bufs);

    const int a_terms = g.a_slot_bytes / A_TERM_BYTES;
    const int n1_terms = g.passes == 3 ? 2 : 1;
    const int plane = g.fp16 ? 2 : 0;
    const uint32_t fmt = g.fp16 ? 0u : 1u;
    // N_IMG_MN piece geometry: [term][64-column group][ks rows of 128 bytes]
    const uint32_t group_stride = (uint32_t)g.ks * 128u;
    const uint32_t mn_term_stride = PAIR ? 2u * group_stride : (uint32_t)((g.BN + 63) / 64) * group_stride;

    if (warp == 0) {
        // ---------------- producer ----------------
        // One thread feeds both rings.  It walks the schedule twice, with one cursor per ring, and
        // serves whichever ring has a free slot, so a full N ring never holds back A tiles (and
        // the other way round).  Every slot is filled by one tiled TMA load (two for the fused
        // pass: R and Q pieces).
        if (lane == 0) {
            int as = 0, ns = 0; uint32_t aph = 0, nph = 0;
            // cursor over (tile, depth block) for the A ring
            int at = tile0, akb = -1; TileCoord ac{}; bool a_done = A_BUF;      // akb < 0: tile not decoded yet
            // cursor over (tile, depth block, piece) for the N ring
            int nt_ = tile0, nkb = -1, npc = 0; TileCoord nc{}; bool n_done = false;
            auto a_seek = [&]() {           // make (at, akb) valid or finish
                while (!a_done) {
                    if (at >= g.total_tiles) { a_done = true; break; }
                    if (akb < 0) { ac = decode_tile<EPI>(batch, g, at, scache, crank); akb = ac.kb_begin; }
                    if (ac.active && akb < ac.kb_end) break;
                    at = next(at); akb = -1;
                }
            };
            auto n_pieces = [&](int kb) { return NMODE == N_IMG_MN ? mn_pieces(g, kb) : g.n_split ? 2 : 1; };
            auto n_seek = [&]() {           // make (nt_, nkb, npc) valid or finish
                while (!n_done) {
                    if (nt_ >= g.total_tiles) { n_done = true; break; }
                    if (nkb < 0) { nc = decode_tile<EPI>(batch, g, nt_, scache, crank); nkb = nc.kb_begin; npc = 0; }
                    if (!nc.active || (SYM && nc.self) || nkb >= nc.kb_end) { nt_ = next(nt_); nkb = -1; npc = 0; continue; }
                    if (npc >= n_pieces(nkb)) { ++nkb; npc = 0; continue; }
                    break;
                }
            };
            a_seek();
            n_seek();
            long long idle_since = -1;
            while (!a_done || !n_done) {
                bool progress = false;
                if (!a_done && mbar_try_wait(a_empty0 + 8 * as, aph ^ 1)) {
                    const uint32_t dst = smem_u32(a_ring + as * g.a_slot_bytes);
                    if (PAIR) {
                        const uint32_t fb = a_full_ld + 8 * as;
                        mbar_arrive_expect_tx_remote(fb, (uint32_t)a_terms * A_TERM_BYTES);
                        if (AMODE == A_IMG_K) tma_load_box_pair(dst, &g.map_a, ac.mt * BM, akb, plane, ac.b, fb);
                        else tma_load_box_pair(dst, &g.map_a, akb * BK, ac.mt * 2, plane, ac.b, fb);
                    } else {
                        const uint32_t fb = a_full0 + 8 * as;
                        mbar_arrive_expect_tx(fb, (uint32_t)a_terms * A_TERM_BYTES);
                        if (AMODE == A_IMG_K) tma_load_box(dst, &g.map_a, ac.mt * BM, akb, plane, ac.b, fb);
                        else tma_load_box(dst, &g.map_a, akb * BK, ac.mt * 2, plane, ac.b, fb);
                    }
                    if (++as == g.a_slots) { as = 0; aph ^= 1; }
                    ++akb;
                    if (akb >= ac.kb_end) { at = next(at); akb = -1; }
                    a_seek();
                    progress = true;
                }
                if (!n_done && mbar_try_wait(n_empty0 + 8 * ns, nph ^ 1)) {
                    const uint32_t fb = PAIR ? n_full_ld + 8 * ns : n_full0 + 8 * ns;
                    const uint32_t dst = smem_u32(n_ring + (size_t)ns * g.n_piece_bytes);
                    if (PAIR) {
                        // this CTA's half of the N-side: per 256-column block its two 64-column groups
                        // (MN-major), or the R piece (leader) / the Q piece (peer) of the fused pass
                        mbar_arrive_expect_tx_remote(fb, (uint32_t)g.n_piece_bytes);
                        if (NMODE == N_IMG_MN) {
                            const uint32_t blk_bytes = (uint32_t)n1_terms * 2u * group_stride;
                            for (int blk = 0; blk * 256 < nc.bn; ++blk)
                                tma_load_box_pair(dst + blk * blk_bytes, &g.map_n1, nkb * BK + npc * g.ks,
                                                  nc.n0 / 64 + blk * 4 + crank * 2, plane, nc.b, fb);
                        } else {
                            tma_load_box_pair(dst, crank == 0 ? &g.map_n1 : &g.map_n2, nc.n0, nkb, plane, nc.b, fb);
                        }
                    } else {
                        if (NMODE == N_IMG_MN) {
                            mbar_arrive_expect_tx(fb, (uint32_t)g.n_piece_bytes);
                            tma_load_box(dst, &g.map_n1, nkb * BK + npc * g.ks, nc.n0 / 64, plane, nc.b, fb);
                        } else if (g.n_split) {
                            mbar_arrive_expect_tx(fb, (uint32_t)((npc == 0 ? n1_terms : g.passes2 == 3 ? 2 : 1) * A_TERM_BYTES));
                            tma_load_box(dst, npc == 0 ? &g.map_n1 : &g.map_n2, nc.n0, nkb, plane, nc.b, fb);
                        } else {
                            mbar_arrive_expect_tx(fb, (uint32_t)g.n_piece_bytes);
                            tma_load_box(dst, &g.map_n1, nc.n0, nkb, plane, nc.b, fb);
                            tma_load_box(dst + n1_terms * A_TERM_BYTES, &g.map_n2, nc.n0, nkb, plane, nc.b, fb);
                        }
                    }
                    if (++ns == g.n_slots) { ns = 0; nph ^= 1; }
                    ++npc;
                    n_seek();
                    progress = true;
                }
                if (progress) {
                    idle_since = -1;
                } else {
                    if (*abort_flag) break;
                    const long long now = clock64();
                    if (idle_since < 0) idle_since = now;
                    else if (now - idle_since > WAIT_LIMIT_CYCLES) { *abort_flag = 1; break; }
                }
            }
        }
    } else if (warp == 1 && NMODE == N_IMG_MN) {
        // ---------------- MMA issuer, MN-major N-side (products with B, Gram, apply) ----------------
        // One thread runs the whole loop.  Its scalar work bounds the products of small rank (a few warps of other
        // roles share its scheduler, so every instruction costs several cycles): what an instruction of the tensor
        // core needs is a pair of 32-bit additions, whole pieces have no inner loop, and nothing is recomputed
        // per depth block.  One 11008 x 4096 matrix, r = 32 / 128: 2240 / 2160 -> 1500 / 1550 cycles a
        // depth block beside the waits for operands.
        if (lane == 0 && crank == 0) {
            constexpr uint32_t MROWS = PAIR ? 256u : 128u;
            constexpr uint32_t a_step = A_MN ? (2048u >> 4) : (32u >> 4), b_step = 2048u >> 4;     // one 16-deep slice
            constexpr uint32_t a_term = A_TERM_BYTES >> 4;
            const uint64_t a_desc = A_MN ? smem_desc(0, 8192, 1024) : smem_desc(0, 16, 1024);
            const uint64_t b_desc = smem_desc(0, group_stride, 1024);
            const uint32_t a_hi = (uint32_t)(a_desc >> 32), b_hi = (uint32_t)(b_desc >> 32);
            const uint32_t a_base = (uint32_t)a_desc + (smem_u32(a_ring) >> 4), b_base = (uint32_t)b_desc + (smem_u32(n_ring) >> 4);
            const uint32_t a_slot = (uint32_t)g.a_slot_bytes >> 4, b_slot = (uint32_t)g.n_piece_bytes >> 4;
            const uint32_t b_term = mn_term_stride >> 4;
            // 256 columns further on: four 64-column groups, or this CTA's two with both terms (pairs)
            const uint32_t b_block = (PAIR ? (uint32_t)n1_terms * 2u * group_stride : 4u * group_stride) >> 4;
            const bool three = g.passes == 3;
            const int a_slots = g.a_slots, n_slots = g.n_slots, ks = g.ks, kdim = g.Kdim;
            const uint32_t idesc_256 = instr_desc(256u, A_MN ? 1u : 0u, 1u, fmt, MROWS);
            int as = 0, ns = 0; uint32_t aph = 0, nph = 0;
            int acc = 0; uint32_t acc_phase = 0;
            bool ok = true;
            for (int t = tile0; t < g.total_tiles && ok; t = next(t)) {
                const TileCoord c = decode_tile<EPI>(batch, g, t, scache, crank);
                if (!c.active) continue;
                if (!mbar_wait(tempty0 + 8 * acc, acc_phase ^ 1, abort_flag)) { ok = false; break; }
                // orders this tile's MMAs after the epilogue's tensor-memory loads.  (The operand waits
                // below need no tcgen05 fence: the operands arrive through the async proxy or behind
                // a proxy fence, and a fence per piece stalled the issuer for hundreds of cycles.)
                tc_fence_after();
                uint32_t d = tmem_base + acc * acc_stride, accum = 0;
                const uint32_t idesc_last = instr_desc((uint32_t)((c.bn - 1) % 256 + 1), A_MN ? 1u : 0u, 1u, fmt, MROWS);
                // depth blocks left of the chunk that has the accumulator at d
                int chunk_left = A_BUF && g.acc_chunks > 1 ? g.kb_per_chunk : c.kb_end - c.kb_begin;
                for (int kb = c.kb_begin; kb < c.kb_end && ok; ++kb) {
                    if (chunk_left-- == 0) { chunk_left = g.kb_per_chunk - 1; d += (uint32_t)g.BN; accum = 0; }
                    if (!mbar_wait(a_full0 + 8 * as, aph, abort_flag)) { ok = false; break; }
                    uint32_t a = a_base + as * a_slot;
                    if (SYM && c.self) {
                        // The A tile, in the layout that a 64-deep piece of its columns has on the N side: a third to all of the
                        // Gram tiles' operands from L2 saved (Gram products of a step, 1.1B model r = 512 2.75 -> 2.42 ms, 8B stage
                        // 2.50 -> 2.19; one 11008 x 4096 matrix r = 128, step 507 -> 497 us).
                        const int depth = min(BK, kdim - kb * BK);
                        if (three && depth == 64) {
                            umma_slices<PAIR, 4, true>(d, a, a_hi, a, a_hi, a_step, a_step, a_term, a_term, idesc_last, accum);
                        } else {
                            for (int j = 0; j * 16 < depth; ++j) {
                                const uint32_t acc_j = j > 0 ? 1u : accum, aj = a + j * a_step;
                                if (three) umma_slices<PAIR, 1, true>(d, aj, a_hi, aj, a_hi, 0, 0, a_term, a_term, idesc_last, acc_j);
                                else umma_slices<PAIR, 1, false>(d, aj, a_hi, aj, a_hi, 0, 0, 0, 0, idesc_last, acc_j);
                            }
                        }
                        accum = 1;
                    } else
                    for (int left = min(BK, kdim - kb * BK); left > 0; left -= ks) {
                        if (!mbar_wait(n_full0 + 8 * ns, nph, abort_flag)) { ok = false; break; }
                        uint32_t b = b_base + ns * b_slot, dc = d;
                        const int depth = min(ks, left);
                        for (int cols = c.bn; cols > 0; cols -= 256) {
                            const uint32_t idesc = cols < 256 ? idesc_last : idesc_256;
                            if (three && depth == 64) {
                                umma_slices<PAIR, 4, true>(dc, a, a_hi, b, b_hi, a_step, b_step, a_term, b_term, idesc, accum);
                            } else if (three && depth == 32) {
                                umma_slices<PAIR, 2, true>(dc, a, a_hi, b, b_hi, a_step, b_step, a_term, b_term, idesc, accum);
                            } else if (three && depth <= 16) {
                                umma_slices<PAIR, 1, true>(dc, a, a_hi, b, b_hi, a_step, b_step, a_term, b_term, idesc, accum);
                            } else if (!three && depth == 64) {
                                umma_slices<PAIR, 4, false>(dc, a, a_hi, b, b_hi, a_step, b_step, a_term, b_term, idesc, accum);
                            } else {
                                for (int j = 0; j * 16 < depth; ++j) {
                                    const uint32_t acc_j = j > 0 ? 1u : accum, aj = a + j * a_step, bj = b + j * b_step;
                                    umma_halves<PAIR>(dc, aj, a_hi, bj, b_hi, idesc, acc_j);
                                    if (three) {
                                        umma_add<PAIR>(dc, aj, a_hi, bj + b_term, b_hi, idesc);
                                        umma_add<PAIR>(dc, aj + a_term, a_hi, bj, b_hi, idesc);
                                    }
                                }
                            }
                            b += b_block; dc += 256;
                        }
                        accum = 1;
                        a += (ks / 16) * a_step;
                        commit_any<PAIR>(n_empty0 + 8 * ns);
                        if (++ns == n_slots) { ns = 0; nph ^= 1; }
                    }
                    if (!ok) break;
                    commit_any<PAIR>(a_empty0 + 8 * as);
                    if (++as == a_slots) { as = 0; aph ^= 1; }
                }
                if (!ok) break;
                commit_any<PAIR>(tfull0 + 8 * acc);
                if (++acc == g.acc_bufs) { acc = 0; acc_phase ^= 1; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer, K-major N-side (fused pass) ----------------
        // One thread issues.  A tcgen05.mma of N = 256 occupies the tensor core for 128 cycles, so the
        // scalar work per instruction has to stay at a handful of operations: every descriptor is a
        // constant high part plus (shared address >> 4), advanced by additions only.
        static_assert(NMODE == N_IMG_MN || (EPI == EPI_K5 && AMODE == A_IMG_K), "only the fused pass has a K-major N-side");
        int as = 0, ns = 0; uint32_t aph = 0, nph = 0;
        int acc = 0; uint32_t acc_phase = 0;
        bool ok = true;
        // descriptor high parts (layout, strides) and address units of 16 bytes
        const uint64_t op_desc = smem_desc(0, 16, 1024);
        const uint32_t op_lo = (uint32_t)op_desc, op_hi = (uint32_t)(op_desc >> 32);
        const uint32_t slice16 = 32u >> 4;               // one 16-deep slice of either operand
        const uint32_t a_ring16 = smem_u32(a_ring) >> 4, n_ring16 = smem_u32(n_ring) >> 4;
        const uint32_t a_slot16 = (uint32_t)g.a_slot_bytes >> 4, n_slot16 = (uint32_t)g.n_piece_bytes >> 4;
        constexpr uint32_t MROWS = PAIR ? 256u : 128u;
        for (int t = tile0; t < g.total_tiles && ok && crank == 0; t = next(t)) {
            const TileCoord c = decode_tile<EPI>(batch, g, t, scache, crank);
            if (!c.active) continue;
            if (!mbar_wait(tempty0 + 8 * acc, acc_phase ^ 1, abort_flag)) { ok = false; break; }
            tc_fence_after();        // as in the issuer above
            const uint32_t dacc = tmem_base + acc * acc_stride;
            for (int kb = c.kb_begin; kb < c.kb_end && ok; ++kb) {
                if (!mbar_wait(a_full0 + 8 * as, aph, abort_flag)) { ok = false; break; }
                const int nsl = min(4, (g.Kdim - kb * BK + 15) / 16);
                // N of the instruction must be a multiple of 16: round a ragged last tile up
                // (rows beyond the matrix are zero in the images; those columns of D are never stored)
                const uint32_t ncols = (uint32_t)((c.bn + 15) / 16 * 16);
                const uint32_t accum = kb > c.kb_begin ? 1u : 0u;
                for (int pc = 0; pc < (g.n_split ? 2 : 1) && ok; ++pc) {
                    if (!mbar_wait(n_full0 + 8 * ns, nph, abort_flag)) { ok = false; break; }
                    if (lane == 0) {
                        const uint32_t a0 = (uint32_t)op_lo + a_ring16 + as * a_slot16, b0 = (uint32_t)op_lo + n_ring16 + ns * n_slot16;
                        if (g.passes == 1 && g.passes2 == 1) {
                            // Single-term operands: the R piece and the Q piece lie back
                            // to back in the slot (256 rows of one K-major tile) and their accumulators in
                            // adjacent columns, so one N = 256 instruction serves both products and reads
                            // the P slice from shared memory once (two of them on a ragged last tile).
                            if (ncols == 128) {
                                const uint32_t idesc = instr_desc(256u, 0u, 0u, fmt, MROWS);
                                for (int j = 0; j < nsl; ++j)
                                    umma_slices<PAIR, 1, false>(dacc, a0 + j * slice16, op_hi, b0 + j * slice16, op_hi, 0, 0, 0, 0, idesc, j ? 1u : accum);
                            } else {
                                const uint32_t idesc = instr_desc(ncols, 0u, 0u, fmt, MROWS);
                                for (int j = 0; j < nsl; ++j) {
                                    umma_slices<PAIR, 1, false>(dacc, a0 + j * slice16, op_hi, b0 + j * slice16, op_hi, 0, 0, 0, 0, idesc, j ? 1u : accum);
                                    umma_slices<PAIR, 1, false>(dacc + g.BN, a0 + j * slice16, op_hi, b0 + (A_TERM_BYTES >> 4) + j * slice16, op_hi, 0, 0, 0, 0,
                                                                idesc, j ? 1u : accum);
                                }
                            }
                        } else {
                            // (never a pair) split terms: the slot holds those of R and Q, or of one of them.  In straight lines: the
                            // issuer bounds this form (28 matrices 2048 wide at r = 256 with three passes for M, step with descriptors
                            // rebuilt in a loop over products 2.04, now 1.95 ms).
                            const uint32_t idesc = instr_desc(ncols, 0u, 0u, fmt, MROWS);
                            constexpr uint32_t term = A_TERM_BYTES >> 4;
                            auto product = [&](uint32_t d, uint32_t b, bool three) {
                                if (nsl == 4) {
                                    if (three) umma_slices<PAIR, 4, true>(d, a0, op_hi, b, op_hi, slice16, slice16, term, term, idesc, accum);
                                    else umma_slices<PAIR, 4, false>(d, a0, op_hi, b, op_hi, slice16, slice16, 0, 0, idesc, accum);
                                    return;
                                }
                                for (int j = 0; j < nsl; ++j) {
                                    const uint32_t aj = a0 + j * slice16, bj = b + j * slice16, acc_j = j ? 1u : accum;
                                    if (three) umma_slices<PAIR, 1, true>(d, aj, op_hi, bj, op_hi, 0, 0, term, term, idesc, acc_j);
                                    else umma_slices<PAIR, 1, false>(d, aj, op_hi, bj, op_hi, 0, 0, 0, 0, idesc, acc_j);
                                }
                            };
                            if (!g.n_split) {
                                product(dacc, b0, g.passes == 3);
                                product(dacc + g.BN, b0 + n1_terms * term, g.passes2 == 3);
                            } else {
                                product(dacc + pc * g.BN, b0, (pc ? g.passes2 : g.passes) == 3);
                            }
                        }
                        commit_any<PAIR>(n_empty0 + 8 * ns);
                    }
                    __syncwarp();
                    if (++ns == g.n_slots) { ns = 0; nph ^= 1; }
                }
                if (!ok) break;
                if (lane == 0) commit_any<PAIR>(a_empty0 + 8 * as);
                __syncwarp();
                if (++as == g.a_slots) { as = 0; aph ^= 1; }
            }
            if (!ok) break;
            if (lane == 0) commit_any<PAIR>(tfull0 + 8 * acc);
            __syncwarp();
            if (++acc == g.acc_bufs) { acc = 0; acc_phase ^= 1; }
        }
    } else if (warp < 2 + NE) {
        // ---------------- epilogue ----------------
        int acc = 0; uint32_t acc_phase = 0;
        bool ok = true;
        const int quarter = warp % 4;                    // tensor-memory lanes 32*quarter .. +31
        if (EPI == EPI_STORE) {
            int scale_b = -1; bool scale_on = false;         // does matrix scale_b want its columns scaled
            for (int t = tile0; t < g.total_tiles && ok; t = next(t)) {
                const TileCoord c = decode_tile<EPI>(batch, g, t, scache, crank);
                if (!c.active) continue;
                const MatWork& w = batch.w[c.b];
                const float* cscale = nullptr;
                if constexpr (!A_BUF) {
                    if (g.cscale_off >= 0) {
                        // (rarely asked for: looked up once per matrix, while its first accumulator is formed)
                        const float* f = reinterpret_cast<const float*>(w.scratch + g.cscale_off);
                        if (c.b != scale_b) { scale_b = c.b; scale_on = f[g.Ncols] != 0.f; }
                        if (scale_on) cscale = f;
                    }
                }
                const int stw = scache.st;
                const Dest& d = (g.out.shift_bit && (stw & g.out.shift_bit)) ? g.out.shifted : g.out.normal;
                const uint32_t taddr = tmem_base + acc * acc_stride + ((uint32_t)(quarter * 32) << 16);
                float* C = d.has_f32 ? pick(w, d.f32) + (int64_t)c.chunk * g.split_stride : nullptr;
                unsigned char* scr = reinterpret_cast<unsigned char*>(w.scratch);
                // (a run of tiles with chunks of their own: image and column squares when the sum is complete)
                const bool whole = !(A_BUF && RUN) || c.chunk == g.run - 1;
                const bool add = !A_BUF && RUN && g.run > 1 && c.chunk > 0;      // Gram product: to what this very thread has stored
                const bool to_img = d.img.off >= 0 && whole;
                float* csq = d.colsq && whole ? reinterpret_cast<float*>(w.scratch + g.colsq_off) +
                                           (int64_t)(c.mt * 4 + quarter) * g.Ncols : nullptr;
                // 32 columns at a time: this warp's 32 x 32 block goes through a 4 KB staging buffer so that
                // global stores run along rows: 8 lines per instruction where one row per lane took 32.  Tiles
                // of 512 columns leave no second accumulator, and the tensor core waits for this (19 % of the first
                // product and 33 % of the second at r = 512, before).  First and second product: six layers of
                // 2048-wide matrices, r = 192 0.772 -> 0.699 and 0.768 -> 0.700 ms, r = 512 0.873 -> 0.870 and 1.044 -> 0.933; 24 layers of 768-wide ones, r = 192 0.407 -> 0.385 and 0.472 -> 0.417.
                // One rolled loop for all products: in launches of a tile or two its code is fetched as it is run.  (Image products in
                // unrolled blocks of 64 columns on four warps: 12000 of the 21000 cycles of a one-tile apply.)
                unsigned char* stg = staging + (warp - 2) * STORE_STAGING_BYTES;
                const int64_t gi0 = (int64_t)c.mt * BM + quarter * 32;
                // (pairs: the CTA whose rows lie beyond the matrix stores nothing)
                const bool has_rows = !PAIR || (int64_t)c.mt * BM < g.Mrows;
                const int bn64 = !has_rows ? 0 : (to_img ? (c.bn + 63) / 64 * 64 : c.bn);
                // (the last tile of a run may have fewer chunks than the others)
                const int tile_chunks = !A_BUF ? 1 : RUN && c.chunk > 0 ? (c.kb_end - c.kb_begin + g.kb_per_chunk - 1) / g.kb_per_chunk : g.acc_chunks;
                const int srow = lane / 4, sch = lane % 4;      // stores: 8 rows x 4 chunks of 8 columns per step
                // Image products: before the first tile's accumulator is there, one trial run of the loop that stores nothing (its
                // code then is in the instruction cache).
                const int cc0 = (warp - 2) / 4 * 32;
                bool live = A_BUF || t != tile0;
                if (live) {
                    if (!mbar_wait(tfull0 + 8 * acc, acc_phase, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                }
                for (int cc = cc0; cc < bn64; cc += 8 * NE) {
                    uint32_t v[2][16];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (cc + 16 * h < c.bn && live) {
                            tmem_ld16(taddr + cc + 16 * h, v[h]);
                        } else {
#pragma unroll
                            for (int i = 0; i < 16; ++i) v[h][i] = 0u;
                        }
                    }
                    tmem_ld_wait();
                    if (!A_BUF && cscale) {
#pragma unroll
                        for (int i = 0; i < 32; i += 4) {
                            if (cc + i < c.bn) {
                                const float4 f = *reinterpret_cast<const float4*>(cscale + c.n0 + cc + i);
                                const float fe[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    v[i / 16][i % 16 + e] = __float_as_uint(__uint_as_float(v[i / 16][i % 16 + e]) * fe[e]);
                            }
                        }
                    }
                    if (A_BUF && RUN && c.chunk > 0 && gi0 + lane < g.Mrows) {
                        // the sum so far of this lane's row, stored by this warp
                        const float* o = C + (gi0 + lane) * g.out.ld + c.n0 + cc;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (cc + 16 * h < c.bn) {
#pragma unroll
                                for (int i = 0; i < 16; i += 4) {
                                    const float4 x = *reinterpret_cast<const float4*>(o + 16 * h + i);
                                    v[h][i] = __float_as_uint(x.x + __uint_as_float(v[h][i]));
                                    v[h][i + 1] = __float_as_uint(x.y + __uint_as_float(v[h][i + 1]));
                                    v[h][i + 2] = __float_as_uint(x.z + __uint_as_float(v[h][i + 2]));
                                    v[h][i + 3] = __float_as_uint(x.w + __uint_as_float(v[h][i + 3]));
                                }
                            }
                        }
                    }
                    for (int ch = 1; ch < tile_chunks; ++ch) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (cc + 16 * h < c.bn) {
                                uint32_t u[16];
                                tmem_ld16(taddr + ch * g.BN + cc + 16 * h, u);
                                tmem_ld_wait();
#pragma unroll
                                for (int i = 0; i < 16; ++i)
                                    v[h][i] = __float_as_uint(__uint_as_float(v[h][i]) + __uint_as_float(u[i]));
                            }
                        }
                    }
#pragma unroll
                    for (int ch = 0; ch < 8; ++ch)
                        *reinterpret_cast<uint4*>(stg + lane * 128 + img_chunk_offset(lane, ch)) =
                            make_uint4(v[ch / 4][ch % 4 * 4], v[ch / 4][ch % 4 * 4 + 1], v[ch / 4][ch % 4 * 4 + 2], v[ch / 4][ch % 4 * 4 + 3]);
                    __syncwarp();
                    const int gj = c.n0 + cc;
                    if (csq) {
                        // column sums of squares over the 32 rows of this warp
                        float sum;
                        if constexpr (A_BUF) {
                            // in registers (22 warps leave none for addresses): fold 32 values over the five lane bits, after
                            // which every lane has the sum of one column
                            float s[32];
#pragma unroll
                            for (int i = 0; i < 32; ++i) { const float x = __uint_as_float(v[i / 16][i % 16]); s[i] = __fmul_rn(x, x); }
#pragma unroll
                            for (int half = 16; half >= 1; half >>= 1) {
                                const bool up = (lane & half) != 0;
#pragma unroll
                                for (int i = 0; i < 16; ++i) {
                                    if (i < half) {
                                        const float send = up ? s[i] : s[i + half];
                                        const float keep = up ? s[i + half] : s[i];
                                        s[i] = keep + __shfl_xor_sync(0xffffffffu, send, half);
                                    }
                                }
                            }
                            sum = s[0];
                        } else {
                            // a column per lane, in less code
                            float q[4] = {};
#pragma unroll 2
                            for (int i = 0; i < 32; i += 4)
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    const float x = *reinterpret_cast<const float*>(stg + (i + e) * 128 + img_chunk_offset(i + e, lane / 4) + lane % 4 * 4);
                                    q[e] = fmaf(x, x, q[e]);
                                }
                            sum = (q[0] + q[1]) + (q[2] + q[3]);
                        }
                        if (cc + lane < c.bn && live) csq[gj + lane] = sum;
                    }
                    // (the image has 128 rows per tile, the fp32 result only those of the matrix)
                    const int rows = live ? (int)min((int64_t)32, g.Mrows - gi0) - srow : 0;
                    const bool col_in = cc + sch * 8 < c.bn;
                    float* Cp = C + (gi0 + srow) * g.out.ld + gj + sch * 8;
                    unsigned char* ip = scr + (to_img ? img_row_offset(d.img, 0, gj / 64, gi0 + srow) : 0) +
                                        img_chunk_offset(srow, gj % 64 / 8 + sch);
                    const int64_t plane_bytes = (int64_t)d.img.panels * d.img.rows_pad * 128;
                    // (all loads first: one behind a store that may alias it would wait for the store)
                    float4 old[4][2];
                    if (add) {
#pragma unroll
                        for (int it = 0; it < 4; ++it) {
                            const bool in = it * 8 < rows && col_in;
                            old[it][0] = in ? *reinterpret_cast<const float4*>(Cp + it * 8 * g.out.ld) : make_float4(0.f, 0.f, 0.f, 0.f);
                            old[it][1] = in ? *reinterpret_cast<const float4*>(Cp + it * 8 * g.out.ld + 4) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                    }
#pragma unroll
                    for (int it = 0; it < 4; ++it) {
                        const unsigned char* sp = stg + (it * 8 + srow) * 128;
                        float4 x = *reinterpret_cast<const float4*>(sp + img_chunk_offset(srow, 2 * sch));
                        float4 y = *reinterpret_cast<const float4*>(sp + img_chunk_offset(srow, 2 * sch + 1));
                        if (add) {
                            x = make_float4(old[it][0].x + x.x, old[it][0].y + x.y, old[it][0].z + x.z, old[it][0].w + x.w);
                            y = make_float4(old[it][1].x + y.x, old[it][1].y + y.y, old[it][1].z + y.z, old[it][1].w + y.w);
                        }
                        if (C && it * 8 < rows && col_in) {
                            *reinterpret_cast<float4*>(Cp + it * 8 * g.out.ld) = x;
                            *reinterpret_cast<float4*>(Cp + it * 8 * g.out.ld + 4) = y;
                        }
                        if (to_img) {
                            const bool st = A_BUF || live;
                            const float f[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
                            uint4 t0, t1;
                            split8(f, t0, t1);
                            if (st) *reinterpret_cast<uint4*>(ip + it * 1024) = t0;
                            if (st) *reinterpret_cast<uint4*>(ip + plane_bytes + it * 1024) = t1;
                            if (d.img.planes == 3 && st) *reinterpret_cast<uint4*>(ip + 2 * plane_bytes + it * 1024) = half8(f, 1.f);
                        }
                    }
                    __syncwarp();
                    if (!live) {
                        if (!mbar_wait(tfull0 + 8 * acc, acc_phase, abort_flag)) { ok = false; break; }
                        tc_fence_after();
                        live = true;
                        cc = cc0 - 8 * NE;
                    }
                }
                if (!ok) break;
                if (!live) {        // (no columns here: the accumulator is only handed on)
                    if (!mbar_wait(tfull0 + 8 * acc, acc_phase, abort_flag)) { ok = false; break; }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) { if (PAIR) mbar_arrive_remote(tempty_ld + 8 * acc); else mbar_arrive(tempty0 + 8 * acc); }
                if (++acc == g.acc_bufs) { acc = 0; acc_phase ^= 1; }
            }
        } else {
            // Fused error feedback and weight update.  Warp (quarter, half) owns rows
            // 32*quarter.. of the tile and columns 64*half.., in two slabs of 32 x 32.  The two
            // accumulator slabs go through a swizzled staging block so that global accesses run
            // along rows (8 lanes x 16 bytes per row).
            const int half = (warp - 2) / 4;
            // The 32 x 32 slabs of M, G, X come in by asynchronous copies (cp.async, no registers) into a per-warp buffer,
            // one or two slabs ahead; each
            // lane then updates its own row in place (accumulators stay in the layout tensor
            // memory gives: one row per lane), and the buffer goes out along rows.
            //   buffer: M | G | X, rows of 128 bytes (fp32) or 64 (bf16), 16-byte chunks swizzled so that
            //   both the row-per-lane and the 8-(or 4-)lanes-per-row accesses avoid bank conflicts
            // (fp32 G or X were fetched into registers, when the slab before was done, and a depth block's operands had one
            // slot.  Step before -> now: 28 matrices 2048 wide, Dion, fp32 X and G, r = 64 1.83 -> 1.50 ms, fp32 X r = 256 2.32 -> 2.19; one
            // 4096 x 4096 matrix r = 128, fp32 X and G 0.399 -> 0.364, fp32 G 0.386 -> 0.359.)
            constexpr int SLAB = slab_bytes(XG), G_AT = 4096, X_AT = G_AT + (G_BF16 ? 2048 : 4096);
            const int nbuf = g.epi_bufs;
            unsigned char* bufs = staging + (size_t)(warp - 2) * nbuf * SLAB;
            const int mrow = lane / 8, mch = lane % 8;      // fp32: 4 rows x 8 chunks per step
            const int hrow = lane / 4, hch = lane % 4;      // bf16: 8 rows x 4 chunks per step
            auto m_off = [](int r, int ch) { return r * 128 + ((ch ^ (r & 7)) << 4); };
            auto h_off = [](int r, int ch) { return r * 64 + ((ch ^ ((r >> 1) & 3)) << 4); };
            // the same for this lane's chunk of step `it` (rows 4 it + mrow and 8 it + hrow)
            const int m_off0 = m_off(mrow, mch), h_off0 = h_off(hrow, hch);
            auto m_step = [&](int it) { return (m_off0 ^ ((it & 1) << 6)) + it * 512; };
            auto h_step = [&](int it) { return h_off0 + it * 512; };
            // The slabs of this warp in order: (tile, 0), (tile, 1), (next tile, 0), ...  A warp has little time
            // per slab (14 KB, 8 warps: at the rate of the memory about 4800 cycles), and most of what it executed
            // was addresses: a tile is decoded once now, rows are reached by additions.  11008 x 4096 at
            // r = 32 / 256 0.123 / 0.132 -> 0.118 / 0.122 ms, six layers of 2048-wide matrices 0.840 / 0.866 -> 0.798 / 0.792.
            struct Slab { int t, slab, b, i0, j0; };
            auto advance = [&](Slab& s) {
                if (s.slab == 0) { s.slab = 1; s.j0 += 32; return; }
                for (s.t += tstride; s.t < g.total_tiles; s.t += tstride) {
                    const TileCoord c = decode_tile<EPI>(batch, g, s.t, scache, crank);
                    if (!c.active) continue;
                    s.slab = 0; s.b = c.b; s.i0 = c.mt * BM + quarter * 32; s.j0 = c.n0 + half * 64;
                    return;
                }
            };
            const int64_t ld = g.ld;
            // rows of the slab from this lane's first one on, if its columns are inside
            auto m_left = [&](const Slab& s) { return s.j0 + mch * 4 < g.Ncols ? g.Mrows - s.i0 - mrow : 0; };
            auto h_left = [&](const Slab& s) { return s.j0 + hch * 8 < g.Ncols ? g.Mrows - s.i0 - hrow : 0; };
            auto issue = [&](const Slab& s, unsigned char* buf) {
                const MatWork& w = batch.w[s.b];
                const uint32_t sb = smem_u32(buf);
                const int64_t midx = (s.i0 + mrow) * ld + s.j0 + mch * 4, hidx = (s.i0 + hrow) * ld + s.j0 + hch * 8;
                const int mleft = m_left(s), hleft = h_left(s);
                auto copy32 = [&](int at, const void* base) {
                    const float* p = reinterpret_cast<const float*>(base) + midx;
#pragma unroll
                    for (int it = 0; it < 8; ++it)
                        if (it * 4 < mleft) cp_async16(sb + at + m_step(it), p + it * 4 * ld);
                };
                auto copy16 = [&](int at, const void* base) {
                    const __nv_bfloat16* p = reinterpret_cast<const __nv_bfloat16*>(base) + hidx;
#pragma unroll
                    for (int it = 0; it < 4; ++it)
                        if (it * 8 < hleft) cp_async16(sb + at + h_step(it), p + it * 8 * ld);
                };
                copy32(0, w.M);
                if constexpr (G_BF16) copy16(G_AT, w.G); else copy32(G_AT, w.G);
                if constexpr (X_BF16) copy16(X_AT, w.X); else copy32(X_AT, w.X);
                cp_async_commit();
            };
            auto process = [&](const Slab& s, unsigned char* buf) -> bool {
                const MatWork& w = batch.w[s.b];
                const int slab = s.slab;
                const float efb = g.fp16 ? g.ef_b * *reinterpret_cast<const float*>(w.scratch + g.rscale_off) : g.ef_b;
                if (slab == 0) {
                    if (!mbar_wait(tfull0 + 8 * acc, acc_phase, abort_flag)) return false;
                    tc_fence_after();
                }
                const uint32_t taddr = tmem_base + acc * acc_stride + ((uint32_t)(quarter * 32) << 16) +
                                       (uint32_t)(half * 64 + slab * 32);
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    uint32_t va[16], vc[16];
                    tmem_ld16(taddr + hh * 16, va);
                    tmem_ld16(taddr + g.BN + hh * 16, vc);
                    tmem_ld_wait();
                    // eight columns of this lane's row, from the slab at `at`
                    auto read8 = [&](auto bf16, int at, int k, float (&f)[8]) {
                        if constexpr (decltype(bf16)::value) {
                            const uint4 u = *reinterpret_cast<const uint4*>(buf + at + h_off(lane, hh * 2 + k));
                            const uint32_t p[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                            for (int i = 0; i < 4; ++i) { f[2 * i] = bf16lo_to_f32(p[i]); f[2 * i + 1] = bf16hi_to_f32(p[i]); }
                        } else {
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                const float4 u = *reinterpret_cast<const float4*>(buf + at + m_off(lane, hh * 4 + 2 * k + i));
                                f[4 * i] = u.x; f[4 * i + 1] = u.y; f[4 * i + 2] = u.z; f[4 * i + 3] = u.w;
                            }
                        }
                    };
                    auto write8 = [&](int at, int k, const float (&f)[8]) {
#pragma unroll
                        for (int i = 0; i < 2; ++i)
                            *reinterpret_cast<float4*>(buf + at + m_off(lane, hh * 4 + 2 * k + i)) =
                                make_float4(f[4 * i], f[4 * i + 1], f[4 * i + 2], f[4 * i + 3]);
                    };
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        float mv[8], gv[8], xv[8];
                        read8(BoolConst<false>(), 0, k, mv);
                        read8(BoolConst<G_BF16>(), G_AT, k, gv);
                        read8(BoolConst<X_BF16>(), X_AT, k, xv);
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const float bval = mv[e] + gv[e];
                            mv[e] = g.ef_a * bval - efb * __uint_as_float(va[8 * k + e]);
                            xv[e] = g.wc * xv[e] - g.wd * __uint_as_float(vc[8 * k + e]);
                        }
                        write8(0, k, mv);
                        if constexpr (X_BF16)
                            *reinterpret_cast<uint4*>(buf + X_AT + h_off(lane, hh * 2 + k)) =
                                make_uint4(pack_bf16x2(xv[0], xv[1]), pack_bf16x2(xv[2], xv[3]), pack_bf16x2(xv[4], xv[5]), pack_bf16x2(xv[6], xv[7]));
                        else
                            write8(X_AT, k, xv);
                    }
                }
                if (slab == 1) {
                    // the accumulators of this tile are in registers / shared memory now
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) { if (PAIR) mbar_arrive_remote(tempty_ld + 8 * acc); else mbar_arrive(tempty0 + 8 * acc); }
                    if (++acc == g.acc_bufs) { acc = 0; acc_phase ^= 1; }
                }
                __syncwarp();
                const int64_t midx = (s.i0 + mrow) * ld + s.j0 + mch * 4, hidx = (s.i0 + hrow) * ld + s.j0 + hch * 8;
                const int mleft = m_left(s), hleft = h_left(s);
                auto store32 = [&](float* p, int at) {
#pragma unroll
                    for (int it = 0; it < 8; ++it)
                        if (it * 4 < mleft)
                            *reinterpret_cast<float4*>(p + it * 4 * ld) = *reinterpret_cast<const float4*>(buf + at + m_step(it));
                };
                store32(w.M + midx, 0);
                if constexpr (X_BF16) {
                    __nv_bfloat16* Xp = reinterpret_cast<__nv_bfloat16*>(w.X) + hidx;
#pragma unroll
                    for (int it = 0; it < 4; ++it)
                        if (it * 8 < hleft)
                            *reinterpret_cast<uint4*>(Xp + it * 8 * ld) = *reinterpret_cast<const uint4*>(buf + X_AT + h_step(it));
                } else {
                    store32(reinterpret_cast<float*>(w.X) + midx, X_AT);
                }
                __syncwarp();
                return true;
            };
            Slab cur{tile0 - tstride, 1, 0, 0, 0};
            int ib = 0;
            advance(cur);
            if (cur.t < g.total_tiles) issue(cur, bufs);
            while (cur.t < g.total_tiles) {
                Slab nxt = cur;
                advance(nxt);
                if (nbuf == 2) {
                    if (nxt.t < g.total_tiles) issue(nxt, bufs + (ib ^ 1) * SLAB);
                    else cp_async_commit();
                    cp_async_wait<1>();
                } else {
                    cp_async_wait<0>();
                }
                __syncwarp();
                if (!process(cur, bufs + ib * SLAB)) break;
                if (nbuf == 2) ib ^= 1;
                else if (nxt.t < g.total_tiles) issue(nxt, bufs);
                cur = nxt;
            }
            cp_async_wait<0>();
        }
    } else if (A_BUF) {
        // ---------------- transform warps: A tile of B = M + G (Alg. 1, buffer step) ----------------
        // 512 threads, two 8-element chunks each per 128 x 64 tile; four chunks (two tiles) are in flight
        // while a thread splits and stores, three of them (as many bytes) with fp32 gradients.  They are 48 of the
        // 80 registers that 22 warps leave a thread, and a load whose register is spilled is waited for at
        // once: what else lives in the loop is two pointers and one offset, and only one chunk is split
        // at a time.  Before, with indexes per chunk, two tiles of either type and both chunks split
        // together, 88 bytes were spilled with bf16 gradients and 292 with fp32; 0 to 24 are now, over all roles.  With the issuer above, one 11008 x 4096
        // matrix, first and second product: r = 32 0.111 -> 0.092 and 0.100 -> 0.063 ms, r = 128 0.134 -> 0.106 and
        // 0.126 -> 0.088; fp32 gradients, r = 32 0.184 -> 0.097 and 0.102 -> 0.068; six layers of 2048-wide matrices,
        // r = 512 0.979 -> 0.869 and 1.145 -> 1.047.
        const int xt = threadIdx.x - 32 * (2 + NE);     // 0 .. 511
        int as = 0; uint32_t aph = 0;
        bool ok = true;
        struct Raw { float4 m[2]; uint32_t gq[G_BF16 ? 4 : 8]; };
        constexpr int NR = G_BF16 ? 4 : 3;        // chunks in flight: 48 registers either way
        constexpr int ROUND = G_BF16 ? 2 : 3;     // tiles after which the chunks are back in the same registers
        // chunk e of a thread.  A_BUF_ROW: operand row = B row, depth = B column: row xt / 8 + 64 e,
        // columns k0 + 8 (xt % 8) .. + 7.  A_BUF_COL: operand row = B column, depth = B row (MN-major tile):
        // row k0 + xt / 16 + 32 e, columns 8 (xt % 16) .. + 7.
        constexpr int E_STEP = AMODE == A_BUF_ROW ? 64 : 32;      // rows of B between a thread's two chunks
        const int xr = AMODE == A_BUF_ROW ? xt / 8 : xt / 16, xc = AMODE == A_BUF_ROW ? xt % 8 : xt % 16;
        const uint32_t dst_off = AMODE == A_BUF_ROW ? xr * 128 + img_chunk_offset(xr, xc)
                                                    : (xc / 8) * 8192 + xr * 128 + img_chunk_offset(xr, xc % 8);
        // Where launches overlap, the first tiles of M and G are on their way to L2 while the kernel before is still at work (prefetches
        // may be early, loads may not: see launch.cuh).  Not elsewhere: the loads that follow at once then queue behind the prefetches
        // (six-kernel steps of 24 matrices 1024 wide at r = 32 238 us with, 235 without, 36 matrices 768 wide at r = 16 189.6 and 188.2).
        // (Prefetches, because registers that are loaded here live on into the
        // loop: 20 to 60 more bytes spilled, 1 % of the large steps.)
        if (tile0 < g.total_tiles) {
            const TileCoord c = decode_tile<EPI>(batch, g, tile0, scache, crank, false);
            const MatWork& w = batch.w[c.b];
            for (int kb = c.kb_begin; kb < min(c.kb_end, c.kb_begin + g.ahead); ++kb)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int64_t row = AMODE == A_BUF_ROW ? (int64_t)c.mt * BM + xr + e * E_STEP : (int64_t)kb * BK + xr + e * E_STEP;
                    const int64_t col = AMODE == A_BUF_ROW ? (int64_t)kb * BK + xc * 8 : (int64_t)c.mt * BM + xc * 8;
                    if (row < (AMODE == A_BUF_ROW ? g.Mrows : g.Kdim) && col < (AMODE == A_BUF_ROW ? g.Kdim : g.Mrows)) {
                        const int64_t idx = row * g.ld + col;
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(w.M + idx));
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const unsigned char*>(w.G) + idx * (G_BF16 ? 2 : 4)));
                    }
                }
        }
        grid_dependency_wait();
        for (int t = tile0; t < g.total_tiles && ok; t = next(t)) {
            const TileCoord c = decode_tile<EPI>(batch, g, t, scache, crank);
            if (!c.active) continue;
            const MatWork& w = batch.w[c.b];
            const int64_t base = AMODE == A_BUF_ROW ? ((int64_t)c.mt * BM + xr) * g.ld + xc * 8
                                                    : (int64_t)xr * g.ld + (int64_t)c.mt * BM + xc * 8;
            const float* Mp = w.M + base;
            const unsigned char* Gp = reinterpret_cast<const unsigned char*>(w.G) + base * (G_BF16 ? 2 : 4);
            // rows left from this thread's first one on (columns of B in the other operand: a multiple of 8, all or none)
            const int rleft = AMODE == A_BUF_ROW ? g.Mrows - c.mt * BM - xr : (c.mt * BM + xc * 8 < g.Mrows ? g.Kdim - xr : 0);
            const int kend = c.kb_end;
            auto fetch = [&](Raw& r, int kb, int e) {
                const bool in = AMODE == A_BUF_ROW ? (e * E_STEP < rleft && kb * BK + xc * 8 < g.Kdim)
                                                   : kb * BK + e * E_STEP < rleft;
                if (in) {
                    const int64_t idx = AMODE == A_BUF_ROW ? (int64_t)(e * E_STEP) * g.ld + kb * BK
                                                           : (int64_t)(kb * BK + e * E_STEP) * g.ld;
                    const float4* mp = reinterpret_cast<const float4*>(Mp + idx);
                    r.m[0] = mp[0]; r.m[1] = mp[1];
                    const uint4* gp = reinterpret_cast<const uint4*>(Gp + idx * (G_BF16 ? 2 : 4));
#pragma unroll
                    for (int i = 0; i < (G_BF16 ? 1 : 2); ++i) {
                        const uint4 u = gp[i];
                        r.gq[4 * i] = u.x; r.gq[4 * i + 1] = u.y; r.gq[4 * i + 2] = u.z; r.gq[4 * i + 3] = u.w;
                    }
                } else {
                    r.m[0] = r.m[1] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int i = 0; i < (G_BF16 ? 4 : 8); ++i) r.gq[i] = 0u;
                }
            };
            // split a chunk into the two bf16 terms and store them
            auto split_store = [&](const Raw& r, unsigned char* dst) {
                float gv[8];
                if constexpr (G_BF16) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) { gv[2 * i] = bf16lo_to_f32(r.gq[i]); gv[2 * i + 1] = bf16hi_to_f32(r.gq[i]); }
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) gv[i] = __uint_as_float(r.gq[i]);
                }
                const float v[8] = {r.m[0].x + gv[0], r.m[0].y + gv[1], r.m[0].z + gv[2], r.m[0].w + gv[3],
                                    r.m[1].x + gv[4], r.m[1].y + gv[5], r.m[1].z + gv[6], r.m[1].w + gv[7]};
                uint4 t0, t1;
                split8(v, t0, t1);
                *reinterpret_cast<uint4*>(dst) = t0;
                *reinterpret_cast<uint4*>(dst + A_TERM_BYTES) = t1;
            };
            Raw r[NR];               // chunk i of the tile sequence (two per tile) is in r[i % NR]
            // tile kb, the u-th of a round: wait for the slot, turn both chunks into terms, signal the MMA issuer
            auto tile = [&](int u, int kb) -> bool {
                if (!mbar_wait(a_empty0 + 8 * as, aph ^ 1, abort_flag)) return false;
                unsigned char* dst = a_ring + as * g.a_slot_bytes + dst_off;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    split_store(r[(2 * u + e) % NR], dst + e * E_STEP * 128);
                    if (kb + (e + NR) / 2 < kend) fetch(r[(2 * u + e) % NR], kb + (e + NR) / 2, (e + NR) % 2);
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) { if (PAIR) mbar_arrive_remote(a_full_ld + 8 * as); else mbar_arrive(a_full0 + 8 * as); }
                if (++as == g.a_slots) { as = 0; aph ^= 1; }
                return true;
            };
#pragma unroll
            for (int i = 0; i < NR; ++i)
                if (c.kb_begin + i / 2 < kend) fetch(r[i], c.kb_begin + i / 2, i % 2);
            for (int kb = c.kb_begin; kb < kend && ok; kb += ROUND) {
#pragma unroll
                for (int u = 0; u < ROUND; ++u)
                    if (ok && kb + u < kend) ok = tile(u, kb + u);
            }
        }
    }

    // ---------------- teardown ----------------
    // A role that gave up on a bounded wait leaves bulk copies into this CTA's shared memory and
    // issued MMAs possibly still in flight.  Nothing more is issued once the flag is up, so a fixed
    // pause far longer than any copy or MMA takes (about a millisecond) lets them land before the
    // shared memory and the tensor memory are given back.
    if (*abort_flag) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) {}
    }
    tc_fence_before();
    __syncthreads();
    // pairs: neither CTA leaves (or frees tensor memory) while the other may still reach its barriers
    if (PAIR) cluster_sync_all();
    tc_fence_after();
    if (*abort_flag && threadIdx.x == 0) {
        for (int b = 0; b < batch.count; ++b) atomicOr(batch.w[b].status, ST_WAIT);
    }
    if (warp == 1) {
        if (PAIR) tmem_dealloc_pair(tmem_base, (uint32_t)g.tmem_cols);
        else tmem_dealloc(tmem_base, (uint32_t)g.tmem_cols);
    }
}

}  // namespace tc

// ------------------------------------------------------------------------------------------
// Host side of the engine
// ------------------------------------------------------------------------------------------
struct TensorScratch {      // where the images of one matrix live inside its scratch area
    ImgRef linv;            // (L^{-1})^T of the current Cholesky        (r x r)
    ImgRef qprev;           // Q_prev                                    (n x r)
    ImgRef w0, w1;          // Y = B Q_prev and the QR intermediates     (max(m,n) x r)
    ImgRef p, r, q;         // P (m x r), R (n x r), Q (n x r); three planes when the fused pass runs in fp16
    int64_t colsq;          // fp32 [4 * ceil(max(m,n)/128)][r] column-square partials
    int64_t cnorm;          // fp32 [r] squared column norms of R
    int64_t rscale;         // fp32 inverse of the scale of R's fp16 plane
    int64_t fdiag, fstat, fscale;   // factor kernel: fp32 [r] Gram diagonal, statistics of the diagonal blocks,
                            // fp32 [r + 1] correction of the rounded diagonal of L^{-1}
    // partial results in memory (1: none) of Y = B Q_prev, of R = B^T P and of the Gram products over m and n rows
    int32_t y_parts, r_parts, gram_parts_m, gram_parts_n;
};

inline bool tensor_engine_supports(int64_t m, int64_t n, int32_t r) {
    return r % 16 == 0 && n % 8 == 0 && m >= 1;
}

inline ImgRef make_img(int64_t off, int64_t rows, int64_t cols, int planes = 2) {
    ImgRef im;
    im.off = off;
    im.rows_pad = (int32_t)((rows + 127) / 128 * 128);
    im.panels = (int32_t)((cols + 63) / 64);
    im.planes = planes;
    im.pad = 0;
    return im;
}
inline int64_t img_bytes(int64_t rows, int64_t cols, int planes = 2) {
    return planes * ((cols + 63) / 64) * ((rows + 127) / 128 * 128) * 128;
}
inline ImgRef no_img() { ImgRef im; im.off = -1; im.rows_pad = 0; im.panels = 0; im.planes = 0; im.pad = 0; return im; }

// The offsets of linv, cnorm, rscale, fdiag, fstat, fscale and colsq depend on r only (everything whose size depends on
// the matrix shape comes after them), so that one Cholesky launch can serve matrices of
// different shapes.  The image of L that the factor kernel works on lies where the image of Q does, which is written after the
// last factorisation (and is as tall: n >= r).
// half_planes: P, R, Q carry the fp16 plane (fused pass in fp16).
inline size_t tensor_scratch_layout(int64_t m, int64_t n, int32_t r, bool half_planes, size_t off, TensorScratch* ts) {
    const int64_t kmax = std::max(m, n);
    off = (off + 1023) / 1024 * 1024;
    auto take = [&](int64_t bytes) { int64_t o = (int64_t)off; off += (size_t)((bytes + 1023) / 1024 * 1024); return o; };
    ts->linv = make_img(take(img_bytes(r, r)), r, r);
    ts->cnorm = take(3 * (int64_t)r * 4 + 32 + CT_STAT_FLOATS * 4);       // (r is a multiple of 16)
    ts->fdiag = ts->cnorm + (int64_t)r * 4;
    ts->fscale = ts->fdiag + (int64_t)r * 4;
    ts->rscale = ts->fscale + (int64_t)r * 4 + 16;
    ts->fstat = ts->rscale + 16;
    ts->colsq = take(4 * ((kmax + 127) / 128) * (int64_t)r * 4);
    const int pl = half_planes ? 3 : 2;
    ts->w0 = make_img(take(img_bytes(kmax, r)), kmax, r);
    ts->w1 = make_img(take(img_bytes(kmax, r)), kmax, r);
    // the image of Q_prev is read by the first product of a step only; w1 is first written after
    // it (first apply of the left QR, same stream): they share their bytes
    ts->qprev = make_img(ts->w1.off, n, r);
    ts->p = make_img(take(img_bytes(m, r, pl)), m, r, pl);
    ts->r = make_img(take(img_bytes(n, r, pl)), n, r, pl);
    ts->q = make_img(take(img_bytes(n, r, pl)), n, r, pl);
    return off;
}
// the work images are sized for max(m, n) rows; a product over `rows` rows sees this view
inline ImgRef img_view(const ImgRef& im, int64_t rows) {
    ImgRef v = im;
    v.rows_pad = (int32_t)((rows + 127) / 128 * 128);
    return v;
}

// cuTensorMapEncodeTiled, fetched through the runtime so that the library does not link libcuda.
typedef CUresult (*TensorMapEncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                      const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                      CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline TensorMapEncodeFn tensor_map_encoder() {
    static TensorMapEncodeFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<TensorMapEncodeFn>(p);
    }
    return fn;
}
// 5-d map over the images `img` of all matrices of a batch: (64 bf16, rows, panels, terms, matrix),
// with the box (64, box_rows, box_panels, box_terms, 1).  The images are stored pre-swizzled, so
// the copy itself does not swizzle; out-of-range parts of a box read as zeros.
inline void encode_img_map(CUtensorMap* map, const Batch& b, const ImgRef& img, int box_rows, int box_panels,
                           int box_terms) {
    TensorMapEncodeFn enc = tensor_map_encoder();
    if (!enc) { engine_error() = 1; return; }
    const cuuint64_t term_bytes = (cuuint64_t)img.panels * img.rows_pad * 128;
    cuuint64_t dims[5] = {64, (cuuint64_t)img.rows_pad, (cuuint64_t)img.panels, (cuuint64_t)img.planes,
                          (cuuint64_t)b.count};
    cuuint64_t strides[4] = {128, (cuuint64_t)img.rows_pad * 128, term_bytes,
                             b.count > 1 ? (cuuint64_t)b.scratch_stride : img.planes * term_bytes};
    cuuint32_t box[5] = {64, (cuuint32_t)box_rows, (cuuint32_t)box_panels, (cuuint32_t)box_terms, 1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    void* base = b.w[0].scratch + img.off;
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, base, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        std::fprintf(stderr, "orthdion: cuTensorMapEncodeTiled failed (%d)\n", (int)r);
        engine_error() = 2;
    }
}

// Multiprocessor count of the current device (looked up once per device ordinal).
constexpr int kMaxDevices = 64;
inline int sm_count() {
    static std::atomic<int> cached[kMaxDevices] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= kMaxDevices) dev = 0;
    int n = cached[dev].load(std::memory_order_relaxed);
    if (n <= 0) {
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 148;
        cached[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

// Which instantiations exist as CTA-pair kernels: every product with an MN-major N-side (the two
// products with B, Gram, apply) and the fused pass on bf16 G and X in its single-term form, where
// the leader loads the R pieces and the peer the Q pieces (operand bytes per element 24 -> 16).
constexpr bool pair_capable(int nmode, int epi, int xg) {
    return nmode == tc::N_IMG_MN || (epi == tc::EPI_K5 && xg == 3);
}

template <class BATCH, int AMODE, int NMODE, int EPI, int XG>
inline cudaError_t set_gemm_attr() {
    constexpr bool GRAM = AMODE == tc::A_IMG_MN;
    cudaError_t e = cudaFuncSetAttribute(tc::gemm_kernel<BATCH, AMODE, NMODE, EPI, XG, false, GRAM>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, tc::SMEM_LIMIT);
    if constexpr (pair_capable(NMODE, EPI, XG)) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(tc::gemm_kernel<BATCH, AMODE, NMODE, EPI, XG, true, GRAM>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, tc::SMEM_LIMIT);
    }
    if constexpr (tc::a_is_buf(AMODE)) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(tc::gemm_kernel<BATCH, AMODE, NMODE, EPI, XG, false, true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, tc::SMEM_LIMIT);
    }
    return e;
}

inline cudaError_t tensor_engine_set_attributes() {
    cudaError_t e;
#define OD_SET(...) \
    if ((e = set_gemm_attr<SmallBatch, __VA_ARGS__>()) != cudaSuccess || (e = set_gemm_attr<Batch, __VA_ARGS__>()) != cudaSuccess) return e;
    OD_SET(tc::A_BUF_ROW, tc::N_IMG_MN, tc::EPI_STORE, 0)
    OD_SET(tc::A_BUF_ROW, tc::N_IMG_MN, tc::EPI_STORE, 1)
    OD_SET(tc::A_BUF_COL, tc::N_IMG_MN, tc::EPI_STORE, 0)
    OD_SET(tc::A_BUF_COL, tc::N_IMG_MN, tc::EPI_STORE, 1)
    OD_SET(tc::A_IMG_MN, tc::N_IMG_MN, tc::EPI_STORE, 0)
    OD_SET(tc::A_IMG_K, tc::N_IMG_MN, tc::EPI_STORE, 0)
    OD_SET(tc::A_IMG_K, tc::N_IMG_K, tc::EPI_K5, 0)
    OD_SET(tc::A_IMG_K, tc::N_IMG_K, tc::EPI_K5, 1)
    OD_SET(tc::A_IMG_K, tc::N_IMG_K, tc::EPI_K5, 2)
    OD_SET(tc::A_IMG_K, tc::N_IMG_K, tc::EPI_K5, 3)
#undef OD_SET
    return cudaSuccess;
}

// half: R's fp16 plane; normalise: image planes of Q = R / column norms (0: Q comes from elsewhere)
inline void launch_pack_right(const Batch& b, int64_t rows, int64_t cols, const TensorScratch& ts, bool half, int normalise, cudaStream_t st) {
    tc::PackRightArgs a{};
    a.rows = (int32_t)rows; a.cols = (int32_t)cols; a.r_img = ts.r; a.q_img = ts.q; a.r_half = half ? 1 : 0; a.normalise = normalise;
    a.cnorm_off = ts.cnorm; a.rscale_off = ts.rscale;
    dim3 grid((unsigned)ts.r.panels, (unsigned)(ts.r.rows_pad / 128), (unsigned)b.count);
    with_table(b, [&](const auto& t) {
        launch(tc::pack_right_kernel<table_t<decltype(t)>>, grid, 256, 0, 1, normalise ? prof::S_COLNORM : prof::S_PACK, st, t, a);
    });
}
// the column squares of `rows` rows, added up
inline void launch_colsum(const Batch& b, const TensorScratch& ts, int64_t rows, int r, Sel dst, int64_t stride, int stage, cudaStream_t st) {
    with_table(b, [&](const auto& t) {
        launch(colsum_kernel<table_t<decltype(t)>>, dim3((unsigned)((r + 63) / 64), 1, (unsigned)b.count), 256, 0, 1, stage, st, t, ts.colsq,
               (int)(4 * ((rows + 127) / 128)), r, dst, stride);
    });
}

inline void launch_pack(const Batch& b, Sel src, int64_t rows, int64_t cols, ImgRef dst, cudaStream_t st, bool init = false) {
    tc::PackArgs a{};
    a.init = init ? 1 : 0;
    a.src = src; a.rows = (int32_t)rows; a.cols = (int32_t)cols; a.dst = dst;
    dim3 grid((unsigned)dst.panels, (unsigned)(dst.rows_pad / 128), (unsigned)b.count);
    with_table(b, [&](const auto& t) { launch(tc::pack_kernel<table_t<decltype(t)>>, grid, 256, 0, 1, prof::S_PACK, st, t, a); });
}

// Fills in the tiling, ring and tensor-memory fields and launches.
template <int AMODE, int NMODE, int EPI, int XG>
inline void launch_gemm(const Batch& b, tc::GemmArgs g, int stage, cudaStream_t st) {
    if (g.fp16) { g.passes = 1; g.passes2 = 1; }
    // CTA pairs need full 256-column instructions: every tile 256 or 512 columns wide (MN-major
    // N-side), or the fused pass in its single-term form with full 128-column tiles.
    bool pair = false;
    if constexpr (pair_capable(NMODE, EPI, XG)) {
        if (NMODE == tc::N_IMG_MN) pair = g.BN % 256 == 0 && g.Ncols % g.BN == 0;
        else pair = g.passes == 1 && g.passes2 == 1 && g.BN == 128 && g.Ncols % 128 == 0;
        if (sm_count() < 2) pair = false;
    }
    g.pair = pair ? 1 : 0;
    g.m_tiles = (g.Mrows + tc::BM - 1) / tc::BM;
    if (pair) g.m_tiles = (g.m_tiles + 1) / 2;      // scheduled row tiles of 256 rows
    g.n_tiles = (g.Ncols + g.BN - 1) / g.BN;
    g.k_blocks = (g.Kdim + tc::BK - 1) / tc::BK;
    if (g.chunks < 1) g.chunks = 1;
    if (g.acc_chunks < 1) g.acc_chunks = 1;
    g.kb_per_chunk = (g.k_blocks + g.chunks - 1) / g.chunks;
    g.kb_per_tile = g.acc_chunks * g.kb_per_chunk;
    g.ksplit = (g.chunks + g.acc_chunks - 1) / g.acc_chunks;
    g.run = g.run ? g.ksplit : 1;
    g.total_tiles = b.count * g.m_tiles * g.n_tiles * g.ksplit;
    g.ahead = overlap_launches() ? 4 : 0;
    g.one_operand = AMODE == tc::A_IMG_MN && g.BN <= (pair ? 256 : 128);
    const int n1_terms = g.passes == 3 ? 2 : 1, n2_terms = g.passes2 == 3 ? 2 : 1;
    const int bn64 = (g.BN + 63) / 64 * 64;
    const int a_terms = (tc::a_is_buf(AMODE) || g.passes == 3 || (EPI == tc::EPI_K5 && g.passes2 == 3)) ? 2 : 1;
    g.a_slot_bytes = a_terms * tc::A_TERM_BYTES;
    g.a_slots = tc::A_RING_BYTES / g.a_slot_bytes;
    // image-to-image products: a third two-term slot (the N ring then holds three pieces as well)
    if (EPI == tc::EPI_STORE && !tc::a_is_buf(AMODE)) g.a_slots = std::min(tc::MAX_A_SLOTS, 6 * tc::A_TERM_BYTES / g.a_slot_bytes);
    g.epi_bufs = 1;
    if (EPI == tc::EPI_K5) {
        // the fused pass: 64 KB of A slots (four single-term ones or two two-term ones) and one
        // epilogue buffer per warp.  bf16 G and X in single terms: a second buffer, paid for with an A slot and N
        // slots; the update is bound by bytes in flight until the products take as long.  Pairs, which keep
        // three of six N slots, below rank 512: 11008 x 4096, one buffer -> two, before the leaner update: r = 32 0.141 ->
        // 0.124 ms, 256 0.149 -> 0.131, 448 0.152 -> 0.148, 512 0.154 -> 0.160.  Single CTAs (widths that are no multiple
        // of 128), which keep one of three (twice as large), up to rank 192: eight 4104 x 4104 r = 16 0.394 -> 0.378, 192
        // 0.402 -> 0.402, 208 0.401 -> 0.456, 400 0.433 -> 0.643; 24 of 2712 x 1000 r = 192 0.210 -> 0.199, 256 0.213 ->
        // 0.227, 400 0.227 -> 0.313.
        g.a_slots = (a_terms == 1) ? 4 : 2;
        if (XG == 3 && a_terms == 1 && g.k_blocks < (pair ? 8 : 4)) { g.a_slots = 3; g.epi_bufs = 2; }
    }
    if (NMODE == tc::N_IMG_MN) {
        if (pair) {
            // each CTA holds half of the columns: same bytes per piece at twice the depth
            g.ks = bn64 <= 256 ? 64 : 32;
            g.n_piece_bytes = n1_terms * (bn64 / 128) * g.ks * 128;
        } else {
            g.ks = bn64 <= 128 ? 64 : (bn64 <= 256 ? 32 : 16);
            g.n_piece_bytes = n1_terms * (bn64 / 64) * g.ks * 128;
        }
    } else {
        g.ks = 64;
        // The R and Q pieces of a depth block in one slot, or in slots of their own where not even two such slots fit (one:
        // nothing is under way while the products run).  bf16 X and G with three passes for M only, two slots of 48 KB ->
        // three of 32: 28 matrices 2048 wide at r = 256 1.93 -> 1.97 ms.
        g.n_piece_bytes = (n1_terms + n2_terms) * tc::A_TERM_BYTES;
        const int room = tc::SMEM_LIMIT - g.a_slots * g.a_slot_bytes - 8 * g.epi_bufs * tc::slab_bytes(XG) - 256 - 1024;
        g.n_split = n1_terms + n2_terms > 2 && room < 2 * g.n_piece_bytes;
        if (g.n_split) g.n_piece_bytes = 2 * tc::A_TERM_BYTES;
        if (pair) g.n_piece_bytes = tc::A_TERM_BYTES;    // the R piece (leader) or the Q piece (peer)
    }
    const int accw = (EPI == tc::EPI_K5) ? 2 * g.BN : g.acc_chunks * g.BN;
    g.acc_bufs = (2 * accw <= 512) ? 2 : 1;
    int cols = 32;
    while (cols < g.acc_bufs * accw) cols *= 2;
    g.tmem_cols = cols;
    int max_n_slots = tc::MAX_N_SLOTS;
    if (tc::a_is_buf(AMODE)) {
        // The loads of M and G under way (96 KB a CTA) need room in the L1 cache, which is what shared memory leaves of
        // 256 KB: up to 196 KB of it are used, where 228 would leave 28 KB of cache.  Three slots in either
        // ring, two in the A ring where three do not fit.  First and second product, as many slots as fit -> this:
        // 11008 x 4096 r = 128 0.102 -> 0.092 and 0.088 -> 0.080 ms, r = 256 0.116 -> 0.105 and 0.099 -> 0.090; six layers of
        // 2048-wide matrices r = 128 0.532 -> 0.468 and 0.569 -> 0.496, r = 192 0.697 -> 0.617 and 0.695 -> 0.608.  (Two slots in the N
        // ring: r = 512 0.858 -> 0.917.)
        max_n_slots = 3;
        g.a_slots = 3;
        if (3 * (size_t)g.a_slot_bytes + 3 * (size_t)g.n_piece_bytes + 4 * tc::STORE_STAGING_BYTES + 2304 > 196 * 1024) g.a_slots = 2;
    }
    const size_t fixed = (size_t)g.a_slots * g.a_slot_bytes +
                         (size_t)tc::epi_warps(AMODE, EPI) * (EPI == tc::EPI_STORE ? tc::STORE_STAGING_BYTES : g.epi_bufs * tc::slab_bytes(XG)) +
                         256 + 1024;
    g.n_slots = (int)std::min<size_t>(max_n_slots, (tc::SMEM_LIMIT - fixed) / (size_t)g.n_piece_bytes);
    // more than half of an SM's shared memory: one CTA per SM, whatever its tensor-memory share
    const size_t smem = std::max<size_t>(fixed + (size_t)g.n_slots * g.n_piece_bytes, 120 * 1024);
    if (AMODE == tc::A_IMG_K) encode_img_map(&g.map_a, b, g.a, 128, 1, a_terms);
    else if (AMODE == tc::A_IMG_MN) encode_img_map(&g.map_a, b, g.a, 64, 2, a_terms);
    if (NMODE == tc::N_IMG_MN) encode_img_map(&g.map_n1, b, g.n1, g.ks, pair ? 2 : bn64 / 64, n1_terms);
    else encode_img_map(&g.map_n1, b, g.n1, 128, 1, n1_terms);
    if (EPI == tc::EPI_K5) encode_img_map(&g.map_n2, b, g.n2, 128, 1, n2_terms);
    if (engine_error()) return;
    constexpr bool GRAM = AMODE == tc::A_IMG_MN;
    constexpr int threads = tc::gemm_threads(AMODE, EPI);
    const dim3 grid((unsigned)(pair ? 2 * std::min(g.total_tiles / g.run, sm_count() / 2) : std::min(g.total_tiles / g.run, sm_count())));
    with_table(b, [&](const auto& t) {
        using BATCH = table_t<decltype(t)>;
        if constexpr (pair_capable(NMODE, EPI, XG)) {
            if (pair) {
                launch(tc::gemm_kernel<BATCH, AMODE, NMODE, EPI, XG, true, GRAM>, grid, threads, smem, 2, stage, st, t, g);
                return;
            }
        }
        if constexpr (tc::a_is_buf(AMODE)) {
            if (g.run > 1) {
                launch(tc::gemm_kernel<BATCH, AMODE, NMODE, EPI, XG, false, true>, grid, threads, smem, 1, stage, st, t, g);
                return;
            }
        }
        launch(tc::gemm_kernel<BATCH, AMODE, NMODE, EPI, XG, false, GRAM>, grid, threads, smem, 1, stage, st, t, g);
    });
}

inline tc::Dest dest_none() {
    tc::Dest d{};
    d.f32 = Sel{W_P, 0, 0}; d.img = no_img(); d.has_f32 = 0; d.colsq = 0;
    return d;
}

// Multiprocessors that the rules below count on: a constant, so that workspace sizes need no device.
constexpr int SPLIT_SMS = 148;

// Depth blocks that a launch takes one after the other when `tiles` row tiles run in `chunks` parts each: waves
// times blocks per part, with two more for filling and emptying a part's pipeline.
inline int64_t product_depth(int64_t tiles, int chunks, int kb) {
    const int64_t waves = (tiles * chunks + SPLIT_SMS - 1) / SPLIT_SMS;
    return waves * ((kb + chunks - 1) / chunks + 2);
}
// Whether the one-kernel QR takes the result (nearly: its limit by shared memory needs the device) and adds the partial
// results up as it loads them.
inline bool summed_by_qr(int r, int64_t out_rows) { return r <= 32 || (r <= QS_MAX_RANK && out_rows <= QS_MAX_ROWS_64); }
// ... and what writing and adding up the partial results costs in the same unit (about a microsecond): a launch, but for
// the one-kernel QR.  (Their bytes have one price here, although one cluster of at most 16 multiprocessors loads what that
// kernel adds up, half of its 45 us at 11008 rows and r = 32.  Steps with this rule against the one without that kernel's term, 8192 to
// 24576 rows: 1.00 to 1.09 times as fast.)
inline int64_t partial_cost(int64_t tiles, int chunks, int r, bool by_qr) { return (by_qr ? 1 : 4) + tiles * chunks * r / 6000; }

// Depth split of the two products with the buffer.  With one matrix (or a few) in a call and a
// small rank, the output has too few row tiles for the device, or one wave and a bit (a 4096-wide factor 32, an
// 11008-wide one 86), and every one of them runs over the whole depth.  The depth is therefore cut into chunks whose
// results are added in a fixed order.  Their number depends on the plan only (rank, rows of the result,
// depth), so that a matrix gets the same bits alone and in any group; ranks above 256 have one.  Where
// it shortens a launch the chunks run as tiles of their own and leave
// fp32 partial results in memory; where it does not, up to rank 128, one tile runs through as many chunks as have
// an accumulator each in the 512 columns of tensor memory, the epilogue adds them up, and where they are not all (five
// to eight chunks above rank 64) the next tile of the same CTA adds the others to what the first one stored.
// The tensor core truncates when it adds into its accumulator, so a sum loses the more the longer its chunk: with 11 to 32
// depth blocks a chunk R = B^T P of a 16384 x 1024 matrix at r = 96 is off by 7e-6, with 64 by 1.3e-5.  Hence at least as
// many chunks, up to eight of at least eight blocks, as fit 74 pairs of tiles, at any rank.
// Up to r = 128 it may be more: the number that makes the launch of one matrix shortest by the two counts above.  Measured
// against the first rule alone: 11008 x 4096, first product, r = 32 0.090 -> 0.074 ms,
// r = 64 0.091 -> 0.086; 20480 x 4096 r = 32 0.170 -> 0.127, r = 128 0.198 -> 0.176.  Against four chunks at most above
// r = 64: one 16384 x 1024 matrix at r = 96 0.470 -> 0.426 ms a step, 2048 x 5632 r = 128 0.379 -> 0.368; in a group, where
// the tiles of a run follow one another, six layers of a 1.1B model at r = 128 1.127 -> 1.155.
// In front of the one-kernel QR a chunk may have two depth blocks.  Against four at least, r = 16: one 256 x 256 step
// 57.5 -> 52.9 us, 512 x 512 68.6 -> 58.8, 768 x 768 58.9 -> 57.5; r = 32 1024 x 1024 70 -> 68; two to eight up to 576 wide mostly 3 to 17 % faster.  What it costs:
// the count is the plan's, and four to eight equal matrices 640 to 1536 wide have tiles enough for the longer
// chunks: 8 x 768 r = 16 76 -> 79.5, 8 x 1024 r = 32 114 -> 125.  In models of 7 to 56 matrices of such widths it comes out even (0.92 to
// 1.05 times).
inline int buffer_chunks(int r, int64_t out_rows, int64_t depth) {
    if (r > 256) return 1;
    const int kb = (int)((depth + tc::BK - 1) / tc::BK), pairs = (int)((out_rows + 255) / 256);
    int want = pairs < 37 && kb >= 32 ? std::min({8, 74 / pairs, kb / 8}) : 1;
    if (r <= 128) {
        const int64_t tiles = (out_rows + tc::BM - 1) / tc::BM;
        int64_t best = product_depth(tiles, 1, kb);
        int fast = 1;
        const bool by_qr = summed_by_qr(r, out_rows);
        for (int v = 2; v <= std::min(r <= 64 ? 8 : 4, kb / (by_qr ? 2 : 4)); ++v) {
            const int64_t cost = product_depth(tiles, v, kb) + partial_cost(tiles, v, r, by_qr);
            if (cost < best) { best = cost; fast = v; }
        }
        want = std::max(want, fast);
    }
    if (want < 2) return 1;
    const int per = (kb + want - 1) / want;
    return (kb + per - 1) / per;             // every chunk non-empty
}
// Partial results in memory of a product in a call of `matrices`: the chunks, or 1 where they stay in tensor memory
// (up to rank 128 always, when the workspace is to be `lean`).
// Measured (before: always in memory, added up, packed and squared by three kernels): 154 matrices of a 1.1B model
// at r = 128 9.7 -> 8.6 ms a step; one 4096 x 4096 matrix at r = 256, three kernels in one, 0.633 -> 0.609 ms.
inline int buffer_ksplit(int r, int64_t out_rows, int64_t depth, int matrices, int lean) {
    const int chunks = buffer_chunks(r, out_rows, depth);
    if (r > 128 || chunks == 1) return chunks;
    if (lean) return 1;
    const int64_t tiles = matrices * ((out_rows + tc::BM - 1) / tc::BM);
    const int kb = (int)((depth + tc::BK - 1) / tc::BK);
    return product_depth(tiles, chunks, kb) + partial_cost(tiles, chunks, r, summed_by_qr(r, out_rows)) < product_depth(tiles, 1, kb) ? chunks : 1;
}

// The chunks of a product with B in `parts` tiles of their own, or in as few tiles as tensor memory allows.
inline void set_chunks(tc::GemmArgs& g, int r, int chunks, int parts) {
    g.chunks = chunks;
    if (parts > 1 || chunks == 1) return;
    const int fit = 512 / r, tiles = (chunks + fit - 1) / fit;
    g.acc_chunks = (chunks + tiles - 1) / tiles;
    g.run = tiles > 1 ? 1 : 0;
}

// Columns per tile of a product with B, out of r (count matrices in the launch).  A wide tile forms B's terms once
// for all columns; narrow ones form them again for every tile (from L2), which pays only where all of
// them run at once on multiprocessors that the wide ones leave idle.  The order in which an entry is summed does
// not depend on the tile.  Measured, one matrix, 512 -> 256 columns: 4096 x 3584 at r = 512 K1 0.161 -> 0.112, K3
// 0.194 -> 0.166 ms; 8192 x 8192 at r = 512 step 1.61 -> 1.44.  With several waves of tiles it loses: sixteen
// 4096 x 4096 matrices at r = 512, four waves of wide tiles against seven narrow ones, K3 of the step 5.65 -> 7.07 ms.
inline int buffer_bn(int r, int64_t out_rows, int count) {
    const int wide = std::min(r, 512);
    if (r <= 256) return wide;
    if (r % 256 == 0) {
        const int64_t tiles = (int64_t)count * ((out_rows + 255) / 256) * (r / 256);
        return tiles <= SPLIT_SMS / 2 ? 256 : wide;
    }
    return (int64_t)count * ((out_rows + tc::BM - 1) / tc::BM) * ((r + 127) / 128) <= SPLIT_SMS ? 128 : wide;
}

// After a product whose chunks ran as tiles of their own: dst (rows x r fp32) <- sum of the partial results
// in chunk order, its operand image and its column squares per 32-row block (added as the epilogue of
// the unsplit form adds them).  One CTA per (64 columns, 32 rows): 256 threads, eight columns each.
struct FinishArgs {
    Sel dst, part;
    int64_t rows;
    int32_t r, ksplit;
    ImgRef img;                 // its geometry decides the launch
    int64_t colsq_off;
    int32_t to_img;
};
template <class BATCH>
__global__ void __launch_bounds__(256)
finish_split_kernel(const __grid_constant__ BATCH batch, FinishArgs a) {
    grid_dependency();
    const MatWork& w = batch.w[blockIdx.z];
    if (*w.status & ST_FAILED) return;
    __shared__ float sq[32][65];
    const int rho = threadIdx.x / 8, c = threadIdx.x % 8;
    const int64_t row = (int64_t)blockIdx.y * 32 + rho;
    const int panel = blockIdx.x, col = panel * 64 + c * 8;
    float v[8] = {};
    if (row < a.rows && col < a.r) {
        const float* P = pick(w, a.part) + row * a.r + col;
        const int64_t stride = a.rows * a.r;
        tc::load8(P, 0, 0, v);
#pragma unroll 4
        for (int k = 1; k < a.ksplit; ++k) {
            float u[8];
            tc::load8(P + k * stride, 0, 0, u);
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] += u[i];
        }
        float4* D = reinterpret_cast<float4*>(pick(w, a.dst) + row * a.r + col);
        D[0] = make_float4(v[0], v[1], v[2], v[3]);
        D[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
    if (a.to_img) {
        uint4 t0, t1;
        split8(v, t0, t1);
        unsigned char* scr = reinterpret_cast<unsigned char*>(w.scratch);
        const int o = img_chunk_offset(rho, c);
        *reinterpret_cast<uint4*>(scr + img_row_offset(a.img, 0, panel, row) + o) = t0;
        *reinterpret_cast<uint4*>(scr + img_row_offset(a.img, 1, panel, row) + o) = t1;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) sq[rho][c * 8 + i] = __fmul_rn(v[i], v[i]);
    __syncthreads();
    if (threadIdx.x < 64 && panel * 64 + threadIdx.x < a.r) {
        float s[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) s[i] = sq[i][threadIdx.x];
#pragma unroll
        for (int h = 16; h >= 1; h >>= 1)
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (i < h) s[i] += s[i + h];
        reinterpret_cast<float*>(w.scratch + a.colsq_off)[(int64_t)blockIdx.y * a.r + panel * 64 + threadIdx.x] = s[0];
    }
}
inline void finish_split_product(const Batch& b, Sel dst, Sel part, int64_t rows, int r, int ksplit, ImgRef img, bool to_img,
                                 int64_t colsq_off, int stage, cudaStream_t st) {
    FinishArgs a{};
    a.dst = dst; a.part = part; a.rows = rows; a.r = r; a.ksplit = ksplit; a.img = img; a.colsq_off = colsq_off; a.to_img = to_img ? 1 : 0;
    with_table(b, [&](const auto& t) {
        launch(finish_split_kernel<table_t<decltype(t)>>, dim3((unsigned)img.panels, (unsigned)(img.rows_pad / 32), (unsigned)b.count), 256, 0, 1,
               stage, st, t, a);
    });
}

// Where a product with B goes.
enum ProductOut : int {
    OUT_IMAGE = 0,     // operand image and column squares (and the fp32 R slot)
    OUT_F32 = 1,       // fp32 slot, or partial results of a depth split, for the small-rank QR kernel
    OUT_SUM = 2,       // fp32 slot only: one shard of the columns, to be summed over the shards
    OUT_NORM = 3       // fp32 slot and column squares, for the column normalisation
};
// Y = (M + G) Q_prev  -> image w0 (+ column squares)              (Alg. 1, buffer and left-factor steps)
// First kernel of a step: its packing of Q_prev also clears the status words.
// part: scratch for the partial results of a depth split (ts.y_parts of them).
inline void tensor_k1(int64_t m, int64_t n, int r, int g_bf16, int passes, const Batch& b, const TensorScratch& ts,
                      Sel part, cudaStream_t st, ProductOut kind) {
    launch_pack(b, Sel{W_Q, 0, 0}, n, r, ts.qprev, st, true);
    const int ksplit = kind == OUT_SUM ? 1 : ts.y_parts;
    tc::GemmArgs g{};
    if (kind != OUT_SUM) set_chunks(g, r, buffer_chunks(r, m, n), ksplit);
    g.Mrows = (int32_t)m; g.Ncols = r; g.Kdim = (int32_t)n; g.BN = buffer_bn(r, m, b.count);
    g.passes = passes; g.passes2 = 1; g.ld = n; g.n1 = ts.qprev; g.a = no_img(); g.n2 = no_img();
    g.colsq_off = ts.colsq;
    g.out.normal = dest_none();
    if (ksplit > 1) { g.out.normal.f32 = part; g.out.normal.has_f32 = 1; g.split_stride = m * r; }
    else if (kind != OUT_IMAGE) { g.out.normal.f32 = Sel{W_P, 0, 0}; g.out.normal.has_f32 = 1; }
    else { g.out.normal.img = img_view(ts.w0, m); g.out.normal.colsq = 1; g.out.normal.has_f32 = g.run; }
    g.out.shifted = g.out.normal; g.out.ld = r;
    if (g_bf16) launch_gemm<tc::A_BUF_ROW, tc::N_IMG_MN, tc::EPI_STORE, 1>(b, g, prof::S_K1, st);
    else launch_gemm<tc::A_BUF_ROW, tc::N_IMG_MN, tc::EPI_STORE, 0>(b, g, prof::S_K1, st);
    // (a sum in parts goes through the fp32 P slot, which holds nothing yet at this point of a step)
    if (ksplit > 1 && kind == OUT_IMAGE)
        finish_split_product(b, Sel{W_P, 0, 0}, part, m, r, ksplit, img_view(ts.w0, m), true, ts.colsq, prof::S_K1, st);
}

// R = (M + G)^T P  -> fp32 R slot, image r (+ column squares)     (Alg. 1, right-factor step)
inline void tensor_k3(int64_t m, int64_t n, int r, int g_bf16, int passes, const Batch& b, const TensorScratch& ts,
                      Sel part, cudaStream_t st, ProductOut kind) {
    const int ksplit = ts.r_parts;
    tc::GemmArgs g{};
    set_chunks(g, r, buffer_chunks(r, n, m), ksplit);
    g.Mrows = (int32_t)n; g.Ncols = r; g.Kdim = (int32_t)m; g.BN = buffer_bn(r, n, b.count);
    g.passes = passes; g.passes2 = 1; g.ld = n; g.n1 = ts.p; g.a = no_img(); g.n2 = no_img();
    g.colsq_off = ts.colsq;
    g.out.normal = dest_none(); g.out.normal.has_f32 = 1;
    if (ksplit > 1) { g.out.normal.f32 = part; g.split_stride = n * r; }
    else {
        g.out.normal.f32 = Sel{W_R, 0, 0};
        if (kind == OUT_IMAGE) g.out.normal.img = ts.r;
        if (kind != OUT_F32) g.out.normal.colsq = 1;
    }
    g.out.shifted = g.out.normal; g.out.ld = r;
    if (g_bf16) launch_gemm<tc::A_BUF_COL, tc::N_IMG_MN, tc::EPI_STORE, 1>(b, g, prof::S_K3, st);
    else launch_gemm<tc::A_BUF_COL, tc::N_IMG_MN, tc::EPI_STORE, 0>(b, g, prof::S_K3, st);
    if (ksplit > 1 && kind != OUT_F32)
        finish_split_product(b, Sel{W_R, 0, 0}, part, n, r, ksplit, ts.r, kind == OUT_IMAGE, ts.colsq, prof::S_K3, st);
}

// Columns per tile of a product between images (`copies`: matrices times depth chunks).  256 columns, in CTA pairs
// where the rank allows, do the least work; 128 where all such tiles run at once on multiprocessors that the wide ones
// leave idle.  A Gram product's tiles above the diagonal count: they are skipped, but the tiles of a launch are dealt
// out in order, so a launch of more tiles than multiprocessors gives some of those two real ones.  (Counted without:
// ten 14336 x 1024 matrices at r = 512, Gram products of a step 0.658 -> 0.940 ms, twelve 2048 x 2048 0.245 -> 0.300; six
// 4096 x 4096 at r = 192 0.167 -> 0.188.)  An entry is summed in the same order either way.
// Measured, 256 -> 128 columns: one 4096 x 4096 matrix at r = 256, Gram products of a step 0.170 -> 0.152 ms, applies 0.110 ->
// 0.090; 4096 x 3584 at r = 512 0.238 -> 0.203 and 0.118 -> 0.095; 28 matrices 1000 wide at r = 272 0.911 -> 0.727 and
// 0.487 -> 0.469.  (64 columns: another 5 % at r = 256, but 0.304 -> 0.357 ms for the Gram products of 11008 x 4096 at r = 1024.)
inline int image_bn(int r, int64_t out_rows, int64_t copies) {
    const int wide = std::min(r, 256);
    if (wide <= 128) return wide;
    const int64_t rows = (out_rows + tc::BM - 1) / tc::BM, cols = (r + 127) / 128;
    return rows * cols * copies <= SPLIT_SMS ? 128 : wide;
}

// Depth split of the Gram product.  The Gram matrix is one output tile at small ranks and ten at r = 1024,
// each with a main loop over all rows of the tall matrix: the depth is cut into chunks whose results are
// added in a fixed order.  Their number depends on the rank and the row count only, so a matrix gets the same
// bits alone and in any group.  The chunks run as tiles of their own and leave partial matrices that a small
// kernel adds up; above r = 256, in calls with tiles enough for the device, and at any rank where a workspace has no room
// for the partial matrices, one CTA takes the chunks of a tile one after the other and adds each to the tile it has stored (the two accumulators alternate, so
// the additions run beside the next chunk's products).
inline int gram_tiles(int r) {               // tiles that touch the lower triangle
    const int rows = r % 256 ? 128 : 256, cols = std::min(r, 256);
    int n = 0;
    for (int i = 0; i * rows < r; ++i)
        for (int j = 0; j * cols < r; ++j)
            if (j * cols <= i * rows + rows - 1) ++n;
    return n;
}
inline int gram_chunks(int r, int64_t rows) {
    const int kb = (int)((rows + tc::BK - 1) / tc::BK);
    // At least 8 depth blocks per chunk at r <= 256, from 64 blocks on sixteen chunks (4096 x 4096, 8 chunks -> 16: r = 256 386 ->
    // 375 us a step, r = 192 359 -> 352; four blocks a chunk everywhere: 24 layers of 768-wide matrices at r = 192 2.04 -> 2.17 ms); 24 above, where the additions cost calls with many matrices
    // some of their Gram time (1.1B model at r = 512 3.03 -> 3.15 ms of an 18 ms step; with 16 blocks 3.31) and 16
    // would give single matrices another 0.05 ms.
    const int want = r <= 256 ? (kb >= 64 ? 16 : kb / 8) : std::min({16, kb / 24, 80 / gram_tiles(r)});
    if (want < 2) return 1;
    const int per = (kb + want - 1) / want;
    return (kb + per - 1) / per;             // every chunk non-empty
}
// Partial matrices in memory of a Gram product in a call of `matrices`.  Above r = 256 the line is where chunks as tiles of
// their own take fewer depth blocks one after the other than undivided tiles, with six more for starting and storing a
// chunk (tiles above the diagonal hold a place too, see image_bn); none in calls of more than two waves of tiles, where
// the partial matrices would be megabytes for each of many matrices, and none when the workspace is to be `lean`.
// Measured, the Gram products of a step, undivided and in chunks: one 11008 x 4096 matrix at r = 1024 0.64 and 0.35 ms,
// one 4096 x 3584 at r = 512 0.36 and 0.26; n x 1024 at r = 512: 4096, 8 matrices 0.276 and 0.213, 12 0.277 and 0.320, 20
// 0.453 and 0.416; 8192, 9 0.430 and 0.324, 12 0.422 and 0.416, 16 0.434 and 0.484, 20 0.745 and 0.588, 28 0.768 and
// 0.766; 14336, 12 0.636 and 0.554, 14 0.648 and 0.628, 16 0.660 and 0.689.  r = 384 (single CTAs): 4096, 12 0.295 and
// 0.215, 20 0.300 and 0.337, 28 0.501 and 0.451; 8192, 16 0.345 and 0.415; 14336, 16 0.526 and 0.510.
inline int gram_ksplit(int r, int64_t rows, int matrices, int lean) {
    if (r <= 256) return lean < 2 ? gram_chunks(r, rows) : 1;
    if (lean) return 1;
    const int room = r % 256 ? SPLIT_SMS : SPLIT_SMS / 2, high = r % 256 ? 128 : 256, wide = std::min(r, 256);
    const int64_t tiles = (int64_t)matrices * ((r + high - 1) / high) * ((r + wide - 1) / wide);
    const int chunks = gram_chunks(r, rows), kb = (int)((rows + tc::BK - 1) / tc::BK);
    auto waves = [&](int64_t t) { return (t + room - 1) / room; };
    return tiles <= 2 * room && waves(tiles * chunks) * ((kb + chunks - 1) / chunks + 6) < waves(tiles) * kb ? chunks : 1;
}

// dst <- sum of the `ksplit` partial results at `part` (4 * total4 floats each, one after the
// other), added in the order of the chunks
template <class BATCH>
__global__ void __launch_bounds__(256)
gram_reduce_kernel(const __grid_constant__ BATCH batch, Sel gram, Sel part, int64_t total4, int ksplit, int only_shift_bit) {
    grid_dependency();
    const MatWork& w = batch.w[blockIdx.z];
    const int st = *w.status;
    if ((st & ST_FAILED) || (only_shift_bit && !(st & only_shift_bit))) return;
    const int64_t q = (int64_t)blockIdx.x * 256 + threadIdx.x;      // float4 index
    if (q >= total4) return;
    const float4* P = reinterpret_cast<const float4*>(pick(w, part));
    float4 acc = P[q];
    for (int s2 = 1; s2 < ksplit; ++s2) {
        const float4 v = P[(int64_t)s2 * total4 + q];
        acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    reinterpret_cast<float4*>(pick(w, gram))[q] = acc;
}

// Gram = src^T src (src: image of a rows x r matrix); only tiles that touch the lower triangle.
// part: scratch for the `ksplit` partial matrices (used when that is more than one).
inline void tensor_gram(int r, int passes, const Batch& b, ImgRef src, int64_t rows, Sel gram, Sel part, int ksplit,
                        int only_shift_bit, cudaStream_t st) {
    const int chunks = gram_chunks(r, rows);
    tc::GemmArgs g{};
    g.Mrows = r; g.Ncols = r; g.Kdim = (int32_t)rows; g.BN = image_bn(r, r, (int64_t)b.count * (ksplit > 1 ? chunks : 1));
    g.passes = passes; g.passes2 = 1; g.a = src; g.n1 = src; g.n2 = no_img(); g.lower_only = 1;
    g.out.normal = dest_none(); g.out.normal.f32 = ksplit > 1 ? part : gram; g.out.normal.has_f32 = 1;
    g.out.shifted = g.out.normal; g.out.ld = r;
    g.cscale_off = -1;
    g.out.shift_bit = only_shift_bit; g.out.only_if_shifted = only_shift_bit ? 1 : 0;
    g.chunks = chunks;
    if (ksplit > 1) g.split_stride = (int64_t)r * r;
    else g.run = 1;
    launch_gemm<tc::A_IMG_MN, tc::N_IMG_MN, tc::EPI_STORE, 0>(b, g, prof::S_GRAM, st);
    if (ksplit > 1) {
        const int64_t total4 = (int64_t)r * r / 4;
        with_table(b, [&](const auto& t) {
            launch(gram_reduce_kernel<table_t<decltype(t)>>, dim3((unsigned)((total4 + 255) / 256), 1, (unsigned)b.count), 256, 0, 1, prof::S_GRAM, st,
                   t, gram, part, total4, ksplit, only_shift_bit);
        });
    }
}

// dst = src * L^{-T}  (src: image of a rows x r matrix; image linv holds (L^{-1})^T, read MN-major)
// unit: the columns of dst are unit vectors (second and third pass): the rounding of the diagonal of
// L^{-1} to two bf16 terms, up to 2^-18 of a column's length and hence 2^-17 in its Gram diagonal, is
// taken out again in the epilogue.
inline void tensor_apply(int r, int passes, const Batch& b, const TensorScratch& ts, ImgRef src, int64_t rows,
                         tc::OutSpec out, bool unit, cudaStream_t st) {
    tc::GemmArgs g{};
    g.Mrows = (int32_t)rows; g.Ncols = r; g.Kdim = r; g.BN = image_bn(r, rows, b.count);
    g.passes = passes; g.passes2 = 1; g.a = src; g.n1 = ts.linv; g.n2 = no_img(); g.tri = 1;
    g.colsq_off = ts.colsq;
    g.cscale_off = unit ? ts.fscale : -1;
    g.out = out;
    launch_gemm<tc::A_IMG_K, tc::N_IMG_MN, tc::EPI_STORE, 0>(b, g, prof::S_APPLY, st);
}

// M <- a (M + G) - b P R^T ;  X <- c X - d P Q^T                  (Alg. 1, update and error-feedback steps)
// fp16 = 1: both products run as one fp16 pass from the fp16 planes of P, R, Q (R's plane must
// have been written by launch_pack_right).
inline void tensor_k5(int64_t m, int64_t n, int r, int g_bf16, int x_bf16, int passes_m, int passes_x, int fp16,
                      float ef_a, float ef_b, float wc, float wd, const Batch& b, const TensorScratch& ts,
                      cudaStream_t st) {
    tc::GemmArgs g{};
    g.fp16 = fp16; g.rscale_off = ts.rscale;
    g.Mrows = (int32_t)m; g.Ncols = (int32_t)n; g.Kdim = r; g.BN = 128;
    g.passes = passes_m; g.passes2 = passes_x; g.ld = n;
    g.a = ts.p; g.n1 = ts.r; g.n2 = ts.q;
    g.ef_a = ef_a; g.ef_b = ef_b; g.wc = wc; g.wd = wd;
    g.out.normal = dest_none(); g.out.shifted = dest_none();
    const int xg = (g_bf16 ? 1 : 0) | (x_bf16 ? 2 : 0);
    switch (xg) {
        case 0: launch_gemm<tc::A_IMG_K, tc::N_IMG_K, tc::EPI_K5, 0>(b, g, prof::S_K5, st); break;
        case 1: launch_gemm<tc::A_IMG_K, tc::N_IMG_K, tc::EPI_K5, 1>(b, g, prof::S_K5, st); break;
        case 2: launch_gemm<tc::A_IMG_K, tc::N_IMG_K, tc::EPI_K5, 2>(b, g, prof::S_K5, st); break;
        default: launch_gemm<tc::A_IMG_K, tc::N_IMG_K, tc::EPI_K5, 3>(b, g, prof::S_K5, st); break;
    }
}

}  // namespace od
