// ccq_gdn_bwd_chunk_tc.cu -- the per-chunk kernels of the CCQ-Gated-DeltaNet backward for bf16 inputs
// with Dk = Dv = 128: bf16 operand tiles in shared memory, accumulators in TMEM, fp32 rows in registers.
//
// The adjoint is the one ccq_gdn_bwd_kernels.cuh states; gdn_bwd_local128_kernel and
// gdn_bwd_kv128_kernel stand in for its local and kv kernels.  Every product's operands are the bf16
// roundings of the same fp32 quantities and accumulate in fp32, as there; what differs is where they live:
//   - an operand is rounded once, into a 128-byte-swizzled tile that serves as a K-major or an MN-major
//     operand of every product that reads it (the kernels of that file convert both operands of every
//     product, a conversion pass and two block barriers each);
//   - an element-wise quantity stays in the registers of the thread that owns it, from the accumulator read
//     that makes it to the last one that needs it; row sums cross the eight threads of a row through one
//     shuffle and four shared-memory partial sums, column sums and column prefix sums run as shuffles over
//     the sixteen rows of a half-warp;
//   - a seventeenth warp issues the products (six rounds in the local kernel, five in the kv one), in an
//     order that lets the next epilogue start on the first half of a round while the rest runs.
// What bounds them: one CTA fits an SM (about 200 KB of tiles, all of TMEM), so a chunk is the latency of its
// load, its rounds and its epilogues (local: 1.9 GB of DRAM traffic at 4.0 TB/s, kv 1.6 GB at 3.6).  Measured on
// GB300 (B = 4, H = 16, T = 4096, 4096 chunks; device times): local 2420 -> 476 us, kv 2770 -> 450 us against the
// kernels of that file, suffix 279 -> 79 us; the training step 6.55 -> 1.89 ms.
//
// Thread layout: 512 compute threads.  Warp w, lane l: TMEM quadrant qd = w % 4, column group grp = w / 4;
// in a 64-row product the thread holds row i = 16 qd + l % 16 and, with hf = l / 16, columns
// 64 hf + 16 grp .. + 15 of a 128-column accumulator or 32 hf + 8 grp .. + 7 of a 64-column one; in a
// 128-row product row 32 qd + l, columns 32 grp .. + 31.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ccq_gdn_bwd.h"
#include "ccq_gdn_bwd_kernels.cuh"
#include "ccq_internal.h"
#include "sm100_ptx.cuh"

namespace ccq {

namespace {

using gbwd::GdnBwdArgs;

constexpr int kC = 64, kD = 128;
constexpr int kCompute = 512, kAll = kCompute + 32;

constexpr uint32_t ID_64x64_KK = make_idesc(64, 64, 0, 0), ID_64x64_MM = make_idesc(64, 64, 1, 1);
constexpr uint32_t ID_64x128_KK = make_idesc(64, 128, 0, 0), ID_64x128_KM = make_idesc(64, 128, 0, 1);
constexpr uint32_t ID_64x128_MM = make_idesc(64, 128, 1, 1), ID_128x128_MM = make_idesc(128, 128, 1, 1);

__device__ __forceinline__ void compute_sync() { named_bar(1, kCompute); }
// The compute threads' tiles and TMEM reads of a round are done: release the issuing warp.
__device__ __forceinline__ void signal_issue(int id) {
    fence_proxy_async_smem();
    tc_fence_before();
    named_bar_arrive(id, kAll);
}

// 256-bit global accesses (32-byte aligned; the workspace arrays are).  The stores, read again by a later kernel
// only, are the first to leave L2, where the next chunk's prefetched inputs wait.
__device__ __forceinline__ void st_global8(float *p, const float *v) {
    uint64_t policy;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    asm volatile("st.global.L2::cache_hint.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8}, %9;" ::"l"(p), "f"(v[0]), "f"(v[1]),
                 "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "l"(policy)
                 : "memory");
}
__device__ __forceinline__ void ld_global8(const float *p, float *v) {
    asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p));
}

// Accumulator columns of a 64-row product, without the wait: NR values at columns [c, c + NR) for lanes
// 0-15 and [c + OFF, c + OFF + NR) for lanes 16-31 (the same sixteen rows).
__device__ __forceinline__ void acc_ld16(uint32_t taddr, float (&v)[16]) {  // OFF = 64
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x32bx2.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16], 64;\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void acc_ld8(uint32_t taddr, float (&v)[8]) {  // OFF = 32
    uint32_t r[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x32bx2.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], 32;\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint4 pack8(const float *f) {
    return make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
}
// The thread's 16 columns of a [64][128] tile (two T64 tiles 8 KB apart) / 8 columns of a [64][64] one: the
// eight lanes of a quarter-warp write one chunk of eight consecutive rows, swizzled apart (no bank conflict).
__device__ __forceinline__ void put16(uint8_t *tile, int i, int hf, int grp, const float (&f)[16]) {
    *reinterpret_cast<uint4 *>(tile + hf * 8192 + t64_chunk(i, 2 * grp)) = pack8(f);
    *reinterpret_cast<uint4 *>(tile + hf * 8192 + t64_chunk(i, 2 * grp + 1)) = pack8(f + 8);
}
__device__ __forceinline__ void put8(uint8_t *tile, int i, int hf, int grp, const float (&f)[8]) {
    *reinterpret_cast<uint4 *>(tile + t64_chunk(i, 4 * hf + grp)) = pack8(f);
}

// The thread's 16 bf16 columns of a [64][128] tile, raw.
struct Raw16 {
    uint4 a, b;
};
__device__ __forceinline__ Raw16 get16(const uint8_t *tile, int i, int hf, int grp) {
    return Raw16{*reinterpret_cast<const uint4 *>(tile + hf * 8192 + t64_chunk(i, 2 * grp)),
                 *reinterpret_cast<const uint4 *>(tile + hf * 8192 + t64_chunk(i, 2 * grp + 1))};
}
__device__ __forceinline__ void unpack16(const Raw16 &x, float (&f)[16]) {
    float lo[8], hi[8];
    unpack_bf16x8(x.a, lo);
    unpack_bf16x8(x.b, hi);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        f[e] = lo[e];
        f[8 + e] = hi[e];
    }
}

// A [64][128] token tile (two swizzled 64-column boxes) of chunk r of (b, h).  Loads go through TMA: a
// thread's own row of a token tensor is 32 bytes in a line of its own (rows are H D apart), and loading
// q, k, v, dO that way held a CTA's first loads for 10 K cycles.
__device__ __forceinline__ void load_tokens(uint8_t *tile, const CUtensorMap *m, uint64_t *bar, int b, int h, int r) {
    tma_load_4d(tile, m, bar, 0, h, r * kC, b);
    tma_load_4d(tile + 8192, m, bar, 64, h, r * kC, b);
}
__device__ __forceinline__ void store_tokens(const CUtensorMap *m, const uint8_t *tile, int b, int h, int r) {
    tma_store_4d(m, tile, 0, h, r * kC, b);
    tma_store_4d(m, tile + 8192, 64, h, r * kC, b);
}
// 2-D tiled store of one box of an fp32 [rows][128] array (make_f32_rows_map).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *m, const void *src, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                     reinterpret_cast<uint64_t>(m)),
                 "r"(c0), "r"(c1), "r"(smem_addr(src))
                 : "memory");
}
// Four (or 4 n) fp32 columns of a row of a swizzled 32-column box.
template <int N>
__device__ __forceinline__ void put_f32(uint8_t *box, int row, int c4, const float *v) {
#pragma unroll
    for (int q = 0; q < N / 4; ++q)
        *reinterpret_cast<float4 *>(box + t64_chunk(row, c4 + q)) =
            make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}

// The fp32 chunk tiles that one kernel writes and the other reads in the same thread layout (R, U, G):
// 32 bytes a thread, consecutive threads consecutive in memory.
__device__ __forceinline__ void st_own16(float *tile, int tid, const float (&f)[16]) {
    st_global8(tile + 8 * tid, f);
    st_global8(tile + 8 * (kCompute + tid), f + 8);
}
__device__ __forceinline__ void ld_own16(const float *tile, int tid, float (&f)[16]) {
    ld_global8(tile + 8 * tid, f);
    ld_global8(tile + 8 * (kCompute + tid), f + 8);
}

// Sums over the sixteen rows of a half-warp of eight columns: leaves in v[0] the sum of column (lane >> 1) & 7.
__device__ __forceinline__ void col_sums(float (&v)[8], int lane) {
#pragma unroll
    for (int m = 4, o = 8; m >= 1; m >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (e < m) {
                const float send = up ? v[e] : v[e + m], keep = up ? v[e + m] : v[e];
                v[e] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Row sums: the eight threads of row i add up (two by shuffle, four through red[4][64]).
__device__ __forceinline__ void row_part(float *red, int grp, int i, int hf, float x) {
    x += __shfl_xor_sync(0xffffffffu, x, 16);
    if (hf == 0) red[grp * kC + i] = x;
}
__device__ __forceinline__ float row_total(const float *red, int i) {
    return (red[i] + red[kC + i]) + (red[2 * kC + i] + red[3 * kC + i]);
}

// The scalars of the chunk's tokens, by the issuing warp (two tokens a lane): in-chunk cumulative log
// decay gc (held past the sequence; summed token by token, one lane), E = e^{gc}, 1 / t, beta, lambda.
__device__ __forceinline__ void token_scalars(const GdnBwdArgs &a, int b, int h, int r, int lane, float *gc, float *E,
                                              float *be, float *tinv, float *lam) {
    const int t0 = r * kC + 2 * lane;
    const bool v0 = t0 < a.T, v1 = t0 + 1 < a.T;
    const size_t r0 = (static_cast<size_t>(b) * a.T + (v0 ? t0 : 0)) * a.H + h;
    const size_t r1 = (static_cast<size_t>(b) * a.T + (v1 ? t0 + 1 : 0)) * a.H + h;
    *reinterpret_cast<float2 *>(gc + 2 * lane) = make_float2(v0 ? a.g[r0] : 0.f, v1 ? a.g[r1] : 0.f);
    be[2 * lane] = v0 ? a.beta[r0] : 0.f;
    be[2 * lane + 1] = v1 ? a.beta[r1] : 0.f;
    if (lam) {
        lam[2 * lane] = v0 ? a.lambda[r0] : 0.f;
        lam[2 * lane + 1] = v1 ? a.lambda[r1] : 0.f;
    }
    const float ts = static_cast<float>((a.t0 ? a.t0[b] : 0) + static_cast<int64_t>(r) * kC);
    tinv[2 * lane] = 1.f / (ts + 1.f + static_cast<float>(2 * lane));
    tinv[2 * lane + 1] = 1.f / (ts + 1.f + static_cast<float>(2 * lane + 1));
    __syncwarp();
    if (lane == 0) {
        float acc = 0.f;
#pragma unroll
        for (int q = 0; q < kC / 4; ++q) {
            float4 x = *reinterpret_cast<const float4 *>(gc + 4 * q);
            x.x = acc + x.x;
            x.y = x.x + x.y;
            x.z = x.y + x.z;
            acc = x.w = x.z + x.w;
            *reinterpret_cast<float4 *>(gc + 4 * q) = x;
        }
    }
    __syncwarp();
    E[2 * lane] = expf(gc[2 * lane]);
    E[2 * lane + 1] = expf(gc[2 * lane + 1]);
}

// Sums over a row's columns in eight interleaved parts (columns p, p + 8, ..., each summed in order, then
// the parts in order): four neighbouring threads take two parts each.  The order is that of row_sums() in
// ccq_gdn_bwd_kernels.cuh.
__device__ __forceinline__ float parts_total(float p0, float p1, int lane) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        s += __shfl_sync(0xffffffffu, p0, (lane & 28) + q);
        s += __shfl_sync(0xffffffffu, p1, (lane & 28) + q);
    }
    return s;
}
// Columns 2 qtr, 2 qtr + 1 of every 16-byte chunk of row `row` of a raw [64][128] tile.
__device__ __forceinline__ void load_parts(const uint8_t *tile, int row, int qtr, uint32_t (&w)[16]) {
#pragma unroll
    for (int c = 0; c < 16; ++c)
        w[c] = *reinterpret_cast<const uint32_t *>(tile + (c >> 3) * 8192 + t64_chunk(row, c & 7) + 4 * qtr);
}
__device__ __forceinline__ float lo_bf16(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_bf16(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
// 1 / |row| of the raw q (threads 0-255) and k (256-511) tiles: row (tid % 256) / 4, the row's four
// threads return the same value; w keeps the values read.  ODD_FIRST (the kv kernel): the k rows' parts are added odd
// part of each pair first, as the generic kv kernel mostly adds them by atomics, so a row's kbar can round to
// another bf16 there than in the local kernel.  Neither order is the more accurate one; the gradients' errors
// against 64 bits are the same with either.
template <bool ODD_FIRST = false>
__device__ __forceinline__ float row_norms(const uint8_t *qt, const uint8_t *kt, int tid, int l2norm, uint32_t (&w)[16]) {
    load_parts(tid < 256 ? qt : kt, (tid & 255) >> 2, tid & 3, w);
    float p0 = 0.f, p1 = 0.f;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        p0 = fmaf(lo_bf16(w[c]), lo_bf16(w[c]), p0);
        p1 = fmaf(hi_bf16(w[c]), hi_bf16(w[c]), p1);
    }
    const bool odd = ODD_FIRST && tid >= 256;
    return gbwd::rnorm_of(parts_total(odd ? p1 : p0, odd ? p0 : p1, tid & 31), l2norm);
}

// K = 64 or 128 products over T64 tiles.  A and B: descriptors of the first K = 16 step; K-major operands
// advance 32 B a step and `*blk` (tile bytes >> 4) every 64, MN-major ones 2 KB a step.
template <int K, bool AM, bool BM>
__device__ __forceinline__ void mma_k(uint32_t d, uint64_t A, int ablk, uint64_t B, int bblk, uint32_t id, bool acc) {
#pragma unroll
    for (int k = 0; k < K / 16; ++k)
        mma_bf16(d, A + (AM ? k * 128 : (k >> 2) * ablk + (k & 3) * 2), B + (BM ? k * 128 : (k >> 2) * bblk + (k & 3) * 2),
                 id, (acc || k > 0) ? 1u : 0u);
}

// L2 prefetch of the token tiles of chunk ch.
__device__ __forceinline__ void prefetch_tokens(const CUtensorMap *m, const GdnBwdArgs &a, int ch) {
    const int r = ch % a.NC, bh = ch / a.NC, b = bh / a.H, h = bh % a.H;
    tma_prefetch_l2_4d(m, 0, h, r * kC, b);
    tma_prefetch_l2_4d(m, 64, h, r * kC, b);
}

// =====================================================================================
// gdn_bwd_local128_kernel: one CTA per (sequence, head, chunk)
// =====================================================================================
namespace lk {
constexpr uint32_t OFF_Q = 0;        // qbar, then dq
constexpr uint32_t OFF_K = 16384;    // kbar
constexpr uint32_t OFF_SK = 32768;   // S^K_r (32 KB)
constexpr uint32_t OFF_H = 65536;    // H_r (32 KB); then, with U and q_clean, Y1 and DC on their way out
constexpr uint32_t OFF_R = 98304;    // v, then R, then W
constexpr uint32_t OFF_U = 114688;   // U
constexpr uint32_t OFF_QC = 131072;  // q_clean
constexpr uint32_t OFF_D = 147456;   // D = scale dO; then, with E D, X1 on its way out
constexpr uint32_t OFF_ED = 163840;  // diag(E) D
constexpr uint32_t OFF_TB = 180224;  // Tt diag(beta), then dP
constexpr uint32_t OFF_SA = 188416;  // (Qbar Kbar^T) o causal, then P, then (W Kbar^T) o causal
constexpr uint32_t OFF_MISC = 196608;
constexpr int F_GC = 0, F_E = 64, F_BE = 128, F_TI = 192, F_LAM = 256, F_M = 320, F_SEG = 448, F_RN = 960,
              F_CQ = 1088, F_RED = 1152, kReds = 4, kFloats = F_RED + kReds * 256;
constexpr int LS = 72;               // row stride (floats) of the fp32 copy of masked Sc in U's and q_clean's place
constexpr uint32_t M_BAR = kFloats * 4, M_TMEM = M_BAR + 96, M_ABORT = M_TMEM + 4;
constexpr uint32_t kSmem = OFF_MISC + M_ABORT + 4 + 1024;
static_assert(kSmem <= 232448, "exceeds the 227 KB per-CTA limit");
enum { BTOK = 0, BIN, B1, B2, B2B, B3, B3B, B4, B5, B5B, B6, kBars };
static_assert(8 * kBars <= 96, "barriers reach the TMEM slot");
static_assert(OFF_QC == OFF_U + 16384 && 64 * LS * 4 <= 32768, "the fp32 staging spans U and q_clean");
// TMEM columns: Sc, then P | dP, then dP Kbar, then W Kbar^T | KH, U, Y1, DC | z, X1, the dqbar terms | (E D) H^T
constexpr uint32_t TM_A = 0, TM_A2 = 64, TM_B = 128, TM_C = 256, TM_D = 384;
}  // namespace lk

// Box g (32 fp32 columns of 128 rows, 16 KB) of a [128][128] array on its way out: H's tile, then U and q_clean.
__device__ __forceinline__ uint8_t *square_box(uint8_t *sm, int g) {
    return sm + (g < 2 ? lk::OFF_H + g * 16384 : lk::OFF_U + (g - 2) * 16384);
}

// Per chunk, everything that does not need dH.  Rounds (products, then the epilogue they feed):
//   1  Sc = Qbar Kbar^T, KH = Kbar H | Z = Qbar S^K     masked Sc, cq, R = V - E KH
//   2  U = Tb R | Z += Sc Kbar                           U, z, q_clean
//   3  P = Qc Kbar^T, dP = D U^T | (E D) H^T, Y1 = Qc^T (E D)   P, dP; E rowsum((Qc H) o D); Y1
//   4  dP Kbar, X1 = P^T D                               dqc, dlambda, W; X1
//   5  Wk = W Kbar^T | W S^K, DC = W^T Qbar              masked Wk, cz; DC
//   6  += Wk Kbar                                        dqbar, dq, the Dm increment
__global__ void __launch_bounds__(kAll, 1)
gdn_bwd_local128_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                        const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_do,
                        const __grid_constant__ CUtensorMap map_dq, const __grid_constant__ CUtensorMap map_x1,
                        const __grid_constant__ CUtensorMap map_y1, const __grid_constant__ CUtensorMap map_dc,
                        const GdnBwdArgs a) {
    using namespace lk;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = smem_align1024(smem_raw);
    const uint32_t sb = smem_addr(sm);
    float *fm = reinterpret_cast<float *>(sm + OFF_MISC);
    float *gc = fm + F_GC, *E = fm + F_E, *be = fm + F_BE, *tinv = fm + F_TI, *lam = fm + F_LAM, *M = fm + F_M;
    float *segs = fm + F_SEG, *rn = fm + F_RN, *cqs = fm + F_CQ, *red = fm + F_RED;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + OFF_MISC + M_BAR);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + OFF_MISC + M_TMEM);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + OFF_MISC + M_ABORT);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ch = blockIdx.x, r = ch % a.NC, bh = ch / a.NC, b = bh / a.H, h = bh % a.H;
    const int n = min(kC, a.T - r * kC);
    const size_t t64 = static_cast<size_t>(ch) * kC * kD;
    int *status = a.status;

    if (warp == kCompute / 32) {
        // ---- the issuing warp
        if (lane == 0) {
            for (int i = 0; i < kBars; ++i) mbar_init(&bar[i], 1);
            *abort_flag = 0;
            fence_barrier_init();
        }
        grid_wait();
        if (lane == 0) {
            mbar_arrive_expect_tx(&bar[BTOK], 4 * 16384 + 512);
            load_tokens(sm + OFF_Q, &map_q, &bar[BTOK], b, h, r);
            load_tokens(sm + OFF_K, &map_k, &bar[BTOK], b, h, r);
            bulk_load(M, a.mk + static_cast<size_t>(ch) * kD, 512, &bar[BTOK]);
            load_tokens(sm + OFF_D, &map_do, &bar[BTOK], b, h, r);
            load_tokens(sm + OFF_R, &map_v, &bar[BTOK], b, h, r);
            mbar_arrive_expect_tx(&bar[BIN], 65536);
            bulk_load(sm + OFF_H, a.hs_img + static_cast<size_t>(ch) * 32768, 32768, &bar[BIN]);
            bulk_load(sm + OFF_SK, a.sk_img + static_cast<size_t>(ch) * 32768, 32768, &bar[BIN]);
        }
        token_scalars(a, b, h, r, lane, gc, E, be, tinv, lam);
        __syncthreads();  // scalars, partial norms, M, TMEM
        const uint32_t tb = *tmem_slot;
        const uint64_t dQ = make_desc(sb + OFF_Q, 16, 1024), dQm = make_desc(sb + OFF_Q, 8192, 1024);
        const uint64_t dK = make_desc(sb + OFF_K, 16, 1024), dKm = make_desc(sb + OFF_K, 8192, 1024);
        const uint64_t dSKm = make_desc(sb + OFF_SK, 16384, 1024);
        const uint64_t dH = make_desc(sb + OFF_H, 16, 1024), dHm = make_desc(sb + OFF_H, 16384, 1024);
        const uint64_t dR = make_desc(sb + OFF_R, 16, 1024), dRm = make_desc(sb + OFF_R, 8192, 1024);
        const uint64_t dU = make_desc(sb + OFF_U, 16, 1024);
        const uint64_t dQC = make_desc(sb + OFF_QC, 16, 1024), dQCm = make_desc(sb + OFF_QC, 8192, 1024);
        const uint64_t dD = make_desc(sb + OFF_D, 16, 1024), dDm = make_desc(sb + OFF_D, 8192, 1024);
        const uint64_t dED = make_desc(sb + OFF_ED, 16, 1024), dEDm = make_desc(sb + OFF_ED, 8192, 1024);
        const uint64_t dTB = make_desc(sb + OFF_TB, 16, 1024);
        const uint64_t dSA = make_desc(sb + OFF_SA, 16, 1024), dSAm = make_desc(sb + OFF_SA, 8192, 1024);
        int last = -1;  // the last committed round, for the drain after a give-up
        auto go = [&] { return lane == 0 && !*abort_flag; };
        named_bar(2, kAll);
        mbar_wait(&bar[BIN], 0, abort_flag, status);
        tc_fence_after();
        if (go()) {
            mma_k<128, false, false>(tb + TM_A, dQ, 512, dK, 512, ID_64x64_KK, false);
            mma_k<128, false, true>(tb + TM_B, dK, 512, dHm, 0, ID_64x128_KM, false);
            mma_commit(&bar[B1]);
            mma_k<128, false, true>(tb + TM_C, dQ, 512, dSKm, 0, ID_64x128_KM, false);
            last = B1;
        }
        named_bar(3, kAll);
        tc_fence_after();
        if (go()) {
            mma_k<64, false, true>(tb + TM_B, dTB, 0, dRm, 0, ID_64x128_KM, false);
            mma_commit(&bar[B2]);
            mma_k<64, false, true>(tb + TM_C, dSA, 0, dKm, 0, ID_64x128_KM, true);
            mma_commit(&bar[B2B]);
            last = B2B;
        }
        named_bar(2, kAll);
        tc_fence_after();
        if (go()) {
            mma_k<128, false, false>(tb + TM_A, dQC, 512, dK, 512, ID_64x64_KK, false);
            mma_k<128, false, false>(tb + TM_A2, dD, 512, dU, 512, ID_64x64_KK, false);
            mma_commit(&bar[B3]);
            mma_k<128, false, false>(tb + TM_D, dED, 512, dH, 1024, ID_64x128_KK, false);
            mma_k<64, true, true>(tb + TM_B, dQCm, 0, dEDm, 0, ID_128x128_MM, false);
            // q_clean as the kv kernel's operand tile (read before B3B: Y1 then goes over it)
            bulk_store(a.qc + t64 / 2, sm + OFF_QC, 16384);
            tma_store_commit();
            tma_store_wait_read();
            mma_commit(&bar[B3B]);
            last = B3B;
        }
        named_bar(3, kAll);
        tc_fence_after();
        if (go()) {
            mma_k<64, false, true>(tb + TM_A, dTB, 0, dKm, 0, ID_64x128_KM, false);
            mma_k<64, true, true>(tb + TM_C, dSAm, 0, dDm, 0, ID_64x128_MM, false);
            mma_commit(&bar[B4]);
            last = B4;
        }
        named_bar(2, kAll);
        tc_fence_after();
        if (go()) {
            mma_k<128, false, false>(tb + TM_A, dR, 512, dK, 512, ID_64x64_KK, false);
            mma_commit(&bar[B5]);
            mma_k<128, false, true>(tb + TM_C, dR, 512, dSKm, 0, ID_64x128_KM, false);
            mma_k<64, true, true>(tb + TM_B, dRm, 0, dQm, 0, ID_128x128_MM, false);
            mma_commit(&bar[B5B]);
            bulk_store(a.w_img + static_cast<size_t>(ch) * 16384, sm + OFF_R, 16384);  // W likewise
            tma_store_commit();
            last = B5B;
        }
        {
            // the chunk one wave later finds its inputs in L2
            const int nx = ch + a.wave;
            if (lane == 0 && a.wave > 0 && nx < static_cast<int>(gridDim.x)) {
                prefetch_tokens(&map_q, a, nx);
                prefetch_tokens(&map_k, a, nx);
                prefetch_tokens(&map_do, a, nx);
                prefetch_tokens(&map_v, a, nx);
                bulk_prefetch_l2(a.hs_img + static_cast<size_t>(nx) * 32768, 32768);
                bulk_prefetch_l2(a.sk_img + static_cast<size_t>(nx) * 32768, 32768);
                bulk_prefetch_l2(a.tt + static_cast<size_t>(nx) * kC * kC, kC * kC * 4);
            }
        }
        named_bar(3, kAll);
        tc_fence_after();
        if (go()) {
            mma_k<64, false, true>(tb + TM_C, dSA, 0, dKm, 0, ID_64x128_KM, true);
            mma_commit(&bar[B6]);
            last = B6;
        }
        if (lane == 0 && *abort_flag) {
            mbar_drain(&bar[BTOK], 0);
            mbar_drain(&bar[BIN], 0);
            if (last >= 0) mbar_drain(&bar[last], 0);
        }
        if (lane == 0) tma_store_wait_read();
        __syncthreads();
        return;
    }

    // ---- the compute threads
    const int qd = warp & 3, grp = warp >> 2, hf = lane >> 4, i = 16 * qd + (lane & 15);
    const int c0 = 64 * hf + 16 * grp, s0 = 32 * hf + 8 * grp;
    if (warp == 0) tmem_alloc(tmem_slot, 512);
    grid_wait();
    const bool valid = i < n;
    const size_t row = (static_cast<size_t>(b) * a.T + r * kC + (valid ? i : 0)) * a.H + h;
    __syncthreads();
    const uint32_t tb = *tmem_slot, tq = tb + (static_cast<uint32_t>(32 * qd) << 16);
    mbar_wait(&bar[BTOK], 0, abort_flag, status);
    const Raw16 qr = get16(sm + OFF_Q, i, hf, grp), kr = get16(sm + OFF_K, i, hf, grp);
    // row norms, and (threads 0-255) the M . qbar terms of cq in the same interleaved parts
    float m0 = 0.f, m1 = 0.f;
    {
        uint32_t w[16];
        const float rr = row_norms(sm + OFF_Q, sm + OFF_K, tid, a.l2norm, w);
        if ((tid & 3) == 0) rn[tid >> 2] = rr;
        if (tid < 256) {
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const float2 mm = *reinterpret_cast<const float2 *>(M + 8 * c + 2 * (tid & 3));
                m0 = fmaf(mm.x, lo_bf16(w[c]) * rr, m0);
                m1 = fmaf(mm.y, hi_bf16(w[c]) * rr, m1);
            }
        }
    }
    compute_sync();
    const float rq = rn[i], rk = rn[kC + i];
    float qb[16], x[16], cum[16];
    float4 *fst = reinterpret_cast<float4 *>(sm + OFF_U);  // fp32 [64][128], 16-byte chunks c ^ (row & 7)
    unpack16(qr, qb);
    unpack16(kr, x);
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        qb[e] *= rq;
        x[e] *= rk;
    }
    put16(sm + OFF_Q, i, hf, grp, qb);
    put16(sm + OFF_K, i, hf, grp, x);
#pragma unroll
    for (int q = 0; q < 4; ++q)
        fst[i * 32 + ((c0 / 4 + q) ^ (i & 7))] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
    {
        float d[16];
        unpack16(get16(sm + OFF_D, i, hf, grp), d);
#pragma unroll
        for (int e = 0; e < 16; ++e) d[e] *= a.scale;
        put16(sm + OFF_D, i, hf, grp, d);
#pragma unroll
        for (int e = 0; e < 16; ++e) d[e] *= E[i];
        put16(sm + OFF_ED, i, hf, grp, d);
    }
    {
        // Tt diag(beta): row tid / 8, columns 8 (tid % 8) .. + 7
        float t[8];
        ld_global8(a.tt + static_cast<size_t>(ch) * kC * kC + 8 * tid, t);
#pragma unroll
        for (int e = 0; e < 8; ++e) t[e] *= be[8 * (tid & 7) + e];
        *reinterpret_cast<uint4 *>(sm + OFF_TB + t64_chunk(tid >> 3, tid & 7)) = pack8(t);
    }
    signal_issue(2);
    // while round 1 runs: CumK_i = M + sum_{j <= i} kbar_j, a thread per column and sixteen rows
    compute_sync();
    {
        const int j = tid & 127, sg = tid >> 7;
        float *col = reinterpret_cast<float *>(fst) + (j & 3);
        float kv[16], acc = 0.f;
#pragma unroll
        for (int l = 0; l < 16; ++l) kv[l] = col[(16 * sg + l) * 128 + 4 * ((j >> 2) ^ (l & 7))];
#pragma unroll
        for (int l = 0; l < 16; ++l) acc += kv[l];
        segs[sg * kD + j] = acc;
        compute_sync();
        float c = M[j];
        for (int s = 0; s < sg; ++s) c += segs[s * kD + j];
#pragma unroll
        for (int l = 0; l < 16; ++l) {
            c += kv[l];
            col[(16 * sg + l) * 128 + 4 * ((j >> 2) ^ (l & 7))] = c;
        }
    }
    compute_sync();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 y = fst[i * 32 + ((c0 / 4 + q) ^ (i & 7))];
        cum[4 * q] = y.x;
        cum[4 * q + 1] = y.y;
        cum[4 * q + 2] = y.z;
        cum[4 * q + 3] = y.w;
    }
    compute_sync();

    // ---- round 1: masked Sc, cq, R
    mbar_wait(&bar[B1], 0, abort_flag, status);
    tc_fence_after();
    float *scf = reinterpret_cast<float *>(sm + OFF_U);  // [64][LS]
    {
        float s[8];
        acc_ld8(tq + TM_A + 8 * grp, s);
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] = s0 + e <= i ? s[e] : 0.f;
        put8(sm + OFF_SA, i, hf, grp, s);
        *reinterpret_cast<float4 *>(scf + i * LS + s0) = make_float4(s[0], s[1], s[2], s[3]);
        *reinterpret_cast<float4 *>(scf + i * LS + s0 + 4) = make_float4(s[4], s[5], s[6], s[7]);
        float v[16];
        unpack16(get16(sm + OFF_R, i, hf, grp), v);
        acc_ld16(tq + TM_B + 16 * grp, x);
        const float ei = E[i];
#pragma unroll
        for (int e = 0; e < 16; ++e) x[e] = fmaf(-ei, x[e], v[e]);
        put16(sm + OFF_R, i, hf, grp, x);
        signal_issue(3);
        st_own16(a.r + t64, tid, x);
    }
    compute_sync();
    if (tid < 256) {
        // cq_i = CumK_i . qbar_i = M . qbar_i + sum_{j <= i} Sc_ij
        const float *sr = scf + (tid >> 2) * LS + 2 * (tid & 3);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float2 y = *reinterpret_cast<const float2 *>(sr + 8 * c);
            m0 += y.x;
            m1 += y.y;
        }
        const float t = parts_total(m0, m1, lane);
        if ((tid & 3) == 0) cqs[tid >> 2] = t;
    }
    compute_sync();
    const float cf = a.centered ? 1.f : 0.f, ti = tinv[i];
    const float cq = cqs[i];
    // ---- round 2: U, z, q_clean
    mbar_wait(&bar[B2], 0, abort_flag, status);
    tc_fence_after();
    acc_ld16(tq + TM_B + 16 * grp, x);
    put16(sm + OFF_U, i, hf, grp, x);
    st_own16(a.u + t64, tid, x);
    mbar_wait(&bar[B2B], 0, abort_flag, status);
    tc_fence_after();
    float z[16];
    acc_ld16(tq + TM_C + 16 * grp, z);
    {
        const float li = lam[i];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            z[e] = z[e] * ti - cf * cum[e] * cq * ti * ti;
            x[e] = qb[e] - li * z[e];
        }
    }
    put16(sm + OFF_QC, i, hf, grp, x);
    signal_issue(2);
    // ---- round 3: P, dP; E rowsum((Qc H) o D); Y1
    float gam[8];  // Gamma o causal
    {
        const float gi = gc[i];
#pragma unroll
        for (int e = 0; e < 8; ++e) gam[e] = s0 + e <= i ? expf(gi - gc[s0 + e]) : 0.f;
    }
    mbar_wait(&bar[B3], 0, abort_flag, status);
    tc_fence_after();
    {
        float p[8];
        acc_ld8(tq + TM_A + 8 * grp, p);
#pragma unroll
        for (int e = 0; e < 8; ++e) p[e] = s0 + e <= i ? p[e] * gam[e] : 0.f;
        put8(sm + OFF_SA, i, hf, grp, p);
        acc_ld8(tq + TM_A2 + 8 * grp, p);
#pragma unroll
        for (int e = 0; e < 8; ++e) p[e] = s0 + e <= i ? p[e] * gam[e] : 0.f;
        put8(sm + OFF_TB, i, hf, grp, p);
    }
    signal_issue(3);
    mbar_wait(&bar[B3B], 0, abort_flag, status);
    tc_fence_after();
    float dqc[16];
    acc_ld16(tq + TM_D + 16 * grp, dqc);
    {
        float part = 0.f;
#pragma unroll
        for (int e = 0; e < 16; ++e) part = fmaf(x[e], dqc[e], part);
        row_part(red, grp, i, hf, part);
        float y[32];
        tmem_ld32(tq + TM_B + 32 * grp, y);
        // Y1 by TMA through the tiles of H, U and q_clean, whose products are done: one 32-column box a group
        put_f32<32>(square_box(sm, grp), 32 * qd + lane, 0, y);
    }
    fence_proxy_async_smem();
    compute_sync();
    if (tid < 4) {
        tma_store_2d(&map_y1, square_box(sm, tid), 32 * tid, ch * kD);
        tma_store_commit();
    }
    // ---- round 4: dqc, dlambda, W; X1
    mbar_wait(&bar[B4], 0, abort_flag, status);
    tc_fence_after();
    acc_ld16(tq + TM_A + 16 * grp, x);
    float mw = 0.f;
    {
        float part = 0.f;
        const float li = lam[i];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            dqc[e] = x[e] + dqc[e];
            part = fmaf(z[e], dqc[e], part);
            z[e] = -li * dqc[e] * ti;  // W = dz / t from here on
            mw = fmaf(M[c0 + e], z[e], mw);
        }
        put16(sm + OFF_R, i, hf, grp, z);
        row_part(red + 256, grp, i, hf, part);
        acc_ld16(tq + TM_C + 16 * grp, x);
    }
    put_f32<16>(sm + OFF_D + (2 * hf + (grp >> 1)) * 8192, i, 4 * (grp & 1), x);  // X1 in the tiles of D and E D
    signal_issue(2);
    // ---- round 5: masked W Kbar^T, cz; DC
    mbar_wait(&bar[B5], 0, abort_flag, status);
    tc_fence_after();
    {
        float s[8], part = mw;
        acc_ld8(tq + TM_A + 8 * grp, s);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            s[e] = s0 + e <= i ? s[e] : 0.f;
            part += s[e];
        }
        put8(sm + OFF_SA, i, hf, grp, s);
        row_part(red + 512, grp, i, hf, part);
    }
    if (tid < 4) tma_store_wait_read();  // Y1 has left its tiles
    signal_issue(3);
    compute_sync();
    if (tid < 4) {
        tma_store_2d(&map_x1, sm + OFF_D + tid * 8192, 32 * tid, ch * kC);
        tma_store_commit();
    }
    const float cz = row_total(red + 512, i) / ti;
    if (grp == 0 && hf == 0) {
        float *vec = a.vec + static_cast<size_t>(ch) * 4 * kC;
        vec[i] = cq;
        vec[kC + i] = cz;
        vec[2 * kC + i] = valid ? row_total(red, i) : 0.f;
        if (valid && a.dlambda) a.dlambda[row] = -row_total(red + 256, i);
    }
    mbar_wait(&bar[B5B], 0, abort_flag, status);
    tc_fence_after();
    {
        float y[32];
        tmem_ld32(tq + TM_B + 32 * grp, y);
        put_f32<32>(square_box(sm, grp), 32 * qd + lane, 0, y);
    }
    fence_proxy_async_smem();
    {
        // the reverse sums G_i = sum_{l >= i} (W_l cq_l t_l + qbar_l cz_l) / t_l^2 for dk (sixteen rows by shuffle,
        // the quadrants' totals through segs); G of the first row is the Dm increment
        const float ct = cq / ti, t2 = ti * ti;
#pragma unroll
        for (int e = 0; e < 16; ++e) z[e] = (z[e] * ct + qb[e] * cz) * t2;
#pragma unroll
        for (int o = 1; o < 16; o <<= 1)
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const float y = __shfl_down_sync(0xffffffffu, z[e], o, 16);
                if ((lane & 15) + o < 16) z[e] += y;
            }
        if ((lane & 15) == 0)
#pragma unroll
            for (int e = 0; e < 16; e += 4)
                *reinterpret_cast<float4 *>(segs + qd * kD + c0 + e) = make_float4(z[e], z[e + 1], z[e + 2], z[e + 3]);
    }
    // ---- round 6: dqbar, dq
    mbar_wait(&bar[B6], 0, abort_flag, status);
    tc_fence_after();
    acc_ld16(tq + TM_C + 16 * grp, x);
    {
        float part = 0.f;
        const float k2 = cf * cz * ti * ti;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            dqc[e] = dqc[e] + x[e] - cum[e] * k2;
            part = fmaf(qb[e], dqc[e], part);
        }
        row_part(red + 768, grp, i, hf, part);
    }
    tc_fence_before();
    compute_sync();
    if (tid < 4) {
        tma_store_2d(&map_dc, square_box(sm, tid), 32 * tid, ch * kD);
        tma_store_commit();
    }
    {
        for (int s = qd + 1; s < 4; ++s)
#pragma unroll
            for (int e = 0; e < 16; e += 4) {
                const float4 y = *reinterpret_cast<const float4 *>(segs + s * kD + c0 + e);
                z[e] += y.x;
                z[e + 1] += y.y;
                z[e + 2] += y.z;
                z[e + 3] += y.w;
            }
        st_own16(a.w + t64, tid, z);
        const float rdot = a.l2norm ? row_total(red + 768, i) : 0.f;
#pragma unroll
        for (int e = 0; e < 16; ++e) x[e] = (dqc[e] - qb[e] * rdot) * rq;
        put16(sm + OFF_Q, i, hf, grp, x);
        fence_proxy_async_smem();
        compute_sync();
        if (tid == 0) {
            store_tokens(&map_dq, sm + OFF_Q, b, h, r);
            tma_store_commit();
        }
    }
    if (tid < 4) tma_store_wait_read();
    if (tid < kD)
        a.dm[static_cast<size_t>(ch) * kD + tid] = -cf * ((segs[tid] + segs[kD + tid]) + (segs[2 * kD + tid] + segs[3 * kD + tid]));
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tb, 512);
    }
}

// =====================================================================================
// gdn_bwd_kv128_kernel: one CTA per (sequence, head, chunk)
// =====================================================================================
namespace kk {
constexpr uint32_t OFF_K = 0;        // kbar, then dk
constexpr uint32_t OFF_Q = 16384;    // qbar
constexpr uint32_t OFF_W = 32768;    // W
constexpr uint32_t OFF_D = 49152;    // D = scale dO, then R, then dR
constexpr uint32_t OFF_DU = 65536;   // dU
constexpr uint32_t OFF_QC = 81920;   // q_clean, then (with U) the staging of dKK^T
constexpr uint32_t OFF_U = 98304;    // U
constexpr uint32_t OFF_DH = 114688;  // dH (32 KB), then DC_{r+1} + DC_{r+1}^T
constexpr uint32_t OFF_H = 147456;   // H_r (32 KB)
constexpr uint32_t OFF_TT = 180224;  // Tt
constexpr uint32_t OFF_DP = 188416;  // dP, then M2
constexpr uint32_t OFF_QK = 196608;  // v (with the next tile), then (Qbar Kbar^T) o causal
constexpr uint32_t OFF_WK = 204800;  // (W Kbar^T) o causal
constexpr uint32_t OFF_DT = 212992;  // dTb, then dKK + dKK^T
constexpr uint32_t OFF_MISC = 221184;
constexpr int F_GC = 0, F_E = 64, F_BE = 128, F_TI = 192, F_PCS = 256, F_CS = 320, F_DB = 384, F_RN = 448,
              F_RED = 576, kReds = 5, kFloats = F_RED + kReds * 256;
constexpr uint32_t M_BAR = kFloats * 4, M_TMEM = M_BAR + 96, M_ABORT = M_TMEM + 4;
constexpr uint32_t kSmem = OFF_MISC + M_ABORT + 4 + 1024;
static_assert(kSmem <= 232448, "exceeds the 227 KB per-CTA limit");
static_assert(OFF_U == OFF_QC + 16384 && 64 * 65 * 4 <= 32768, "the dKK staging spans q_clean and U");
static_assert(M_BAR % 8 == 0, "barrier alignment");
enum { BTOK = 0, BIN, BDC, B1, B1B, B2, B2B, B3, B4, B5, kBars };
static_assert(8 * kBars <= 96, "barriers reach the TMEM slot");
// TMEM columns: t, then dR, then dR H^T | S, dP, then U dH^T | KK | QK, WK, then the sum of dk's other
// products | dTb, then M2, then dA
constexpr uint32_t TM_T = 0, TM_S = 128, TM_P = 192, TM_KK = 256, TM_ACC = 320, TM_WK = 384, TM_X = 448;
constexpr int LS = 65;  // row stride of the dKK staging (floats)
}  // namespace kk

// Per chunk: dv, dk, dbeta, dg.  Rounds:
//   1  t = Kbar dH, S = Qc Kbar^T, dP = D U^T | QK, WK, KK       dU, dP, sums of dP o S; masked QK, WK
//   2  Tt^T dU, dTb = dU R^T | dP^T Qc + QK^T W + WK^T Qbar, U dH^T     dR = dv, dTb
//   3  M2 = Tt^T dTb | dR H^T                                    M2 diag(beta)
//   4  dA = M2 Tt^T                                              dKK + dKK^T
//   5  += (dKK + dKK^T) Kbar + Kbar (DC + DC^T)                  dk
__global__ void __launch_bounds__(kAll, 1)
gdn_bwd_kv128_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                     const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_do,
                     const __grid_constant__ CUtensorMap map_dv, const __grid_constant__ CUtensorMap map_dk,
                     const GdnBwdArgs a) {
    using namespace kk;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = smem_align1024(smem_raw);
    const uint32_t sb = smem_addr(sm);
    float *fm = reinterpret_cast<float *>(sm + OFF_MISC);
    float *gc = fm + F_GC, *E = fm + F_E, *be = fm + F_BE, *tinv = fm + F_TI, *pcs = fm + F_PCS, *cs = fm + F_CS;
    float *db1 = fm + F_DB, *rn = fm + F_RN, *red = fm + F_RED;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + OFF_MISC + M_BAR);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + OFF_MISC + M_TMEM);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + OFF_MISC + M_ABORT);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ch = blockIdx.x, r = ch % a.NC, bh = ch / a.NC, b = bh / a.H, h = bh % a.H;
    const int n = min(kC, a.T - r * kC);
    const size_t t64 = static_cast<size_t>(ch) * kC * kD;
    const float *vec = a.vec + static_cast<size_t>(ch) * 4 * kC;
    const float cf = a.centered ? 1.f : 0.f;
    int *status = a.status;

    if (warp == kCompute / 32) {
        // ---- the issuing warp
        if (lane == 0) {
            for (int i = 0; i < kBars; ++i) mbar_init(&bar[i], 1);
            *abort_flag = 0;
            fence_barrier_init();
        }
        grid_wait();
        if (lane == 0) {
            const size_t img = static_cast<size_t>(ch) * 32768;
            mbar_arrive_expect_tx(&bar[BTOK], 4 * 16384);
            load_tokens(sm + OFF_K, &map_k, &bar[BTOK], b, h, r);
            load_tokens(sm + OFF_Q, &map_q, &bar[BTOK], b, h, r);
            load_tokens(sm + OFF_D, &map_do, &bar[BTOK], b, h, r);
            load_tokens(sm + OFF_QK, &map_v, &bar[BTOK], b, h, r);
            mbar_arrive_expect_tx(&bar[BIN], 2 * 16384 + 65536);
            bulk_load(sm + OFF_DH, a.dh_img + img, 32768, &bar[BIN]);
            bulk_load(sm + OFF_QC, a.qc + t64 / 2, 16384, &bar[BIN]);
            bulk_load(sm + OFF_W, a.w_img + static_cast<size_t>(ch) * 16384, 16384, &bar[BIN]);
            bulk_load(sm + OFF_H, a.hs_img + img, 32768, &bar[BIN]);
        }
        token_scalars(a, b, h, r, lane, gc, E, be, tinv, nullptr);
        __syncthreads();
        const uint32_t tb = *tmem_slot;
        const uint64_t dK = make_desc(sb + OFF_K, 16, 1024), dKm = make_desc(sb + OFF_K, 8192, 1024);
        const uint64_t dQ = make_desc(sb + OFF_Q, 16, 1024), dQm = make_desc(sb + OFF_Q, 8192, 1024);
        const uint64_t dW = make_desc(sb + OFF_W, 16, 1024), dWm = make_desc(sb + OFF_W, 8192, 1024);
        const uint64_t dD = make_desc(sb + OFF_D, 16, 1024);  // D, R, dR
        const uint64_t dDU = make_desc(sb + OFF_DU, 16, 1024), dDUm = make_desc(sb + OFF_DU, 8192, 1024);
        const uint64_t dQC = make_desc(sb + OFF_QC, 16, 1024), dQCm = make_desc(sb + OFF_QC, 8192, 1024);
        const uint64_t dU = make_desc(sb + OFF_U, 16, 1024);
        const uint64_t dDH = make_desc(sb + OFF_DH, 16, 1024), dDHm = make_desc(sb + OFF_DH, 16384, 1024);
        const uint64_t dH = make_desc(sb + OFF_H, 16, 1024);
        const uint64_t dTT = make_desc(sb + OFF_TT, 16, 1024), dTTm = make_desc(sb + OFF_TT, 8192, 1024);
        const uint64_t dDP = make_desc(sb + OFF_DP, 16, 1024), dDPm = make_desc(sb + OFF_DP, 8192, 1024);
        const uint64_t dQKm = make_desc(sb + OFF_QK, 8192, 1024), dWKm = make_desc(sb + OFF_WK, 8192, 1024);
        const uint64_t dDT = make_desc(sb + OFF_DT, 16, 1024), dDTm = make_desc(sb + OFF_DT, 8192, 1024);
        int last = -1;
        auto go = [&] { return lane == 0 && !*abort_flag; };
        named_bar(2, kAll);
        mbar_wait(&bar[BIN], 0, abort_flag, status);
        tc_fence_after();
        if (go()) {
            mma_k<128, false, true>(tb + TM_T, dK, 512, dDHm, 0, ID_64x128_KM, false);
            mma_k<128, false, false>(tb + TM_S, dQC, 512, dK, 512, ID_64x64_KK, false);
            mma_k<128, false, false>(tb + TM_P, dD, 512, dU, 512, ID_64x64_KK, false);
            mma_commit(&bar[B1]);
            mma_k<128, false, false>(tb + TM_ACC, dQ, 512, dK, 512, ID_64x64_KK, false);
            mma_k<128, false, false>(tb + TM_WK, dW, 512, dK, 512, ID_64x64_KK, false);
            mma_k<128, false, false>(tb + TM_KK, dK, 512, dK, 512, ID_64x64_KK, false);
            mma_commit(&bar[B1B]);
            last = B1B;
        }
        named_bar(3, kAll);
        tc_fence_after();
        if (go()) {
            mma_k<64, true, true>(tb + TM_T, dTTm, 0, dDUm, 0, ID_64x128_MM, false);
            mma_k<128, false, false>(tb + TM_X, dDU, 512, dD, 512, ID_64x64_KK, false);
            mma_commit(&bar[B2]);
            last = B2;
        }
        named_bar(2, kAll);
        tc_fence_after();
        if (go()) {
            mma_k<64, true, true>(tb + TM_ACC, dDPm, 0, dQCm, 0, ID_64x128_MM, false);
            mma_k<64, true, true>(tb + TM_ACC, dQKm, 0, dWm, 0, ID_64x128_MM, true);
            mma_k<64, true, true>(tb + TM_ACC, dWKm, 0, dQm, 0, ID_64x128_MM, true);
            mma_k<128, false, false>(tb + TM_S, dU, 512, dDH, 1024, ID_64x128_KK, false);
            mma_commit(&bar[B2B]);
            last = B2B;
        }
        named_bar(3, kAll);
        tc_fence_after();
        if (go()) {
            mma_k<64, true, true>(tb + TM_X, dTTm, 0, dDTm, 0, ID_64x64_MM, false);
            mma_commit(&bar[B3]);
            mma_k<128, false, false>(tb + TM_T, dD, 512, dH, 1024, ID_64x128_KK, false);
            last = B3;
        }
        // dH's last reader is done: DC + DC^T into its place
        mbar_wait(&bar[B2B], 0, abort_flag, status);
        const bool dcs = go();
        if (dcs) {
            mbar_arrive_expect_tx(&bar[BDC], 32768);
            bulk_load(sm + OFF_DH, a.dcs_img + static_cast<size_t>(ch) * 32768, 32768, &bar[BDC]);
        }
        {
            // the chunk one wave later finds its inputs in L2
            const int nx = ch + a.wave;
            if (lane == 0 && a.wave > 0 && nx < static_cast<int>(gridDim.x)) {
                const size_t nimg = static_cast<size_t>(nx) * 32768, n64 = static_cast<size_t>(nx) * kC * kD;
                prefetch_tokens(&map_k, a, nx);
                prefetch_tokens(&map_q, a, nx);
                prefetch_tokens(&map_do, a, nx);
                prefetch_tokens(&map_v, a, nx);
                bulk_prefetch_l2(a.dh_img + nimg, 32768);
                bulk_prefetch_l2(a.u + n64, kC * kD * 4);
                bulk_prefetch_l2(a.w_img + static_cast<size_t>(nx) * 16384, 16384);
                bulk_prefetch_l2(a.qc + n64 / 2, kC * kD * 2);
                bulk_prefetch_l2(a.tt + static_cast<size_t>(nx) * kC * kC, kC * kC * 4);
                bulk_prefetch_l2(a.hs_img + nimg, 32768);
                bulk_prefetch_l2(a.r + n64, kC * kD * 4);
                bulk_prefetch_l2(a.x1 + n64, kC * kD * 4);
                bulk_prefetch_l2(a.dcs_img + nimg, 32768);
            }
        }
        named_bar(2, kAll);
        tc_fence_after();
        if (go()) {
            mma_k<64, false, false>(tb + TM_X, dDP, 0, dTT, 0, ID_64x64_KK, false);
            mma_commit(&bar[B4]);
            last = B4;
        }
        named_bar(3, kAll);
        mbar_wait(&bar[BDC], 0, abort_flag, status);
        tc_fence_after();
        if (go()) {
            mma_k<64, false, true>(tb + TM_ACC, dDT, 0, dKm, 0, ID_64x128_KM, true);
            mma_k<128, false, true>(tb + TM_ACC, dK, 512, dDHm, 0, ID_64x128_KM, true);
            mma_commit(&bar[B5]);
            last = B5;
        }
        if (lane == 0 && *abort_flag) {
            mbar_drain(&bar[BTOK], 0);
            mbar_drain(&bar[BIN], 0);
            if (dcs) mbar_drain(&bar[BDC], 0);
            if (last >= 0) mbar_drain(&bar[last], 0);
        }
        __syncthreads();  // the row sums below are complete
        if (warp == kCompute / 32) {
            // dg: the in-chunk reverse cumulative sum of dgc, two tokens a lane; dbeta
            float d[2];
            float kd_all = 0.f;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int j = 2 * lane + u;
                const float rs = row_total(red + 256, j), kd = row_total(red + 512, j);
                const float prs = row_total(red + 768, j), gkh = row_total(red + 1024, j);
                kd_all += kd;
                d[u] = j < n ? be[j] * rs - cs[j] + prs - pcs[j] + vec[2 * kC + j] - kd - gkh : 0.f;
                if (j < n) a.dbeta[(static_cast<size_t>(b) * a.T + r * kC + j) * a.H + h] = db1[j] + rs;
            }
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) kd_all += __shfl_xor_sync(0xffffffffu, kd_all, o);
            // e^{gc_last} <dH, H> + sum_i kd_i at the last row
#pragma unroll
            for (int u = 0; u < 2; ++u)
                if (2 * lane + u == n - 1) d[u] += E[kC - 1] * (vec[3 * kC] + vec[3 * kC + 1]) + kd_all;
            float p = d[0] + d[1];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float y = __shfl_down_sync(0xffffffffu, p, o);
                if (lane + o < 32) p += y;
            }
            const size_t out = (static_cast<size_t>(b) * a.T + r * kC + 2 * lane) * a.H + h;
            if (2 * lane < n) a.dg[out] = p;
            if (2 * lane + 1 < n) a.dg[out + a.H] = p - d[0];
        }
        return;
    }

    // ---- the compute threads
    const int qd = warp & 3, grp = warp >> 2, hf = lane >> 4, i = 16 * qd + (lane & 15);
    const int c0 = 64 * hf + 16 * grp, s0 = 32 * hf + 8 * grp;
    if (warp == 0) tmem_alloc(tmem_slot, 512);
    grid_wait();
    float u[16], x[16];
    ld_own16(a.u + t64, tid, u);
    if (tid < kC) pcs[tid] = cs[tid] = db1[tid] = 0.f;
    put16(sm + OFF_U, i, hf, grp, u);
    {
        float t[8];
        ld_global8(a.tt + static_cast<size_t>(ch) * kC * kC + 8 * tid, t);
        *reinterpret_cast<uint4 *>(sm + OFF_TT + t64_chunk(tid >> 3, tid & 7)) = pack8(t);
    }
    __syncthreads();
    const uint32_t tb = *tmem_slot, tq = tb + (static_cast<uint32_t>(32 * qd) << 16);
    mbar_wait(&bar[BTOK], 0, abort_flag, status);
    const Raw16 kr = get16(sm + OFF_K, i, hf, grp), qr = get16(sm + OFF_Q, i, hf, grp), vr = get16(sm + OFF_QK, i, hf, grp);
    unpack16(get16(sm + OFF_D, i, hf, grp), x);
#pragma unroll
    for (int e = 0; e < 16; ++e) x[e] *= a.scale;
    put16(sm + OFF_D, i, hf, grp, x);
    {
        uint32_t w[16];
        const float rr = row_norms<true>(sm + OFF_Q, sm + OFF_K, tid, a.l2norm, w);
        if ((tid & 3) == 0) rn[tid >> 2] = rr;
    }
    compute_sync();
    const float rq = rn[i], rk = rn[kC + i];
    unpack16(qr, x);
#pragma unroll
    for (int e = 0; e < 16; ++e) x[e] *= rq;
    put16(sm + OFF_Q, i, hf, grp, x);
    unpack16(kr, x);
#pragma unroll
    for (int e = 0; e < 16; ++e) x[e] *= rk;
    put16(sm + OFF_K, i, hf, grp, x);
    signal_issue(2);
    // while round 1 runs: R, X1
    float du[16], rr[16];
    ld_global8(a.x1 + t64 + i * kD + c0, du);
    ld_global8(a.x1 + t64 + i * kD + c0 + 8, du + 8);
    ld_own16(a.r + t64, tid, rr);
    float gam[8];
    {
        const float gi = gc[i];
#pragma unroll
        for (int e = 0; e < 8; ++e) gam[e] = s0 + e <= i ? expf(gi - gc[s0 + e]) : 0.f;
    }
    const float ed = expf(gc[kC - 1] - gc[i]);
    // ---- round 1: dU, dP
    mbar_wait(&bar[B1], 0, abort_flag, status);
    tc_fence_after();
    put16(sm + OFF_D, i, hf, grp, rr);  // R in D's place
    {
        acc_ld16(tq + TM_T + 16 * grp, x);
        float part = 0.f;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            part = fmaf(u[e], ed * x[e], part);
            du[e] = fmaf(ed, x[e], du[e]);
        }
        put16(sm + OFF_DU, i, hf, grp, du);
        row_part(red + 512, grp, i, hf, part);
        float s[8], p[8];
        acc_ld8(tq + TM_S + 8 * grp, s);
        acc_ld8(tq + TM_P + 8 * grp, p);
        part = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            p[e] = s0 + e <= i ? p[e] * gam[e] : 0.f;
            s[e] *= p[e];
            part += s[e];
        }
        put8(sm + OFF_DP, i, hf, grp, p);
        signal_issue(3);
        row_part(red + 768, grp, i, hf, part);
        col_sums(s, lane);
        if (!(lane & 1)) atomicAdd(&pcs[s0 + ((lane >> 1) & 7)], s[0]);
    }
    mbar_wait(&bar[B1B], 0, abort_flag, status);
    tc_fence_after();
    {
        float s[8];
        acc_ld8(tq + TM_ACC + 8 * grp, s);
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] = s0 + e <= i ? s[e] : 0.f;
        put8(sm + OFF_QK, i, hf, grp, s);
        acc_ld8(tq + TM_WK + 8 * grp, s);
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] = s0 + e <= i ? s[e] : 0.f;
        put8(sm + OFF_WK, i, hf, grp, s);
    }
    signal_issue(2);
    // ---- round 2: dR = dv, dTb
    float tt[8];
    ld_global8(a.tt + static_cast<size_t>(ch) * kC * kC + i * kC + s0, tt);
    mbar_wait(&bar[B2], 0, abort_flag, status);
    tc_fence_after();
    {
        acc_ld16(tq + TM_T + 16 * grp, x);
        float v[16], part = 0.f;
        unpack16(vr, v);
        const float bi = be[i];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            x[e] *= bi;
            part = fmaf(v[e] - rr[e], x[e], part);
        }
        put16(sm + OFF_D, i, hf, grp, x);  // dR in R's place
        float t[8];
        acc_ld8(tq + TM_X + 8 * grp, t);
        put8(sm + OFF_DT, i, hf, grp, t);
        signal_issue(3);
        row_part(red + 1024, grp, i, hf, part);
#pragma unroll
        for (int e = 0; e < 8; ++e) t[e] *= tt[e];
        col_sums(t, lane);
        if (!(lane & 1)) atomicAdd(&db1[s0 + ((lane >> 1) & 7)], t[0]);
    }
    compute_sync();
    if (tid == 0) {  // dv is the bf16 tile of dR (signal_issue's fence came before the barrier)
        store_tokens(&map_dv, sm + OFF_D, b, h, r);
        tma_store_commit();
    }
    // ---- round 3: M2
    mbar_wait(&bar[B2B], 0, abort_flag, status);
    mbar_wait(&bar[B3], 0, abort_flag, status);
    tc_fence_after();
    {
        float m[8];
        acc_ld8(tq + TM_X + 8 * grp, m);
#pragma unroll
        for (int e = 0; e < 8; ++e) m[e] *= be[s0 + e];
        put8(sm + OFF_DP, i, hf, grp, m);
    }
    signal_issue(2);
    // ---- round 4: dKK + dKK^T
    float *stage = reinterpret_cast<float *>(sm + OFF_QC);
    mbar_wait(&bar[B4], 0, abort_flag, status);
    tc_fence_after();
    {
        float da[8], kk2[8];
        acc_ld8(tq + TM_X + 8 * grp, da);
        acc_ld8(tq + TM_KK + 8 * grp, kk2);
        float part = 0.f;
        const float bi = be[i];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int j = s0 + e;
            const float y = j < i ? -da[e] : 0.f;
            const float xx = y * gam[e] * kk2[e];
            part += xx;
            da[e] = y * bi * gam[e];  // dKK
            kk2[e] = bi * xx;
            stage[i * LS + j] = da[e];
        }
        row_part(red + 256, grp, i, hf, part);
        col_sums(kk2, lane);
        if (!(lane & 1)) atomicAdd(&cs[s0 + ((lane >> 1) & 7)], kk2[0]);
        tc_fence_before();
        compute_sync();
#pragma unroll
        for (int e = 0; e < 8; ++e) da[e] += stage[(s0 + e) * LS + i];
        put8(sm + OFF_DT, i, hf, grp, da);
    }
    signal_issue(3);
    float dmv[16];  // Dm - c G, then dk
    {
        ld_own16(a.w + t64, tid, dmv);  // G (gdn_bwd_local128_kernel)
        ld_global8(a.dm + static_cast<size_t>(ch) * kD + c0, x);
        ld_global8(a.dm + static_cast<size_t>(ch) * kD + c0 + 8, x + 8);
#pragma unroll
        for (int e = 0; e < 16; ++e) dmv[e] = x[e] - cf * dmv[e];
    }
    // ---- round 5: dk
    mbar_wait(&bar[B5], 0, abort_flag, status);
    tc_fence_after();
    {
        const float ei = E[i];
        acc_ld16(tq + TM_ACC + 16 * grp, x);
#pragma unroll
        for (int e = 0; e < 16; ++e) dmv[e] += x[e];
        acc_ld16(tq + TM_S + 16 * grp, x);
#pragma unroll
        for (int e = 0; e < 16; ++e) dmv[e] = fmaf(ed, x[e], dmv[e]);
        acc_ld16(tq + TM_T + 16 * grp, x);
#pragma unroll
        for (int e = 0; e < 16; ++e) dmv[e] = fmaf(-ei, x[e], dmv[e]);
        unpack16(kr, x);
        float part = 0.f;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            x[e] *= rk;
            part = fmaf(x[e], dmv[e], part);
        }
        row_part(red, grp, i, hf, part);
    }
    tc_fence_before();
    compute_sync();
    {
        const float rdot = a.l2norm ? row_total(red, i) : 0.f;
#pragma unroll
        for (int e = 0; e < 16; ++e) x[e] = (dmv[e] - x[e] * rdot) * rk;
        put16(sm + OFF_K, i, hf, grp, x);
        fence_proxy_async_smem();
        compute_sync();
        if (tid == 0) {
            store_tokens(&map_dk, sm + OFF_K, b, h, r);
            tma_store_commit();
            tma_store_wait_read();
        }
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tb, 512);
    }
}

// =====================================================================================
// gdn_bwd_suffix128_kernel: exclusive suffix over the chunks of a sequence and head of the increments of
// DC and Dm
// =====================================================================================
// acc = dC_T + sum_{s > r} dc[s] per element; DC_{r+1} + DC_{r+1}^T goes out as the kv kernel's bf16
// operand tile (half the bytes of the fp32 array, and no transposed reads there), the full sum is dC0.  A
// CTA walks the chunks with one pair of 32 x 32 blocks (bi, bj), (bj, bi) in registers (four elements of
// each a thread), the partner block through shared memory; loads run four chunks ahead.  HBM-bound: 96 KB a
// chunk.  The last CTA of a sequence and head does Dm.
constexpr int kSufPairs = 10, kSufAhead = 4;
__global__ void __launch_bounds__(256) gdn_bwd_suffix128_kernel(const GdnBwdArgs a) {
    __shared__ float tile[2][2][32][33];
    const int bh = blockIdx.x / (kSufPairs + 1), pr = blockIdx.x % (kSufPairs + 1), tid = threadIdx.x, NC = a.NC;
    const size_t ch0 = static_cast<size_t>(bh) * NC;
    grid_wait();
    if (pr == kSufPairs) {
        if (tid >= kD) return;
        float acc = a.dmT ? a.dmT[static_cast<size_t>(bh) * kD + tid] : 0.f;
        for (int r0 = NC - 1; r0 >= 0; r0 -= 8) {
            float x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = r0 - u >= 0 ? a.dm[(ch0 + r0 - u) * kD + tid] : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (r0 - u >= 0) {
                    a.dm[(ch0 + r0 - u) * kD + tid] = acc;
                    acc += x[u];
                }
        }
        if (a.dm0) a.dm0[static_cast<size_t>(bh) * kD + tid] = acc;
        return;
    }
    // pair pr of blocks bi <= bj: (0,0) (0,1) (0,2) (0,3) (1,1) (1,2) (1,3) (2,2) (2,3) (3,3)
    const int bi = pr < 4 ? 0 : pr < 7 ? 1 : pr < 9 ? 2 : 3;
    const int bj = pr < 4 ? pr : pr < 7 ? pr - 3 : pr < 9 ? pr - 5 : 3;
    const int y = tid >> 3, x4 = 4 * (tid & 7);
    const size_t eA = static_cast<size_t>(32 * bi + y) * kD + 32 * bj + x4;  // block (bi, bj): row y, columns x4 ..
    const size_t eB = static_cast<size_t>(32 * bj + y) * kD + 32 * bi + x4;  // block (bj, bi)
    const size_t st = static_cast<size_t>(bh) * kD * kD;
    float A[4] = {0.f, 0.f, 0.f, 0.f}, Bv[4] = {0.f, 0.f, 0.f, 0.f};
    auto ld4 = [](const float *p, float (&v)[4]) {
        const float4 f = *reinterpret_cast<const float4 *>(p);
        v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
    };
    if (a.dCT) {
        ld4(a.dCT + st + eA, A);
        ld4(a.dCT + st + eB, Bv);
    }
    float qa[kSufAhead][4], qb[kSufAhead][4];
    auto fetch = [&](int u, int r) {
        if (r < 0) return;
        ld4(a.dc + (ch0 + r) * kD * kD + eA, qa[u]);
        ld4(a.dc + (ch0 + r) * kD * kD + eB, qb[u]);
    };
#pragma unroll
    for (int u = 0; u < kSufAhead; ++u) fetch(u, NC - 1 - u);
    auto out4 = [&](int r, int row, int col, const float (&v)[4]) {
        uint8_t *img = a.dcs_img + (ch0 + r) * 32768 + (col >> 6) * 16384;
        *reinterpret_cast<uint2 *>(img + t64_offset(row, col & 63)) = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
    };
    for (int rb = NC - 1; rb >= 0; rb -= kSufAhead) {
#pragma unroll
        for (int u = 0; u < kSufAhead; ++u) {
            const int r = rb - u;
            if (r < 0) break;
            float (*tA)[33] = tile[u & 1][0], (*tB)[33] = tile[u & 1][1];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                tA[y][x4 + e] = A[e];
                tB[y][x4 + e] = Bv[e];
            }
            __syncthreads();
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = A[e] + tB[x4 + e][y];
            out4(r, 32 * bi + y, 32 * bj + x4, v);
            if (bi != bj) {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = Bv[e] + tA[x4 + e][y];
                out4(r, 32 * bj + y, 32 * bi + x4, v);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                A[e] += qa[u][e];
                Bv[e] += qb[u][e];
            }
            fetch(u, r - kSufAhead);
        }
    }
    if (a.dC0) {
        *reinterpret_cast<float4 *>(a.dC0 + st + eA) = make_float4(A[0], A[1], A[2], A[3]);
        if (bi != bj) *reinterpret_cast<float4 *>(a.dC0 + st + eB) = make_float4(Bv[0], Bv[1], Bv[2], Bv[3]);
    }
}

}  // namespace

cudaError_t launch_gdn_local128(const gbwd::GdnBwdArgs &a, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(gdn_bwd_local128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(lk::kSmem));
    if (e != cudaSuccess) return e;
    const long long chunks = static_cast<long long>(a.B) * a.H * a.NC;
    CUtensorMap q, k, v, d, dq, x1, y1, dc;
    if (!make_token_map(&q, a.q, 2, a.B, a.T, a.H, kD, 64, true) ||
        !make_token_map(&k, a.k, 2, a.B, a.T, a.H, kD, 64, true) ||
        !make_token_map(&v, a.v, 2, a.B, a.T, a.H, kD, 64, true) ||
        !make_token_map(&d, a.dout, 2, a.B, a.T, a.H, kD, 64, true) ||
        !make_token_map(&dq, a.dq, 2, a.B, a.T, a.H, kD, 64, true) ||
        !make_f32_rows_map(&x1, a.x1, chunks * kC, kD, 32, kC) ||
        !make_f32_rows_map(&y1, a.y1, chunks * kD, kD, 32, kD) || !make_f32_rows_map(&dc, a.dc, chunks * kD, kD, 32, kD))
        return cudaErrorInvalidValue;
    return launch_after(gdn_bwd_local128_kernel, static_cast<unsigned>(chunks), kAll, lk::kSmem, s, q, k, v, d, dq, x1, y1,
                        dc, a);
}

cudaError_t launch_gdn_suffix128(const gbwd::GdnBwdArgs &a, cudaStream_t s) {
    return launch_after(gdn_bwd_suffix128_kernel, static_cast<unsigned>(a.B * a.H * (kSufPairs + 1)), 256, 0, s, a);
}

cudaError_t launch_gdn_kv128(const gbwd::GdnBwdArgs &a, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(gdn_bwd_kv128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kk::kSmem));
    if (e != cudaSuccess) return e;
    CUtensorMap q, k, v, d, dv, dk;
    if (!make_token_map(&q, a.q, 2, a.B, a.T, a.H, kD, 64, true) ||
        !make_token_map(&k, a.k, 2, a.B, a.T, a.H, kD, 64, true) ||
        !make_token_map(&v, a.v, 2, a.B, a.T, a.H, kD, 64, true) ||
        !make_token_map(&d, a.dout, 2, a.B, a.T, a.H, kD, 64, true) ||
        !make_token_map(&dv, a.dv, 2, a.B, a.T, a.H, kD, 64, true) ||
        !make_token_map(&dk, a.dk, 2, a.B, a.T, a.H, kD, 64, true))
        return cudaErrorInvalidValue;
    return launch_after(gdn_bwd_kv128_kernel, static_cast<unsigned>(a.B * a.H * a.NC), kAll, kk::kSmem, s, q, k, v, d, dv,
                        dk, a);
}

}  // namespace ccq
