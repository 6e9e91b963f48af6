// ccq_gdn_segment.cu -- sequence-segment parallelism for long CCQ-Gated-DeltaNet sequences.
//
// With few (batch, head) sequences, each sequence is cut into `nseg` segments of whole
// chunks, as for CCQ-GLA (ccq_gla_segment.cu).  The gated delta state is affine in the
// state entering a chunk: with H = S^T [Dk][Dv], Tb = Tt diag(beta) and the chunk factors
// of ccq_gdn_chunk.cu,
//   H_{r+1} = A_r H_r + B_r,   A_r = e^{gC} I - Kd^T Tb Ke,   Ke = Diag(e^{gc}) Kbar,
//   Kd = Diag(e^{gC - gc}) Kbar,   B_r = Kd^T Tb V,
// every factor an exponential of a non-positive argument, so a segment maps its entering
// state H to P H + Q, with P the product of its A_r and Q the state it reaches from zero.
// The covariance C and key sum m are plain sums.  Three launches replace the long walk:
//   1. gdn_segment_state_kernel: per (sequence, segment), from a zero state, Q, P, dC, dm.
//      P is updated exactly like the state without its V term, so one set of products
//      serves both: with Z = [Q | P] (Dk x 2Dv),
//        Y^T = Z^T Ke^T,  R^T = [V^T - Y_Q^T | -Y_P^T],  U^T = R^T Tb^T,
//        [Q | P] = e^{gC} [Q | P] + Kd^T U
//      (M = 128 products over the transposed operands, so everything fits 512 TMEM columns).
//      Eight warps (EPI) carry the chain of a chunk -- Z, Y, R, U, the update -- and eight more (PREP) the next
//      chunk's factors beside it: kbar and Ke once Y of this chunk has read Ke, Kd once the update has read
//      Kd.  What bounds it is EPI's chain of four products and their epilogues; with one set of warps
//      doing the preparation in turn a chunk took 8.4 K cycles, now 7.0 K.
//   2. gdn_segment_combine_kernel: per (sequence, 16 state columns), H_{s+1} = P_s H_s + Q_s,
//      C and m by prefix sums, in fp32; each slot then holds its segment's entering states.
//   3. gdn_chunk_kernel with one CTA per (sequence, segment) (ccq_gdn_chunk.cu).
// Workspace per (sequence, segment): kGdnSegFloats floats -- S (Q, then the entering H),
// P, C (dC, then the entering C), m (dm, then the entering m), and 128 spare.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ccq_internal.h"
#include "sm100_ptx.cuh"

namespace ccq {

namespace {

constexpr int kC = 64;
constexpr int kD = 128;
constexpr int kEpi = 256, kPrep = 256, kThreads = kEpi + kPrep;
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kSS = kD * kD;

// shared memory: two slots of {k 16K, v 16K, Tb 8K}, then Ke, Kd, Z, R/U and scratch
constexpr uint32_t SL_BYTES = 40960;
constexpr uint32_t SL_K = 0, SL_V = 16384, SL_TB = 32768;
constexpr uint32_t OFF_KE = 81920;    // 16K  e^{gc} kbar (K-major B of Y^T)
constexpr uint32_t OFF_KD = 98304;    // 16K  e^{gC - gc} kbar (MN-major A of the state update)
constexpr uint32_t OFF_Z = 114688;    // 64K  bf16 [Q | P], [128 rows][256 cols] as four T64 tiles
constexpr uint32_t OFF_RU = 180224;   // 32K  bf16 R^T, then U^T: [256 rows][64 cols] as two T64 tiles
constexpr uint32_t OFF_MISC = 212992;
constexpr uint32_t M_GC = 0;      // [64] cumulative log decay
constexpr uint32_t M_EP = 256;    // [64] e^{gc}
constexpr uint32_t M_EN = 512;    // [64] e^{gC - gc}
constexpr uint32_t M_RK = 768;    // [64] 1/|k|
constexpr uint32_t M_DMP = 1024;  // [4][128] key-sum quarters
constexpr uint32_t M_HS = 3072;   // [2] e^{gC} of the chunk, by parity
constexpr uint32_t M_BAR = 3080;
enum { BAR_IN0 = 0, BAR_IN1, BAR_Y, BAR_U, BAR_S, BAR_PA, BAR_PB, kBars };  // inputs, products, PREP's two parts
constexpr uint32_t M_TMEM = M_BAR + 8 * kBars, M_ABORT = M_TMEM + 4;
constexpr uint32_t kSmem = OFF_MISC + 4096 + 1024;
static_assert(kSmem <= 232448, "smem");

// TMEM columns
constexpr uint32_t TM_X = 0, TM_PT = 128, TM_DC = 256, TM_YU = 384;  // Q, P, dC, Y^T / U^T

constexpr uint32_t ID_Y = make_idesc(128, 64, 1, 0);     // Y^T = Z^T Ke^T
constexpr uint32_t ID_U = make_idesc(128, 64, 0, 0);     // U^T = R^T Tb^T
constexpr uint32_t ID_ST = make_idesc(128, 256, 1, 0);   // [Q | P] += Kd^T U
constexpr uint32_t ID_DC = make_idesc(128, 128, 1, 1);   // dC += Kbar^T Kbar

__device__ __forceinline__ void store_row_chunk(uint8_t *tile, int row, int chunk, const float *w) {
    uint4 u;
    u.x = pack_bf16(w[0], w[1]);
    u.y = pack_bf16(w[2], w[3]);
    u.z = pack_bf16(w[4], w[5]);
    u.w = pack_bf16(w[6], w[7]);
    *reinterpret_cast<uint4 *>(tile + t64_chunk(row, chunk)) = u;
}

__global__ void __launch_bounds__(kThreads, 1)
gdn_segment_state_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                         const __grid_constant__ CUtensorMap map_tb, const ChunkArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = smem_align1024(smem_raw);
    const uint32_t sb = smem_addr(sm);
    uint8_t *misc = sm + OFF_MISC;
    float *gc = reinterpret_cast<float *>(misc + M_GC);
    float *epv = reinterpret_cast<float *>(misc + M_EP);
    float *env = reinterpret_cast<float *>(misc + M_EN);
    float *rkv = reinterpret_cast<float *>(misc + M_RK);
    float *dmp = reinterpret_cast<float *>(misc + M_DMP);
    float *hsv = reinterpret_cast<float *>(misc + M_HS);
    uint64_t *bar = reinterpret_cast<uint64_t *>(misc + M_BAR);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(misc + M_TMEM);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(misc + M_ABORT);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int seq = blockIdx.x / a.nst, seg = blockIdx.x % a.nst;
    const int b = seq / a.H, h = seq % a.H;
    const int T = a.T, H = a.H;
    const int NCt = (T + kC - 1) / kC;
    const int cb = seg * a.st_chunks;
    const int n = min(a.st_chunks, a.seg_chunks * (a.nseg - 1) - cb);  // chunks of this segment (>= 1)
    const int wrow0 = seq * NCt * kC;                 // first Tb row of this sequence
    int *status = a.status;

    if (tid == 0) {
        for (int i = 0; i < kBars; ++i) mbar_init(&bar[i], 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 0) tmem_alloc(tslot, 512);
    grid_wait();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *tslot;
    const uint32_t tq = tbase + (static_cast<uint32_t>(32 * (warp & 3)) << 16);
    auto issue_in = [&](int r) {  // k, v, Tb of local chunk r into slot r & 1
        const int s = r & 1, tg = (cb + r) * kC;
        uint8_t *base = sm + s * SL_BYTES;
        mbar_arrive_expect_tx(&bar[s], 5 * 8192);
        tma_load_4d(base + SL_K, &map_k, &bar[s], 0, h, tg, b);
        tma_load_4d(base + SL_K + 8192, &map_k, &bar[s], 64, h, tg, b);
        tma_load_4d(base + SL_V, &map_v, &bar[s], 0, h, tg, b);
        tma_load_4d(base + SL_V + 8192, &map_v, &bar[s], 64, h, tg, b);
        tma_load_2d(base + SL_TB, &map_tb, &bar[s], 0, wrow0 + (cb + r) * kC);
    };
    float *out = a.seg_ws + (static_cast<size_t>(seq) * a.nseg + seg) * kGdnSegFloats;

    if (warp >= kEpi / 32) {
        // =============================================================== PREP
        const int pt = tid - kEpi;
        if (pt == 0) {
            tma_prefetch_desc(&map_k);
            tma_prefetch_desc(&map_v);
            tma_prefetch_desc(&map_tb);
            issue_in(0);
        }
        int issued = 1;  // chunks whose loads were issued
        float g_reg = 0.f;
        if (pt < 64) {
            const int t = cb * kC + pt;
            g_reg = t < T ? a.g[(static_cast<size_t>(b) * T + t) * H + h] : 0.f;
        }
        float dm_acc = 0.f;  // key sum of dim pt (pt < 128)
        for (int r = 0; r < n; ++r) {
            const int s = r & 1;
            uint8_t *slot = sm + s * SL_BYTES;
            // cumulative decay, factors, norms; then kbar and Ke (whose last reader is Y of chunk r - 1), Kd
            // (the update of chunk r - 1), key sum
            if (pt < 64) {
                gc[pt] = g_reg;
                const int t = (cb + r + 1) * kC + pt;
                g_reg = t < T ? a.g[(static_cast<size_t>(b) * T + t) * H + h] : 0.f;
            }
            mbar_wait(&bar[BAR_IN0 + s], (r >> 1) & 1, abort_flag, status);
            named_bar(2, kPrep);
            if (pt < 32) {
                const float x0 = gc[2 * lane], x1 = gc[2 * lane + 1];
                float pv = x0 + x1;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float y = __shfl_up_sync(0xffffffffu, pv, o);
                    if (lane >= o) pv += y;
                }
                gc[2 * lane] = pv - x1;
                gc[2 * lane + 1] = pv;
            }
            // row norms: thread = (row j, column quarter)
            const int j = pt >> 2, qq = pt & 3;
            uint8_t *kq = slot + SL_K + (qq >> 1) * 8192;
            uint4 kv[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) kv[c] = *reinterpret_cast<const uint4 *>(kq + t64_chunk(j, 4 * (qq & 1) + c));
            {
                uint64_t s0 = 0, s1 = 0;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint64_t p0 = f2_from_bf16x2(kv[c].x), p1 = f2_from_bf16x2(kv[c].y),
                                   p2 = f2_from_bf16x2(kv[c].z), p3 = f2_from_bf16x2(kv[c].w);
                    s0 = f2_fma(p0, p0, s0); s1 = f2_fma(p1, p1, s1);
                    s0 = f2_fma(p2, p2, s0); s1 = f2_fma(p3, p3, s1);
                }
                const float2 sv = f2_split(f2_add(s0, s1));
                float ss = sv.x + sv.y;
                ss += __shfl_xor_sync(0xffffffffu, ss, 1);
                ss += __shfl_xor_sync(0xffffffffu, ss, 2);
                if (qq == 0) rkv[j] = a.l2norm ? rsqrtf(fmaxf(ss, 1e-12f)) : 1.f;
            }
            named_bar(2, kPrep);  // gc, rk visible
            const float gC = gc[63];
            if (pt < 64) {
                epv[pt] = fast_exp2(gc[pt] * kLog2e);         // e^{gc} <= 1
                env[pt] = fast_exp2((gC - gc[pt]) * kLog2e);  // e^{gC - gc} <= 1
                if (pt == 0) hsv[s] = fast_exp2(gC * kLog2e);
            }
            named_bar(2, kPrep);  // factors visible
            const float rk = rkv[j];
            const uint64_t rk2 = f2_make(rk, rk), ep2 = f2_make(epv[j], epv[j]), en2 = f2_make(env[j], env[j]);
            if (r > 0) mbar_wait(&bar[BAR_Y], (r - 1) & 1, abort_flag, status);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t w[4] = {kv[c].x, kv[c].y, kv[c].z, kv[c].w};
                uint32_t ob[4], oe[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint64_t kb = f2_mul(f2_from_bf16x2(w[u]), rk2);
                    ob[u] = bf16x2_from_f2(kb);
                    oe[u] = bf16x2_from_f2(f2_mul(kb, ep2));
                }
                const uint32_t off = (qq >> 1) * 8192 + t64_chunk(j, 4 * (qq & 1) + c);
                *reinterpret_cast<uint4 *>(slot + SL_K + off) = make_uint4(ob[0], ob[1], ob[2], ob[3]);
                *reinterpret_cast<uint4 *>(sm + OFF_KE + off) = make_uint4(oe[0], oe[1], oe[2], oe[3]);
            }
            fence_proxy_async_smem();
            named_bar(2, kPrep);  // kbar, Ke written
            if (pt == 0) mbar_arrive(&bar[BAR_PA]);
            // key sum: thread = (dim pair, token quarter)
            {
                const int p = pt & 63, tq4 = pt >> 6, d0 = 2 * p;
                const uint8_t *kt = slot + SL_K + (d0 >> 6) * 8192;
                uint64_t acc = 0;
#pragma unroll
                for (int u = 0; u < 16; ++u)
                    acc = f2_add(acc, f2_from_bf16x2(*reinterpret_cast<const uint32_t *>(kt + t64_offset(16 * tq4 + u, d0 & 63))));
                const float2 sv = f2_split(acc);
                dmp[tq4 * kD + d0] = sv.x;
                dmp[tq4 * kD + d0 + 1] = sv.y;
            }
            if (r > 0) mbar_wait(&bar[BAR_S], (r - 1) & 1, abort_flag, status);
            // the update of chunk r - 1 has run: its slot is free too
            if (pt == 0 && r + 1 < n && !*abort_flag) {
                issue_in(r + 1);
                issued = r + 2;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t w[4] = {kv[c].x, kv[c].y, kv[c].z, kv[c].w};
                uint32_t od[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    od[u] = bf16x2_from_f2(f2_mul(f2_mul(f2_from_bf16x2(w[u]), rk2), en2));
                *reinterpret_cast<uint4 *>(sm + OFF_KD + (qq >> 1) * 8192 + t64_chunk(j, 4 * (qq & 1) + c)) =
                    make_uint4(od[0], od[1], od[2], od[3]);
            }
            fence_proxy_async_smem();
            named_bar(2, kPrep);  // Kd, the key-sum quarters written
            if (pt == 0) mbar_arrive(&bar[BAR_PB]);
            if (pt < kD) dm_acc += (dmp[pt] + dmp[kD + pt]) + (dmp[2 * kD + pt] + dmp[3 * kD + pt]);
        }
        if (pt < kD) out[3 * kSS + pt] = dm_acc;
        if (pt == 0 && *abort_flag)  // after a give-up, wait (bounded) for the loads still in flight
            for (int r = issued > 2 ? issued - 2 : 0; r < issued; ++r) mbar_drain(&bar[BAR_IN0 + (r & 1)], (r >> 1) & 1);
    } else {
        // =============================================================== EPI
        const int hz = warp >> 2;                // column half of the state pair / of R^T, U^T
        const int row = 32 * (warp & 3) + lane;  // TMEM lane: state row a, or R^T / U^T row d
        // Q = 0, P = I, dC = 0 (this thread: row `row`, the 128 columns of half hz)
        {
            float x[32];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
#pragma unroll
                for (int e = 0; e < 32; ++e) x[e] = (hz == 1 && 32 * c + e == row) ? 1.f : 0.f;
                tmem_st32(tq + (hz ? TM_PT : TM_X) + 32 * c, x);
#pragma unroll
                for (int e = 0; e < 32; ++e) x[e] = 0.f;
                if (hz == 0) tmem_st32(tq + TM_DC + 32 * c, x);
            }
            tmem_wait_st();
        }
        tc_fence_before();
        for (int r = 0; r < n; ++r) {
            const int s = r & 1, par = r & 1;
            uint8_t *slot = sm + s * SL_BYTES;
            // ---- Z = [Q | P] as bf16; the TMEM copies scaled by e^{gC}, onto which the state
            // update of this chunk accumulates
            if (r > 0) mbar_wait(&bar[BAR_S], (r - 1) & 1, abort_flag, status);
            mbar_wait(&bar[BAR_PA], par, abort_flag, status);
            tc_fence_after();
            {
                const float hs = hsv[s];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float x[32];
                    tmem_ld32(tq + (hz ? TM_PT : TM_X) + 32 * c, x);
                    uint8_t *tile = sm + OFF_Z + (2 * hz + (c >> 1)) * 16384;
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4) store_row_chunk(tile, row, 4 * (c & 1) + q4, x + 8 * q4);
#pragma unroll
                    for (int e = 0; e < 32; ++e) x[e] *= hs;
                    tmem_st32(tq + (hz ? TM_PT : TM_X) + 32 * c, x);
                }
                tmem_wait_st();
            }
            fence_proxy_async_smem();
            tc_fence_before();
            named_bar(1, kEpi);  // Z written
            // ---- Y^T = Z^T Ke^T (two M = 128 halves, N = 64 tokens, K = 128); dC += Kbar^T Kbar
            if (tid == 0 && !*abort_flag) {
                tc_fence_after();
                const uint64_t dKe = make_desc(sb + OFF_KE, 16, 1024);
                for (int half = 0; half < 2; ++half) {
                    const uint64_t dZ = make_desc(sb + OFF_Z + half * 32768, 16384, 1024);
                    for (int k = 0; k < 8; ++k)
                        mma_bf16(tbase + TM_YU + 64 * half, dZ + k * 128, dKe + (k >> 2) * 512 + (k & 3) * 2, ID_Y,
                                 k != 0);
                }
                mma_commit(&bar[BAR_Y]);
                const uint64_t dKm = make_desc(sb + s * SL_BYTES + SL_K, 8192, 1024);
                for (int k = 0; k < 4; ++k) mma_bf16(tbase + TM_DC, dKm + k * 128, dKm + k * 128, ID_DC, 1);
            }
            mbar_wait(&bar[BAR_Y], par, abort_flag, status);
            tc_fence_after();
            // ---- R^T: [V^T - Y_Q^T | -Y_P^T], this thread row d = `row` of half hz
            {
                const uint8_t *vt = slot + SL_V + (row >> 6) * 8192;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    float y[32];
                    tmem_ld32(tq + TM_YU + 64 * hz + 32 * c, y);
                    if (hz == 0) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) {
                            const float vv = __bfloat162float(
                                *reinterpret_cast<const __nv_bfloat16 *>(vt + t64_offset(32 * c + e, row & 63)));
                            y[e] = vv - y[e];
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e) y[e] = -y[e];
                    }
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4) store_row_chunk(sm + OFF_RU + hz * 16384, row, 4 * c + q4, y + 8 * q4);
                }
            }
            fence_proxy_async_smem();
            tc_fence_before();
            named_bar(1, kEpi);
            // ---- U^T = R^T Tb^T (two halves, N = 64 tokens, K = 64 tokens)
            if (tid == 0 && !*abort_flag) {
                tc_fence_after();
                const uint64_t dTb = make_desc(sb + s * SL_BYTES + SL_TB, 16, 1024);
                for (int half = 0; half < 2; ++half) {
                    const uint64_t dR = make_desc(sb + OFF_RU + half * 16384, 16, 1024);
                    for (int k = 0; k < 4; ++k) mma_bf16(tbase + TM_YU + 64 * half, dR + k * 2, dTb + k * 2, ID_U, k != 0);
                }
                mma_commit(&bar[BAR_U]);
            }
            mbar_wait(&bar[BAR_U], par, abort_flag, status);
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                float y[32];
                tmem_ld32(tq + TM_YU + 64 * hz + 32 * c, y);
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) store_row_chunk(sm + OFF_RU + hz * 16384, row, 4 * c + q4, y + 8 * q4);
            }
            fence_proxy_async_smem();
            tc_fence_before();
            named_bar(1, kEpi);
            // ---- [Q | P] += Kd^T U (N = 256: U^T rows 0..255 across both tiles)
            if (tid == 0) {
                mbar_wait(&bar[BAR_PB], par, abort_flag, status);
                if (!*abort_flag) {
                    tc_fence_after();
                    const uint64_t dKDm = make_desc(sb + OFF_KD, 8192, 1024);
                    const uint64_t dU = make_desc(sb + OFF_RU, 16, 1024);
                    for (int k = 0; k < 4; ++k) mma_bf16(tbase + TM_X, dKDm + k * 128, dU + k * 2, ID_ST, 1);
                    mma_commit(&bar[BAR_S]);
                }
            }
        }
        // ---- outputs: Q, P, dC
        if (n > 0) mbar_wait(&bar[BAR_S], (n - 1) & 1, abort_flag, status);
        tc_fence_after();
        {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float x[32];
                tmem_ld32(tq + (hz ? TM_PT : TM_X) + 32 * c, x);
                float4 *dst = reinterpret_cast<float4 *>(out + hz * kSS + row * kD + 32 * c);
#pragma unroll
                for (int e = 0; e < 8; ++e) dst[e] = make_float4(x[4 * e], x[4 * e + 1], x[4 * e + 2], x[4 * e + 3]);
                if (hz == 0) {
                    tmem_ld32(tq + TM_DC + 32 * c, x);
                    float4 *dc = reinterpret_cast<float4 *>(out + 2 * kSS + row * kD + 32 * c);
#pragma unroll
                    for (int e = 0; e < 8; ++e) dc[e] = make_float4(x[4 * e], x[4 * e + 1], x[4 * e + 2], x[4 * e + 3]);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tbase, 512);
    }
}

// Per (sequence, block of 16 state columns): walks the segments, replacing each slot's
// S (Q), C (dC) and m (dm) with the states entering that segment:
//   H_{s+1} = P_s H_s + Q_s,  C_{s+1} = C_s + dC_s,  m_{s+1} = m_s + dm_s.
// P_s passes through shared memory in halves of 64 columns, two buffers filled by cp.async a half ahead (rows
// padded to kPS floats: the reads of eight rows at a time hit 32 banks); Q and dC of segment s+1 are in flight
// while segment s computes.  What bounds it is the latency of a step -- 64 KB of P a CTA from L2 and 128 x 128 x 16
// multiply-adds -- so two CTAs share an SM.  B = 2, H = 16, three steps: 26.2 us (P a step ahead in registers and
// one CTA an SM: two rounds of CTAs, 28.6 us).
constexpr int kCols = 16;
constexpr int kPS = 64 + 4;
constexpr int kCombineSmem = (2 * kD * kPS + 2 * kD * kCols) * 4;

__global__ void __launch_bounds__(256, 2)
gdn_segment_combine_kernel(const ChunkArgs a) {
    extern __shared__ float csm[];
    float *Ps = csm;                   // [2][128][kPS]
    float *hs = csm + 2 * kD * kPS;    // [2][128][16] the entering H, by the step's parity
    grid_wait();
    const int nblk = kD / kCols;
    const int seq = blockIdx.x / nblk, cblk = blockIdx.x % nblk;
    const size_t sq = static_cast<size_t>(seq);
    const int tid = threadIdx.x;
    // rows arow, arow + 64 and four columns a thread: a warp's reads of P are eight rows, of H four 16-byte
    // pieces of a row, six wavefronts per four reduction steps (one row and eight columns took ten)
    const int arow = tid >> 2, cl = 4 * (tid & 3), c0 = kCols * cblk + cl;
    float hreg[8], creg[8];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const size_t e = sq * kSS + static_cast<size_t>(arow + 64 * u) * kD + c0;
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 hv = a.S0 ? *reinterpret_cast<const float4 *>(a.S0 + e) : z;
        const float4 cv = a.C0 ? *reinterpret_cast<const float4 *>(a.C0 + e) : z;
        hreg[4 * u] = hv.x; hreg[4 * u + 1] = hv.y; hreg[4 * u + 2] = hv.z; hreg[4 * u + 3] = hv.w;
        creg[4 * u] = cv.x; creg[4 * u + 1] = cv.y; creg[4 * u + 2] = cv.z; creg[4 * u + 3] = cv.w;
    }
    float mreg = (cblk == 0 && tid < kD) ? (a.m0 ? a.m0[sq * kD + tid] : 0.f) : 0.f;
    auto slot_of = [&](int s) { return a.seg_ws + (sq * a.nseg + s) * kGdnSegFloats; };
    // half hf of P_s into buffer hf
    auto load_half = [&](int s, int hf) {
        const float *P = slot_of(s) + kSS + 64 * hf;
        float *dst = Ps + hf * kD * kPS;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int it = tid + 256 * u, rw = it >> 4, cc = it & 15;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst + rw * kPS + 4 * cc)),
                         "l"(P + rw * kD + 4 * cc)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float4 qv[2], dv[2];
    auto load_next = [&](int s) {
        const float *slot = slot_of(s);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            qv[u] = *reinterpret_cast<const float4 *>(slot + (arow + 64 * u) * kD + c0);
            dv[u] = *reinterpret_cast<const float4 *>(slot + 2 * kSS + (arow + 64 * u) * kD + c0);
        }
    };
    // the states entering segment s, over what the state pass left in its slot
    auto entering = [&](int s) {
        float *slot = slot_of(s);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            *reinterpret_cast<float4 *>(slot + (arow + 64 * u) * kD + c0) =
                make_float4(hreg[4 * u], hreg[4 * u + 1], hreg[4 * u + 2], hreg[4 * u + 3]);
            *reinterpret_cast<float4 *>(slot + 2 * kSS + (arow + 64 * u) * kD + c0) =
                make_float4(creg[4 * u], creg[4 * u + 1], creg[4 * u + 2], creg[4 * u + 3]);
        }
        if (cblk == 0 && tid < kD) slot[3 * kSS + tid] = mreg;
    };
    load_half(0, 0);
    load_half(0, 1);
    load_next(0);
    for (int s = 0; s < a.nst; ++s) {
        float *hcur = hs + (s & 1) * kD * kCols;
#pragma unroll
        for (int u = 0; u < 2; ++u)
            *reinterpret_cast<float4 *>(hcur + (arow + 64 * u) * kCols + cl) =
                make_float4(hreg[4 * u], hreg[4 * u + 1], hreg[4 * u + 2], hreg[4 * u + 3]);
        float acc[8] = {qv[0].x, qv[0].y, qv[0].z, qv[0].w, qv[1].x, qv[1].y, qv[1].z, qv[1].w};  // Q_s
        const float dcv[8] = {dv[0].x, dv[0].y, dv[0].z, dv[0].w, dv[1].x, dv[1].y, dv[1].z, dv[1].w};
        if (s + 1 < a.nst) load_next(s + 1);
        const float dm = cblk == 0 && tid < kD ? slot_of(s)[3 * kSS + tid] : 0.f;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            // at most the half after this one in flight
            if (hf == 0 || s + 1 < a.nst) asm volatile("cp.async.wait_group 1;" ::: "memory");
            else asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            const float *P = Ps + hf * kD * kPS + arow * kPS;
#pragma unroll 4
            for (int bb = 0; bb < 64; bb += 4) {
                float pw[2][4];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float4 p4 = *reinterpret_cast<const float4 *>(P + 64 * u * kPS + bb);
                    pw[u][0] = p4.x; pw[u][1] = p4.y; pw[u][2] = p4.z; pw[u][3] = p4.w;
                }
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const float4 h4 = *reinterpret_cast<const float4 *>(hcur + (64 * hf + bb + t) * kCols + cl);
                    const float hv[4] = {h4.x, h4.y, h4.z, h4.w};
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc[u] = fmaf(pw[u >> 2][t], hv[u & 3], acc[u]);
                }
            }
            if (s + 1 < a.nst) {
                __syncthreads();  // the buffer has been read
                load_half(s + 1, hf);
            }
        }
        // (with halves of one chunk segment, nst = nseg = 2, the second half starts no segment)
        if (s == 0 || a.nst < a.nseg) entering(s);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            hreg[u] = acc[u];
            creg[u] += dcv[u];
        }
        mreg += dm;
    }
    entering(a.nseg - 1);
}

}  // namespace

cudaError_t launch_gdn_segments(const ChunkArgs &args, const GdnMaps &m, cudaStream_t s) {
    ChunkArgs a = args;
    state_segments(a);
    cudaError_t e = launch_gdn_wy(a, m, s);
    if (e != cudaSuccess) return e;
    static bool attr_set = false;
    if (!attr_set) {
        e = cudaFuncSetAttribute(gdn_segment_state_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(kSmem));
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    e = launch_after(gdn_segment_state_kernel, a.B * a.H * a.nst, kThreads, kSmem, s, m.k, m.v, m.tb, a);
    if (e != cudaSuccess) return e;
    static bool attr_combine = false;
    if (!attr_combine) {
        e = cudaFuncSetAttribute(gdn_segment_combine_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kCombineSmem);
        if (e != cudaSuccess) return e;
        attr_combine = true;
    }
    e = launch_after(gdn_segment_combine_kernel, a.B * a.H * (kD / kCols), 256, kCombineSmem, s, a);
    if (e != cudaSuccess) return e;
    return launch_gdn_chunk_only(a, m, s);
}

}  // namespace ccq
