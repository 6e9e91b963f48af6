// ccq_recurrent_block.cu -- the fp32 CCQ forward over a token sequence, 32 tokens at a time.
//
// Serves what the chunkwise tensor-core kernels do not: fp32 inputs, Dk = Dv = 64, algo RECURRENT (any gate
// strength).  The backbone state S is walked token by token, as Algorithm 2 writes it (its decays are applied
// one by one, so there is no gate range); everything of the CCQ read that does not depend on S is formed for 32
// tokens at once, since C and m enter only through the queries:
//   q_clean_t = qbar_t - lambda_t (C_t qbar_t / t - m_t (m_t . qbar_t) / t^2),
//   C_t qbar_t = C qbar_t + sum_{j <= t in block} (kbar_j . qbar_t) kbar_j,  m_t . qbar_t likewise,
// with C, m the sums entering the block (App. B with a 32-token block).
//
// Layout: a cluster of NS CTAs (256 threads each) per (batch, head).  CTA s owns Dk / NS rows of C (shared
// memory) and Dv / NS columns of S (registers); it forms the key-query scores of 32 / NS tokens and the
// q_clean columns of its rows of C, and hands both to the other CTAs through distributed shared memory, so a
// block costs two cluster barriers.  In the walk of S a column belongs to 256 NS / Dv neighbouring threads,
// which share its rows: per token a thread reads its rows of alpha, kbar, q_clean from shared memory, and
// the column's output (and, for the delta rule, kbar^T S) is a shuffle sum inside the warp -- no barrier.
// The next block's inputs are in flight during the walk.
//
// What bounds it: latency, over a block's stages one after the other -- norms, scores, queries, the sum of C, two
// cluster barriers -- with a CTA's eight warps alone on an SM, and only last the walk's chain of a token (shared-memory
// reads, multiply-adds, shuffles).  GLA, d = 64, eight CTAs a sequence: a block of 32 tokens takes 5.3 us, of which the
// walk is 1.4 (a block of two tokens takes that much less); the delta rule 8.4 and 4.6.  fp32, d = 64, B = 1, H = 2,
// T = 256: 47 us, where the token-by-token kernel (six block barriers and a global load a token, one CTA per (batch,
// head)) takes 277.  Short sequences stay with that kernel (recurrent_block_pays()).
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>

#include "ccq_internal.h"

namespace ccq {

namespace {

namespace cg = cooperative_groups;

constexpr int kL = 32;         // tokens a block
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Four consecutive values at element index e of a bf16 (code 0) or fp32 tensor.
__device__ __forceinline__ float4 load4(const void *p, size_t e, int dtype) {
    if (dtype == 0) {
        const uint2 u = *reinterpret_cast<const uint2 *>(static_cast<const __nv_bfloat16 *>(p) + e);
        return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                           __uint_as_float(u.y & 0xffff0000u));
    }
    return *reinterpret_cast<const float4 *>(static_cast<const float *>(p) + e);
}

template <int D, int NS>
struct Shape {
    static constexpr int DS = D / NS;           // rows of C, columns of S of a CTA
    static constexpr int TPC = kThreads / DS;   // threads a column of S
    static constexpr int RPT = D / TPC;         // rows of S a thread
    static constexpr int V = RPT < 4 ? RPT : 4; // consecutive rows a thread
    static constexpr int NV = RPT / V;
    static constexpr int LT = kL / NS;          // tokens whose scores a CTA forms
    static constexpr int LD = D + 4;            // row stride of qbar, kbar, q_clean (16-byte accesses of a row a lane)
    static constexpr int NQ = kL * D / 4 / kThreads;
    static constexpr int NVV = (kL * DS / 4 + kThreads - 1) / kThreads;
    static constexpr int F_Q = 0, F_K = F_Q + kL * LD, F_A = F_K + kL * LD, F_QC = F_A + kL * D, F_V = F_QC + kL * LD,
                         F_C = F_V + kL * DS, F_SC = F_C + DS * D, F_M = F_SC + kL * (kL + 1), F_CQ = F_M + D,
                         F_LAM = F_CQ + kL, F_G = F_LAM + kL, F_B = F_G + kL, F_QK = F_B + kL, kFloats = F_QK + kL;
    static_assert(TPC >= 2 && TPC <= 32 && RPT >= 2, "a column's threads share a warp");
    static_assert(kFloats * 4 <= 232448, "exceeds the 227 KB per-CTA limit");
};

template <int N>
__device__ __forceinline__ void ldv(const float *p, float (&r)[N]) {
    if constexpr (N == 4) {
        const float4 x = *reinterpret_cast<const float4 *>(p);
        r[0] = x.x; r[1] = x.y; r[2] = x.z; r[3] = x.w;
    } else {
        static_assert(N == 2, "two or four values");
        const float2 x = *reinterpret_cast<const float2 *>(p);
        r[0] = x.x; r[1] = x.y;
    }
}

template <int D, int BB, int NS>
__global__ void __launch_bounds__(kThreads, 1) recurrent_block_kernel(const RecurrentArgs a) {
    using P = Shape<D, NS>;
    constexpr int DS = P::DS, LD = P::LD;
    extern __shared__ float4 rb_smem4[];
    float *sm = reinterpret_cast<float *>(rb_smem4);
    float *qn = sm + P::F_Q, *kn = sm + P::F_K, *al = sm + P::F_A, *qc = sm + P::F_QC, *vs = sm + P::F_V;
    float *C = sm + P::F_C, *sc = sm + P::F_SC, *m = sm + P::F_M, *cq = sm + P::F_CQ, *lam = sm + P::F_LAM;
    float *gs = sm + P::F_G, *be = sm + P::F_B, *qk = sm + P::F_QK;
    constexpr int LSC = kL + 1;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bh = blockIdx.x / NS, s = blockIdx.x % NS, b = bh / a.H, h = bh % a.H;
    const size_t base = static_cast<size_t>(bh);
    const int d0 = s * DS;  // first row of C / column of S of this CTA
    auto sync_cluster = [&] {
        if constexpr (NS > 1) cg::this_cluster().sync();
        else __syncthreads();
    };
    // an element of the same shared array in CTA r of the cluster
    auto peer = [&](float *p, int r) -> float * {
        if constexpr (NS > 1) return cg::this_cluster().map_shared_rank(p, r);
        else return p;
    };

    // ---- states: S in registers (column c of this CTA, rows V tl + V TPC u + e), C and m in shared memory
    const int c = tid / P::TPC, tl = tid % P::TPC;
    float S[P::NV][P::V];
#pragma unroll
    for (int u = 0; u < P::NV; ++u)
#pragma unroll
        for (int e = 0; e < P::V; ++e) {
            const int r = P::V * (tl + P::TPC * u) + e;
            S[u][e] = a.S0 ? a.S0[(base * D + r) * D + d0 + c] : 0.f;
        }
    for (int i = tid; i < DS * D; i += kThreads) C[i] = a.C0 ? a.C0[(base * D + d0) * D + i] : 0.f;
    for (int i = tid; i < D; i += kThreads) m[i] = a.m0 ? a.m0[base * D + i] : 0.f;
    const int64_t t0 = a.t0 ? a.t0[b] : 0;

    // ---- the inputs of a block, four values a load (zero past the sequence)
    float4 pq[P::NQ], pk[P::NQ], pg[P::NQ], pv[P::NVV];
    float pl = 0.f, ps = 0.f, pb = 0.f;
    auto fetch = [&](int tb) {
#pragma unroll
        for (int u = 0; u < P::NQ; ++u) {
            const int i = tid + kThreads * u, t = tb + i / (D / 4), col = 4 * (i % (D / 4));
            pq[u] = pk[u] = pg[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (t < a.T) {
                const size_t e = ((static_cast<size_t>(b) * a.T + t) * a.H + h) * D + col;
                pq[u] = load4(a.q, e, a.in_dtype);
                pk[u] = load4(a.k, e, a.in_dtype);
                if (BB == 0) pg[u] = load4(a.gate, e, a.gate_dtype);
            }
        }
#pragma unroll
        for (int u = 0; u < P::NVV; ++u) {
            const int i = tid + kThreads * u, t = tb + i / (DS / 4), col = d0 + 4 * (i % (DS / 4));
            pv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < kL * DS / 4 && t < a.T)
                pv[u] = load4(a.v, ((static_cast<size_t>(b) * a.T + t) * a.H + h) * D + col, a.in_dtype);
        }
        pl = ps = pb = 0.f;  // past the sequence: lambda = 0, a decay of 1 and beta = 0
        if (tid < kL && tb + tid < a.T) {
            const size_t e = (static_cast<size_t>(b) * a.T + tb + tid) * a.H + h;
            pl = a.lambda[e];
            if (BB == 1) {
                ps = static_cast<const float *>(a.gate)[e];
                pb = a.beta[e];
            }
        }
    };
    fetch(0);
    sync_cluster();  // every CTA of the cluster runs before its shared memory is written

    for (int tb = 0; tb < a.T; tb += kL) {
        const int n = min(kL, a.T - tb);
        // ---- stage the block
#pragma unroll
        for (int u = 0; u < P::NQ; ++u) {
            const int i = tid + kThreads * u, t = i / (D / 4), col = 4 * (i % (D / 4));
            *reinterpret_cast<float4 *>(qn + t * LD + col) = pq[u];
            *reinterpret_cast<float4 *>(kn + t * LD + col) = pk[u];
            if (BB == 0)
                *reinterpret_cast<float4 *>(al + t * D + col) =
                    make_float4(__expf(pg[u].x), __expf(pg[u].y), __expf(pg[u].z), __expf(pg[u].w));
        }
#pragma unroll
        for (int u = 0; u < P::NVV; ++u) {
            const int i = tid + kThreads * u;
            if (i < kL * DS / 4) *reinterpret_cast<float4 *>(vs + 4 * i) = pv[u];
        }
        if (tid < kL) {
            lam[tid] = pl;
            if (BB == 1) {
                gs[tid] = __expf(ps);
                be[tid] = pb;
            }
        }
        __syncthreads();
        // ---- l2 norms and m . qbar: a warp takes four tokens
        {
            constexpr int E = D / 32;
            float xq[4][E], xk[4][E], sq[4], sk[4], mq[4], mv[E];
#pragma unroll
            for (int e = 0; e < E; ++e) mv[e] = m[lane + 32 * e];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                sq[r] = sk[r] = mq[r] = 0.f;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    xq[r][e] = qn[(warp + 8 * r) * LD + lane + 32 * e];
                    xk[r][e] = kn[(warp + 8 * r) * LD + lane + 32 * e];
                    sq[r] += xq[r][e] * xq[r][e];
                    sk[r] += xk[r][e] * xk[r][e];
                    mq[r] = fmaf(mv[e], xq[r][e], mq[r]);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    sq[r] += __shfl_xor_sync(0xffffffffu, sq[r], o);
                    sk[r] += __shfl_xor_sync(0xffffffffu, sk[r], o);
                    mq[r] += __shfl_xor_sync(0xffffffffu, mq[r], o);
                }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float rq = a.l2norm ? rsqrtf(fmaxf(sq[r], 1e-12f)) : 1.f;
                const float rk = a.l2norm ? rsqrtf(fmaxf(sk[r], 1e-12f)) : 1.f;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    qn[(warp + 8 * r) * LD + lane + 32 * e] = xq[r][e] * rq;
                    kn[(warp + 8 * r) * LD + lane + 32 * e] = xk[r][e] * rk;
                }
                // (a row whose square overflows has qbar = 0, so m . qbar = 0 whatever m . q is)
                if (lane == 0) cq[warp + 8 * r] = rq > 0.f ? mq[r] * rq : 0.f;
            }
        }
        __syncthreads();
        // ---- scores of this CTA's tokens: sc_tj = [j <= t] qbar_t . kbar_j, lane = j
        {
            constexpr int R = P::LT >= 8 ? P::LT / 8 : 1;  // tokens a warp
            const int lt = warp * R;
            if (lt < P::LT) {
                const int t1 = s * P::LT + lt;
                float acc[R];
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] = 0.f;
#pragma unroll 4
                for (int x = 0; x < D; x += 4) {
                    const float4 kv = *reinterpret_cast<const float4 *>(kn + lane * LD + x);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float4 qv = *reinterpret_cast<const float4 *>(qn + (t1 + r) * LD + x);
                        acc[r] = fmaf(kv.x, qv.x, acc[r]);
                        acc[r] = fmaf(kv.y, qv.y, acc[r]);
                        acc[r] = fmaf(kv.z, qv.z, acc[r]);
                        acc[r] = fmaf(kv.w, qv.w, acc[r]);
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float x = lane <= t1 + r ? acc[r] : 0.f;
#pragma unroll
                    for (int p = 0; p < NS; ++p) *peer(sc + (t1 + r) * LSC + lane, p) = x;
                }
            }
        }
        sync_cluster();
        // ---- q_clean columns of this CTA's rows of C: lane = token, warp = rows d
        {
            const float tinv = 1.f / static_cast<float>(t0 + tb + lane + 1);
            const float mq = cq[lane], lt = lam[lane];
            constexpr int U = DS / kWarps < 4 ? DS / kWarps : 4;  // rows at a time
            for (int u0 = 0; u0 < DS / kWarps; u0 += U) {
                float z[U], z4[U][4], ms[U], cs = mq;  // four chains a row for C qbar; cs = m_t . qbar_t
                const int dl = warp * (DS / kWarps) + u0;  // local rows dl .. dl + U - 1
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    z4[u][0] = z4[u][1] = z4[u][2] = z4[u][3] = 0.f;
                    ms[u] = m[d0 + dl + u];
                }
#pragma unroll(U <= 2 ? 16 : 4)
                for (int x = 0; x < D; x += 4) {
                    const float4 qv = *reinterpret_cast<const float4 *>(qn + lane * LD + x);
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const float4 cv = *reinterpret_cast<const float4 *>(C + (dl + u) * D + x);
                        z4[u][0] = fmaf(cv.x, qv.x, z4[u][0]);
                        z4[u][1] = fmaf(cv.y, qv.y, z4[u][1]);
                        z4[u][2] = fmaf(cv.z, qv.z, z4[u][2]);
                        z4[u][3] = fmaf(cv.w, qv.w, z4[u][3]);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) z[u] = (z4[u][0] + z4[u][1]) + (z4[u][2] + z4[u][3]);
#pragma unroll(U <= 2 ? 16 : 8)
                for (int j = 0; j < kL; ++j) {
                    const float w = sc[lane * LSC + j];
                    cs += w;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        // (selected, not left to the zero score: a later token's key may be infinite or NaN)
                        const float kv = j <= lane ? kn[j * LD + d0 + dl + u] : 0.f;
                        z[u] = fmaf(w, kv, z[u]);
                        ms[u] += kv;
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int d = d0 + dl + u;
                    float sig = z[u] * tinv;
                    if (a.centered) sig -= ms[u] * cs * tinv * tinv;
                    qc[lane * LD + d] = qn[lane * LD + d] - lt * sig;
                }
            }
        }
        if constexpr (NS > 1) {
            // to the other CTAs, 16 bytes a store
            __syncthreads();
            constexpr int per = kL * DS / 4;
            for (int i = tid; i < per * (NS - 1); i += kThreads) {
                const int p = (s + 1 + i / per) % NS, x = i % per, off = (x / (DS / 4)) * LD + d0 + 4 * (x % (DS / 4));
                *reinterpret_cast<float4 *>(peer(qc + off, p)) = *reinterpret_cast<const float4 *>(qc + off);
            }
        }
        sync_cluster();
        // ---- C += sum_j kbar_j kbar_j^T (this CTA's rows), m += sum_j kbar_j; the next block's loads
        if (tb + kL < a.T) fetch(tb + kL);
        {
            constexpr int PC = D / 4;               // 16-byte columns of a row
            constexpr int RG = kThreads / PC;       // rows a pass
            const int p4 = 4 * (tid % PC), rg = tid / PC;
            constexpr int U = DS / RG < 4 ? (DS / RG > 0 ? DS / RG : 1) : 4;
            for (int r0 = rg; r0 < DS; r0 += RG * U) {
                float4 acc[U];
#pragma unroll
                for (int u = 0; u < U; ++u) acc[u] = *reinterpret_cast<const float4 *>(C + (r0 + RG * u) * D + p4);
#pragma unroll 8
                for (int j = 0; j < kL; ++j) {
                    const float4 kv = *reinterpret_cast<const float4 *>(kn + j * LD + p4);
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const float kr = kn[j * LD + d0 + r0 + RG * u];
                        acc[u].x = fmaf(kr, kv.x, acc[u].x);
                        acc[u].y = fmaf(kr, kv.y, acc[u].y);
                        acc[u].z = fmaf(kr, kv.z, acc[u].z);
                        acc[u].w = fmaf(kr, kv.w, acc[u].w);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) *reinterpret_cast<float4 *>(C + (r0 + RG * u) * D + p4) = acc[u];
            }
            if (tid < D) {
                float x = m[tid];
#pragma unroll 8
                for (int j = 0; j < kL; ++j) x += kn[j * LD + tid];
                m[tid] = x;
            }
        }
        if (BB == 1) {
            // q_clean . kbar of the tokens
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                float x = 0.f;
#pragma unroll
                for (int e = 0; e < D / 32; ++e)
                    x = fmaf(qc[(warp + 8 * r) * LD + lane + 32 * e], kn[(warp + 8 * r) * LD + lane + 32 * e], x);
                x = warp_sum(x);
                if (lane == 0) qk[warp + 8 * r] = x;
            }
            __syncthreads();
        }
        // ---- the backbone, token by token; o takes v's place.  The reads of a group of G tokens come
        // before its stores (rows past the sequence have kbar = 0, a decay of 1 and beta = 0: no change)
        constexpr int G = P::RPT > 8 ? (BB == 0 ? 4 : 2) : (BB == 0 ? 8 : 4);
        constexpr bool kKeep = P::RPT <= 16;  // delta rule: a token's kbar rows stay in registers
        for (int t0g = 0; t0g < n; t0g += G) {
            float vv[G], r0[G], r1[G];  // GLA: q_clean . S in r0; GDN: kbar . S, q_clean . S
#pragma unroll
            for (int g = 0; g < G; ++g) vv[g] = vs[(t0g + g) * DS + c];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int t = t0g + g;
                r0[g] = r1[g] = 0.f;
                if (BB == 0) {
#pragma unroll
                    for (int u = 0; u < P::NV; ++u) {
                        const int r = P::V * (tl + P::TPC * u);
                        float av[P::V], kv[P::V], qv[P::V];
                        ldv<P::V>(al + t * D + r, av);
                        ldv<P::V>(kn + t * LD + r, kv);
                        ldv<P::V>(qc + t * LD + r, qv);
#pragma unroll
                        for (int e = 0; e < P::V; ++e) {
                            S[u][e] = fmaf(av[e], S[u][e], kv[e] * vv[g]);
                            r0[g] = fmaf(S[u][e], qv[e], r0[g]);
                        }
                    }
                } else {
                    const float ag = gs[t], bt = be[t];
                    float kv[kKeep ? P::NV : 1][P::V], p0[P::V], p1[P::V];
#pragma unroll
                    for (int e = 0; e < P::V; ++e) p0[e] = p1[e] = 0.f;
#pragma unroll
                    for (int u = 0; u < P::NV; ++u) {
                        const int r = P::V * (tl + P::TPC * u), uk = kKeep ? u : 0;
                        float qv[P::V];
                        ldv<P::V>(kn + t * LD + r, kv[uk]);
                        ldv<P::V>(qc + t * LD + r, qv);
#pragma unroll
                        for (int e = 0; e < P::V; ++e) {
                            p0[e] = fmaf(kv[uk][e], S[u][e], p0[e]);
                            p1[e] = fmaf(qv[e], S[u][e], p1[e]);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < P::V; ++e) {
                        r0[g] += p0[e];
                        r1[g] += p1[e];
                    }
#pragma unroll
                    for (int o = P::TPC / 2; o > 0; o >>= 1) r0[g] += __shfl_xor_sync(0xffffffffu, r0[g], o);
                    // S <- alpha S + kbar (beta (v - alpha kbar^T S))
                    // (past the sequence S stays as it is, where 0 times an infinite kbar^T S would not leave it)
                    const float w = t < n ? bt * (vv[g] - ag * r0[g]) : 0.f;
#pragma unroll
                    for (int u = 0; u < P::NV; ++u) {
                        if (!kKeep) ldv<P::V>(kn + t * LD + P::V * (tl + P::TPC * u), kv[0]);
#pragma unroll
                        for (int e = 0; e < P::V; ++e) S[u][e] = fmaf(kv[kKeep ? u : 0][e], w, ag * S[u][e]);
                    }
                }
            }
#pragma unroll
            for (int o = P::TPC / 2; o > 0; o >>= 1)
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    if (BB == 0) r0[g] += __shfl_xor_sync(0xffffffffu, r0[g], o);
                    else r1[g] += __shfl_xor_sync(0xffffffffu, r1[g], o);
                }
            if (tl == 0)
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const int t = t0g + g;
                    // (delta rule: o = S_new^T q_clean expanded in the old state)
                    vs[t * DS + c] = BB == 0 ? a.scale * r0[g]
                                             : a.scale * (gs[t] * r1[g] - gs[t] * be[t] * qk[t] * r0[g] +
                                                          be[t] * qk[t] * vv[g]);
                }
        }
        __syncthreads();
        for (int i = tid; i < n * (DS / 4); i += kThreads) {
            const int t = i / (DS / 4), col = d0 + 4 * (i % (DS / 4));
            const float4 x = *reinterpret_cast<const float4 *>(vs + 4 * i);
            const size_t e = ((static_cast<size_t>(b) * a.T + tb + t) * a.H + h) * D + col;
            if (a.in_dtype == 0) {
                const __nv_bfloat162 lo = __floats2bfloat162_rn(x.x, x.y), hi = __floats2bfloat162_rn(x.z, x.w);
                uint2 y;
                y.x = *reinterpret_cast<const uint32_t *>(&lo);
                y.y = *reinterpret_cast<const uint32_t *>(&hi);
                *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(a.o) + e) = y;
            } else {
                *reinterpret_cast<float4 *>(static_cast<float *>(a.o) + e) = x;
            }
        }
        __syncthreads();
    }

    // ---- final states
    if (a.ST) {
#pragma unroll
        for (int u = 0; u < P::NV; ++u)
#pragma unroll
            for (int e = 0; e < P::V; ++e)
                a.ST[(base * D + P::V * (tl + P::TPC * u) + e) * D + d0 + c] = S[u][e];
    }
    if (a.CT)
        for (int i = tid; i < DS * D; i += kThreads) a.CT[(base * D + d0) * D + i] = C[i];
    if (a.mT && s == 0)
        for (int i = tid; i < D; i += kThreads) a.mT[base * D + i] = m[i];
}

template <int D, int BB, int NS>
struct Launch {
    static constexpr size_t kSmem = Shape<D, NS>::kFloats * sizeof(float);
    cudaLaunchAttribute at;
    cudaLaunchConfig_t cfg = {};

    Launch(long long seqs, cudaStream_t st) {
        cfg.gridDim = dim3(static_cast<unsigned>(seqs * NS));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmem;
        cfg.stream = st;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = NS;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
    }
    static cudaError_t allow() {
        return cudaFuncSetAttribute(recurrent_block_kernel<D, BB, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    static_cast<int>(kSmem));
    }
};

template <int D, int BB, int NS>
cudaError_t launch_ns(const RecurrentArgs &a, cudaStream_t st) {
    cudaError_t e = Launch<D, BB, NS>::allow();
    if (e != cudaSuccess) return e;
    Launch<D, BB, NS> l(static_cast<long long>(a.B) * a.H, st);
    return cudaLaunchKernelEx(&l.cfg, recurrent_block_kernel<D, BB, NS>, a);
}

// The clusters of NS CTAs that the current device runs at once, at one CTA an SM (the larger ones do not share
// one).  0 where it cannot be asked.
template <int D, int BB, int NS>
int resident() {
    static std::atomic<int> known[64];  // by device, 1 + the count
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int n = known[dev].load(std::memory_order_relaxed) - 1;
    if (n < 0) {
        Launch<D, BB, NS> l(1, nullptr);
        if (Launch<D, BB, NS>::allow() != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, recurrent_block_kernel<D, BB, NS>, &l.cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        known[dev].store(n + 1, std::memory_order_relaxed);
    }
    return n;
}

// The CTAs of a (batch, head): as many as keep every cluster resident, since a block's cost falls with them and a
// second round of clusters doubles it.  The clusters that fit are fewer than the SMs by count, as one lies within a
// GPC: on GB300 15 of eight CTAs, 36 of four, 76 of two.  d = 128, T = 256, GLA: 83 us a sequence on eight CTAs,
// 120 on four, 193 on two, 256 on one; sixteen sequences 120 us on four CTAs each, 164 on eight.
template <int D, int BB>
int cluster_ctas(long long seqs) {
    return seqs <= resident<D, BB, 8>() ? 8 : seqs <= resident<D, BB, 4>() ? 4 : seqs <= resident<D, BB, 2>() ? 2 : 1;
}

template <int D, int BB>
cudaError_t launch_d(const RecurrentArgs &a, cudaStream_t st) {
    switch (cluster_ctas<D, BB>(static_cast<long long>(a.B) * a.H)) {
        case 8: return launch_ns<D, BB, 8>(a, st);
        case 4: return launch_ns<D, BB, 4>(a, st);
        case 2: return launch_ns<D, BB, 2>(a, st);
        default: return launch_ns<D, BB, 1>(a, st);
    }
}

// The longest sequence for which the token-by-token kernel is the faster one.  A first block costs what `first`
// tokens there do (measured at 1 to 4096 sequences and 2 to 40 tokens; the columns: eight, four, two CTAs a sequence
// and one): with d = 128 and GLA the kernels meet at 12 us with one sequence, at 16 with 20, at 32 with 100, and
// with more sequences than SMs both take proportionally longer.  With d = 64 two CTAs of the token-by-token kernel
// share an SM at little cost, so it loses by a round of one CTA an SM (the only one, or the last of few), and over
// many rounds the states' traffic costs the blocks more.  A further block costs 13 to 16 tokens.
template <int D, int BB>
int token_limit(const RecurrentArgs &a) {
    constexpr int first[2][2][4] = {{{4, 5, 7, 22}, {3, 4, 5, 17}}, {{4, 6, 10, 17}, {3, 5, 7, 13}}};
    const long long seqs = static_cast<long long>(a.B) * a.H, sms = std::max(1, resident<D, BB, 1>());
    const long long rounds = (seqs + sms - 1) / sms;
    const int ns = cluster_ctas<D, BB>(seqs);
    int limit = first[D == 128][BB][ns == 8 ? 0 : ns == 4 ? 1 : ns == 2 ? 2 : 3];
    if (D == 64 && ns == 1) limit += rounds >= 10 ? 5 : rounds & 1 ? -static_cast<int>(limit / (2 * rounds)) : 0;
    return limit + (D == 128 && rounds == 1 ? 16 : 13) * (std::max(a.T - 1, 0) / kL);
}

}  // namespace

cudaError_t launch_recurrent_block(const RecurrentArgs &a, cudaStream_t s) {
    if (a.Dk == 128) return a.backbone == 0 ? launch_d<128, 0>(a, s) : launch_d<128, 1>(a, s);
    return a.backbone == 0 ? launch_d<64, 0>(a, s) : launch_d<64, 1>(a, s);
}

bool recurrent_block_pays(const RecurrentArgs &a) {
    if (a.Dk == 128) return a.T > (a.backbone == 0 ? token_limit<128, 0>(a) : token_limit<128, 1>(a));
    return a.T > (a.backbone == 0 ? token_limit<64, 0>(a) : token_limit<64, 1>(a));
}

}  // namespace ccq
