// Chunkwise Gated DeltaNet scan in plain fp32 FMA (Eq. 1 with Eq. 3).
//
// The tight-tolerance path (fp32 I/O, small or unusual head sizes).  One CTA owns VC state columns of one (sequence, value
// head) -- the columns of the state do not depend on one another -- keeps them in shared memory and walks the sequence in
// blocks of kC tokens.  Inside a block, with cg the running sum of g and
// S the incoming state, the per-token pseudo-values u_t solve the unit lower-triangular
// system
//     u_t + sum_{i<t} beta_t e^{cg_t-cg_i} (k_t.k_i) u_i = beta_t (v_t - e^{cg_t} S^T k_t)
// (solved here by forward substitution, lane = token), then
//     o_t = scale ( e^{cg_t} S^T q_t + sum_{i<=t} e^{cg_t-cg_i} (q_t.k_i) u_i )
//     S  <- e^{cg_C} S + sum_i e^{cg_C-cg_i} k_i u_i^T .
// Every exponent is a difference that is <= 0 for g <= 0, so nothing overflows.
//
// A small call is one CTA per head and a chain of blocks: what counts is the time of one block, and there the reads of shared
// memory (one per FMA in the direct form).  So the products work on register tiles (2 x 2 tokens, four tokens or rows per
// value read) with 16-byte reads along the contraction, the running sum is a warp scan, and the substitution hands u_i round
// by shuffles instead of leaving 31 dependent sums to one thread.  Measured on B200 with two heads of
// 64 x 64: the composition of four chunks and a scan of 64 tokens, 69.7 -> 28.7 us for the two calls (register tiles and four
// times the CTAs).
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"

namespace lkv {

namespace {

namespace cg = cooperative_groups;

constexpr int kC = 32;  // tokens per block

// row stride (floats) of the q and k tiles: 16-byte rows, successive rows four banks apart
__host__ __device__ constexpr int row_stride(int dk) { return (((dk + 3) / 4) | 1) * 4; }
// the same for products in steps of 16 channels: rows of a multiple of 16, every fourth row 16 banks on
__host__ __device__ constexpr int cluster_stride(int dk) { return (dk + 15) / 16 * 16 + 4; }
constexpr int kLdA = kC + 4;   // row stride of the coupling matrix A (read by lane = row)

template <typename T, int VC>
__global__ void __launch_bounds__(256) gdn_scan_fp32_kernel(const __grid_constant__ GdnArgs a) {
    constexpr int NG = 256 / VC;   // thread groups along tokens / state rows
    constexpr int TPER = kC / NG;  // tokens per thread in the token-parallel steps
    static_assert(kC % NG == 0 && TPER >= 1, "block shape");
    constexpr int kLdU = VC + 1;
    extern __shared__ __align__(16) float smem[];
    const int dk = a.d_k, dv = a.d_v;
    const int ks = row_stride(dk);
    float *Qs = smem;                      // [kC][ks], zero beyond dk
    float *Ks = Qs + kC * ks;              // [kC][ks]
    float *Am = Ks + kC * ks;              // [kC][kLdA]
    float *Pm = Am + kC * kLdA;            // [kC][kC]
    float *cg = Pm + kC * kC;              // [kC]
    float *bs = cg + kC;                   // [kC]
    float *ec = bs + kC;                   // [kC]   e^{cg_C - cg_i}
    float *S = ec + kC;                    // [dk][VC]
    float *Us = S + dk * VC;               // [kC][kLdU]   right-hand side, then u
    pdl_launch();
    pdl_wait();

    const int h = blockIdx.x, seq = a.cu[a.n_ranges + 1 + blockIdx.y];   // launch order: longest sequence first
    const bool tr = seq >= a.tr_first;                                    // transition sequence
    const int rg = tr ? seq - a.tr_first + a.tr_src0 : seq;
    const int hk = h / (a.H_v / a.H_k);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j = tid % VC, tg = tid / VC;
    const int j0 = blockIdx.z * VC;   // first column of this CTA
    const int t_begin = a.cu[rg], t_end = a.cu[rg + 1];
    const T *q = static_cast<const T *>(a.q);
    const T *k = static_cast<const T *>(a.k);
    const T *v = tr ? nullptr : static_cast<const T *>(a.v);
    T *o = tr ? nullptr : static_cast<T *>(a.o);
    // where this sequence's initial state lies (nullptr = zero) and where its final state goes (nullptr = nowhere)
    auto state_at = [&](int i) { return (static_cast<size_t>(i) * a.H_v + h) * dk * dv + j0; };
    const bool more = seq >= a.n_s0, own = tr && a.tr_out != nullptr;
    const float *S0 = more ? a.S0_more : a.S0;
    float *ST = own ? a.tr_out : seq >= a.st_first ? a.S_T : nullptr;
    const size_t obase = state_at(own ? seq - a.tr_first : seq - a.st_first);

    if (a.s0_identity || tr || !S0) {
        const bool id = a.s0_identity || tr;
        for (int m = tg; m < dk; m += NG) S[m * VC + j] = id && m == j0 + j ? 1.f : 0.f;
    } else {
        S0 += state_at(more ? seq - a.n_s0 : seq);
#pragma unroll 4
        for (int m = tg; m < dk; m += NG) S[m * VC + j] = S0[static_cast<size_t>(m) * dv + j];
    }
    for (int t = warp; t < kC; t += 8)
        for (int m = dk + lane; m < ks; m += 32) Qs[t * ks + m] = Ks[t * ks + m] = 0.f;

    for (int t0 = t_begin; t0 < t_end; t0 += kC) {
        const int n = min(kC, t_end - t0);
        // q, k: warp = token, lane = channel; v stays with the thread that forms its right-hand side
        for (int m = lane; m < dk; m += 32) {
            float qr[4], kr[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = warp + 8 * u;
                const size_t off = (static_cast<size_t>(t0 + t) * a.H_k + hk) * dk + m;
                qr[u] = t < n ? to_f32<T>(q[off]) : 0.f;
                kr[u] = t < n ? to_f32<T>(k[off]) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                Qs[(warp + 8 * u) * ks + m] = qr[u];
                Ks[(warp + 8 * u) * ks + m] = kr[u];
            }
        }
        float vr[TPER];
#pragma unroll
        for (int u = 0; u < TPER; ++u) {
            const int t = tg + NG * u;
            vr[u] = v && t < n ? to_f32<T>(v[(static_cast<size_t>(t0 + t) * a.H_v + h) * dv + j0 + j]) : 0.f;
        }
        if (warp == 0) {
            const bool ok = lane < n;  // a padded token is the identity step: g = 0, beta = 0
            float run = ok ? a.g[static_cast<size_t>(t0 + lane) * a.H_v + h] : 0.f;
            bs[lane] = ok ? a.beta[static_cast<size_t>(t0 + lane) * a.H_v + h] : 0.f;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const float up = __shfl_up_sync(0xffffffffu, run, d);
                if (lane >= d) run += up;
            }
            cg[lane] = run;
            ec[lane] = expf(__shfl_sync(0xffffffffu, run, 31) - run);
        }
        __syncthreads();
        // coupling matrices: thread = tokens t, t + 16 against the earlier tokens i, i + 16
        {
            const int t = tid >> 4, i = tid & 15;
            float kk[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, qk[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
            for (int m = 0; m < dk; m += 4) {
                float4 kt[2], qt[2], ki[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    kt[u] = *reinterpret_cast<const float4 *>(Ks + (t + 16 * u) * ks + m);
                    qt[u] = *reinterpret_cast<const float4 *>(Qs + (t + 16 * u) * ks + m);
                    ki[u] = *reinterpret_cast<const float4 *>(Ks + (i + 16 * u) * ks + m);
                }
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
                        kk[u][w] = fmaf(kt[u].x, ki[w].x, kk[u][w]); qk[u][w] = fmaf(qt[u].x, ki[w].x, qk[u][w]);
                        kk[u][w] = fmaf(kt[u].y, ki[w].y, kk[u][w]); qk[u][w] = fmaf(qt[u].y, ki[w].y, qk[u][w]);
                        kk[u][w] = fmaf(kt[u].z, ki[w].z, kk[u][w]); qk[u][w] = fmaf(qt[u].z, ki[w].z, qk[u][w]);
                        kk[u][w] = fmaf(kt[u].w, ki[w].w, kk[u][w]); qk[u][w] = fmaf(qt[u].w, ki[w].w, qk[u][w]);
                    }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                    const int tt = t + 16 * u, ii = i + 16 * w;
                    const float dec = ii <= tt ? expf(cg[tt] - cg[ii]) : 0.f;
                    Pm[tt * kC + ii] = ii <= tt ? dec * qk[u][w] : 0.f;
                    Am[tt * kLdA + ii] = ii < tt ? bs[tt] * dec * kk[u][w] : 0.f;
                }
        }
        // state products K S and Q S: thread (tg, j) owns tokens tg, tg + NG, ... of column j
        float kS[TPER], qS[TPER];
#pragma unroll
        for (int u = 0; u < TPER; ++u) { kS[u] = 0.f; qS[u] = 0.f; }
        {
            const int dk4 = dk & ~3;
            for (int m = 0; m < dk4; m += 4) {
                float s[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) s[c] = S[(m + c) * VC + j];
#pragma unroll
                for (int u = 0; u < TPER; ++u) {
                    const float4 kv = *reinterpret_cast<const float4 *>(Ks + (tg + NG * u) * ks + m);
                    const float4 qv = *reinterpret_cast<const float4 *>(Qs + (tg + NG * u) * ks + m);
                    kS[u] = fmaf(kv.x, s[0], kS[u]); qS[u] = fmaf(qv.x, s[0], qS[u]);
                    kS[u] = fmaf(kv.y, s[1], kS[u]); qS[u] = fmaf(qv.y, s[1], qS[u]);
                    kS[u] = fmaf(kv.z, s[2], kS[u]); qS[u] = fmaf(qv.z, s[2], qS[u]);
                    kS[u] = fmaf(kv.w, s[3], kS[u]); qS[u] = fmaf(qv.w, s[3], qS[u]);
                }
            }
            for (int m = dk4; m < dk; ++m) {
                const float s = S[m * VC + j];
#pragma unroll
                for (int u = 0; u < TPER; ++u) {
                    kS[u] = fmaf(Ks[(tg + NG * u) * ks + m], s, kS[u]);
                    qS[u] = fmaf(Qs[(tg + NG * u) * ks + m], s, qS[u]);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < TPER; ++u) {
            const int t = tg + NG * u;
            Us[t * kLdU + j] = bs[t] * (vr[u] - expf(cg[t]) * kS[u]);
        }
        __syncthreads();
        // forward substitution down the block: lane = token, a warp has VC / 8 columns, NC at a time
        {
            constexpr int NC = VC / 8 < 4 ? VC / 8 : 4;
            float ar[kC];
#pragma unroll
            for (int i = 0; i < kC; i += 4) *reinterpret_cast<float4 *>(ar + i) = *reinterpret_cast<const float4 *>(Am + lane * kLdA + i);
#pragma unroll 1
            for (int c0 = warp * (VC / 8); c0 < (warp + 1) * (VC / 8); c0 += NC) {
                float r[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) r[c] = Us[lane * kLdU + c0 + c];
#pragma unroll
                for (int i = 0; i < kC - 1; ++i)   // A is zero in the lanes up to i: u_i is final there
#pragma unroll
                    for (int c = 0; c < NC; ++c) r[c] = fmaf(-ar[i], __shfl_sync(0xffffffffu, r[c], i), r[c]);
#pragma unroll
                for (int c = 0; c < NC; ++c) Us[lane * kLdU + c0 + c] = r[c];
            }
        }
        __syncthreads();
        // outputs: P is zero above the diagonal
        if (o) {
            float acc[TPER];
#pragma unroll
            for (int u = 0; u < TPER; ++u) acc[u] = expf(cg[tg + NG * u]) * qS[u];
#pragma unroll 2
            for (int i = 0; i < kC; i += 4) {
                float uv[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) uv[c] = Us[(i + c) * kLdU + j];
#pragma unroll
                for (int u = 0; u < TPER; ++u) {
                    const float4 p = *reinterpret_cast<const float4 *>(Pm + (tg + NG * u) * kC + i);
                    acc[u] = fmaf(p.x, uv[0], acc[u]); acc[u] = fmaf(p.y, uv[1], acc[u]);
                    acc[u] = fmaf(p.z, uv[2], acc[u]); acc[u] = fmaf(p.w, uv[3], acc[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < TPER; ++u) {
                const int t = tg + NG * u;
                if (t < n) o[(static_cast<size_t>(t0 + t) * a.H_v + h) * dv + j0 + j] = from_f32<T>(a.scale * acc[u]);
            }
        }
        // state carry: thread (tg, j) owns four rows at a time of column j
        {
            float w[kC];
#pragma unroll
            for (int i = 0; i < kC; ++i) w[i] = ec[i] * Us[i * kLdU + j];
            const float gam = expf(cg[kC - 1]);
            for (int m = 4 * tg; m < dk; m += 4 * NG) {
                float acc[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[c] = m + c < dk ? gam * S[(m + c) * VC + j] : 0.f;
#pragma unroll
                for (int i = 0; i < kC; ++i) {
                    const float4 kv = *reinterpret_cast<const float4 *>(Ks + i * ks + m);
                    acc[0] = fmaf(kv.x, w[i], acc[0]); acc[1] = fmaf(kv.y, w[i], acc[1]);
                    acc[2] = fmaf(kv.z, w[i], acc[2]); acc[3] = fmaf(kv.w, w[i], acc[3]);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (m + c < dk) S[(m + c) * VC + j] = acc[c];
            }
        }
        __syncthreads();
    }
    if (ST) {
        __syncthreads();
#pragma unroll 4
        for (int m = tg; m < dk; m += NG) {
            const size_t e = static_cast<size_t>(m) * dv + j;
            float x = S[m * VC + j];
            if (a.S_add) x += a.S_add[state_at(seq) + e];
            store_state(ST, a.st_bf16, obase + e, x);
        }
    }
}

// The same for calls of few heads and sequences, where the time of a block is all that counts: eight columns a CTA, and the CTAs of a head
// in clusters of CS (d_v = 16, 32, 64 and more: 2, 4, 8), which form a part of the coupling matrices each and write it to one another.
// What bounds the products is what shared memory returns, a value a lane and warp a cycle, so they are one product in register tiles:
// the 64 rows [k; q] of the block against 32 / CS rows of k and the eight columns of S (kept transposed), 4 x (8 + 32 / CS) / 4 values a
// thread, the contraction split over four lanes (every other four channels of 16).  After that nothing leaves a warp: lane = token, warp =
// column for the right-hand side, the substitution and the outputs, lane = channel for the state.  Tokens of the next block are copied
// (fp32) while the other CTAs' parts are waited for.  Two heads of 64 x 64: a block 5.2 -> 3.1 us (product 0.7, substitution 0.5, outputs and
// state 0.8, the rest barriers and hand-overs); 64, 512 tokens 12.7, 85.4 -> 9.1, 52.8 us.  Slower: 16 columns a CTA, a row of k and
// q a lane and no cluster 13.9, 78; the tokens by bulk copies, a row each, 12.5, 78.5; copied at the start of a block 11.1, 62.5.
template <typename T, int CS>
__global__ void __cluster_dims__(1, 1, CS) __launch_bounds__(256) gdn_scan_fp32_cluster_kernel(const __grid_constant__ GdnArgs a) {
    constexpr int VC = 8, kOwn = kC / CS, NCT = (kOwn + VC) / 4;   // columns of the coupling matrices; product columns a thread
    const cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) float smem[];
    const int dk = a.d_k, dv = a.d_v, ks = cluster_stride(dk), dkp = ks - 4;
    float *KQ = smem;                         // two stages: [k; q] [2 kC][ks], zero beyond dk
    float *St = KQ + 4 * kC * ks;             // [VC][ks]: S^T, zero beyond dk
    float *Am = St + VC * ks;                 // two copies (of successive blocks) of A, P: [kC i][kC t] each
    float *sS = Am + 4 * kC * kC;             // S^T k, S^T q: [2][VC][kC]
    float *cgs = sS + 2 * VC * kC, *bs = cgs + 2 * kC;   // two copies each: running sum of g, beta
    float2 *U = reinterpret_cast<float2 *>(bs + 2 * kC);   // [VC][kC]: u, u times e^{cg_C - cg_i}
    pdl_launch();
    pdl_wait();
    const int h = blockIdx.x, seq = a.cu[a.n_ranges + 1 + blockIdx.y];   // launch order: longest sequence first
    const bool tr = seq >= a.tr_first;                                    // transition sequence
    const int rg = tr ? seq - a.tr_first + a.tr_src0 : seq;
    const int hk = h / (a.H_v / a.H_k);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = blockIdx.z % CS;
    const int j = blockIdx.z * VC + warp;     // this warp's column
    const int t_begin = a.cu[rg], t_end = a.cu[rg + 1];
    const T *q = static_cast<const T *>(a.q);
    const T *k = static_cast<const T *>(a.k);
    const T *v = tr ? nullptr : static_cast<const T *>(a.v);
    T *o = tr ? nullptr : static_cast<T *>(a.o);
    auto state_at = [&](int i) { return (static_cast<size_t>(i) * a.H_v + h) * dk * dv + j; };
    const bool more = seq >= a.n_s0, own = tr && a.tr_out != nullptr, id = a.s0_identity || tr;
    const float *S0 = more ? a.S0_more : a.S0;
    float *ST = own ? a.tr_out : seq >= a.st_first ? a.S_T : nullptr;
    const size_t obase = state_at(own ? seq - a.tr_first : seq - a.st_first);

    auto async16 = [](float *dst, const void *src) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
    };
    // k, q of the block at t0 into a stage (warp = tokens warp, warp + 8, ..); g, beta and v of it into registers
    constexpr bool async = std::is_same<T, float>::value;
    float g_next = 0.f, b_next = 0.f, v_next = 0.f;
    auto fetch = [&](int t0, int stage) {
        float *st = KQ + (stage * 2 * kC + warp) * ks;
        const size_t first = (static_cast<size_t>(t0 + warp) * a.H_k + hk) * dk, step = static_cast<size_t>(8) * a.H_k * dk;
        if (async && dk % 4 == 0) {
            for (int m = 4 * lane; m < dk; m += 128) {
                float *dst = st + m;
#pragma unroll
                for (int u = 0; u < kC / 8; ++u) {
                    if (t0 + warp + 8 * u < t_end) {
                        async16(dst + 8 * u * ks, k + first + m + u * step);
                        async16(dst + (kC + 8 * u) * ks, q + first + m + u * step);
                    } else {
                        *reinterpret_cast<float4 *>(dst + 8 * u * ks) = *reinterpret_cast<float4 *>(dst + (kC + 8 * u) * ks) = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
            }
        } else {
            for (int m = lane; m < dk; m += 32) {
                float *dst = st + m;
                float kr[kC / 8], qr[kC / 8];
#pragma unroll
                for (int u = 0; u < kC / 8; ++u) {
                    const bool in = t0 + warp + 8 * u < t_end;
                    kr[u] = in ? to_f32<T>(k[first + m + u * step]) : 0.f;
                    qr[u] = in ? to_f32<T>(q[first + m + u * step]) : 0.f;
                }
#pragma unroll
                for (int u = 0; u < kC / 8; ++u) {
                    dst[8 * u * ks] = kr[u];
                    dst[(kC + 8 * u) * ks] = qr[u];
                }
            }
        }
        if (async) asm volatile("cp.async.commit_group;" ::: "memory");
        const int t = t0 + lane;   // a padded token is the identity step: g = 0, beta = 0
        const bool ok = t < t_end;
        g_next = ok ? a.g[static_cast<size_t>(t) * a.H_v + h] : 0.f;
        b_next = ok ? a.beta[static_cast<size_t>(t) * a.H_v + h] : 0.f;
        v_next = v && ok ? to_f32<T>(v[(static_cast<size_t>(t) * a.H_v + h) * dv + j]) : 0.f;
    };
    if (t_begin < t_end) fetch(t_begin, 0);
    // the state, and zeros beyond dk
    if (!id && S0) S0 += state_at(more ? seq - a.n_s0 : seq);
    for (int m = lane; m < dkp; m += 32) {
        float x = 0.f;
        if (m < dk) x = id ? (m == j ? 1.f : 0.f) : S0 ? S0[static_cast<size_t>(m) * dv] : 0.f;
        St[warp * ks + m] = x;
    }
    for (int e = tid; e < 4 * kC * 16; e += 256)   // (at most 15 zeros a row)
        if (dk + (e & 15) < dkp) KQ[(e >> 4) * ks + dk + (e & 15)] = 0.f;
    cluster.sync();   // the others have started: their shared memory may be written

    // the product's tile of this thread, shared by four lanes: rows row0 .., columns col0, col0 + 4, ..
    const int part = lane & 3, row0 = 4 * ((tid >> 2) & 15), col0 = tid >> 6;
    int odd = 0;
    for (int t0 = t_begin; t0 < t_end; t0 += kC, odd ^= 1) {
        const float *Ks = KQ + odd * 2 * kC * ks;
        float *A = Am + odd * 2 * kC * kC, *P = A + kC * kC;
        const float bt = b_next, vt = v_next;
        float cg = g_next;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const float up = __shfl_up_sync(0xffffffffu, cg, d);
            if (lane >= d) cg += up;
        }
        if (warp == 0) {
            cgs[odd * kC + lane] = cg;
            bs[odd * kC + lane] = bt;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();   // this block's k, q and the state are there; everybody has left the other stage
        float acc[4][NCT];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int c = 0; c < NCT; ++c) acc[u][c] = 0.f;
        const float *rp = Ks + row0 * ks + 4 * part;
        const float *cp[NCT];
#pragma unroll
        for (int c = 0; c < NCT; ++c) cp[c] = (4 * c < kOwn ? Ks + (rank * kOwn + col0 + 4 * c) * ks : St + (col0 + 4 * c - kOwn) * ks) + 4 * part;
#pragma unroll 2
        for (int m = 0; m < dkp; m += 16) {
            float4 x[4], y[NCT];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = *reinterpret_cast<const float4 *>(rp + u * ks + m);
#pragma unroll
            for (int c = 0; c < NCT; ++c) y[c] = *reinterpret_cast<const float4 *>(cp[c] + m);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int c = 0; c < NCT; ++c) {
                    acc[u][c] = fmaf(x[u].x, y[c].x, acc[u][c]);
                    acc[u][c] = fmaf(x[u].y, y[c].y, acc[u][c]);
                    acc[u][c] = fmaf(x[u].z, y[c].z, acc[u][c]);
                    acc[u][c] = fmaf(x[u].w, y[c].w, acc[u][c]);
                }
        }
        // the four parts added up: lane `part` keeps row row0 + part
        const int row = row0 + part, t = row & (kC - 1);
        const float cgt = cgs[odd * kC + t], bst = bs[odd * kC + t];
#pragma unroll
        for (int c = 0; c < NCT; ++c) {
            const float g0 = part & 2 ? acc[0][c] : acc[2][c], g1 = part & 2 ? acc[1][c] : acc[3][c];
            float k0 = part & 2 ? acc[2][c] : acc[0][c], k1 = part & 2 ? acc[3][c] : acc[1][c];
            k0 += __shfl_xor_sync(0xffffffffu, g0, 2);
            k1 += __shfl_xor_sync(0xffffffffu, g1, 2);
            const float give = part & 1 ? k0 : k1;
            const float x = (part & 1 ? k1 : k0) + __shfl_xor_sync(0xffffffffu, give, 1);
            const int col = col0 + 4 * c;
            if (4 * c < kOwn) {
                const int i = rank * kOwn + col;
                const bool in = row < kC ? i < t : i <= t;
                const float dec = in ? expf(cgt - cgs[odd * kC + i]) : 0.f;
                const float y = in ? (row < kC ? bst * dec * x : dec * x) : 0.f;
                float *dst = (row < kC ? A : P) + i * kC + t;
#pragma unroll
                for (int r = 0; r < CS; ++r) *cluster.map_shared_rank(dst, r) = y;
            } else {
                sS[((row < kC ? 0 : VC) + col - kOwn) * kC + t] = x;
            }
        }
        // the others' parts, and the next block's tokens while they are waited for
        cluster.barrier_arrive();
        if (t0 + kC < t_end) fetch(t0 + kC, odd ^ 1);
        cluster.barrier_wait();
        // forward substitution down the block: lane = token
        const float et = expf(cg);
        float r = bt * (vt - et * sS[warp * kC + lane]);
        {
            float ar[kC];
#pragma unroll
            for (int i = 0; i < kC - 1; ++i) ar[i] = A[i * kC + lane];
#pragma unroll
            for (int i = 0; i < kC - 1; ++i)   // A is zero in the lanes up to i: u_i is final there
                r = fmaf(-ar[i], __shfl_sync(0xffffffffu, r, i), r);
        }
        const float last = __shfl_sync(0xffffffffu, cg, 31), gam = expf(last);
        float2 *u = U + warp * kC;
        u[lane] = make_float2(r, expf(last - cg) * r);
        __syncwarp();
        // outputs (P is zero above the diagonal) and new state, two channels a lane, in one loop: their reads are in flight together
        float x = et * sS[(VC + warp) * kC + lane];
        for (int mb = 0; mb < dkp; mb += 64) {   // (all lanes: each has a token's outputs)
            const int m0 = min(mb + lane, dkp - 1), m1 = min(mb + lane + 32, dkp - 1);
            float y0 = gam * St[warp * ks + m0], y1 = gam * St[warp * ks + m1];
#pragma unroll 8
            for (int i = 0; i < kC; ++i) {
                const float2 uw = u[i];
                if (mb == 0) x = fmaf(P[i * kC + lane], uw.x, x);
                y0 = fmaf(Ks[i * ks + m0], uw.y, y0);
                y1 = fmaf(Ks[i * ks + m1], uw.y, y1);
            }
            __syncwarp();   // (the last channel may have been read by several lanes)
            if (mb + lane < dkp) St[warp * ks + m0] = y0;
            if (mb + lane + 32 < dkp) St[warp * ks + m1] = y1;
        }
        if (o && t0 + lane < t_end) o[(static_cast<size_t>(t0 + lane) * a.H_v + h) * dv + j] = from_f32<T>(a.scale * x);
        __syncwarp();
    }
    if (ST)
        for (int m = lane; m < dk; m += 32) {
            const size_t e = static_cast<size_t>(m) * dv;
            float x = St[warp * ks + m];
            if (a.S_add) x += a.S_add[state_at(seq) + e];
            store_state(ST, a.st_bf16, obase + e, x);
        }
}

size_t smem_bytes(int dk, int vc) {
    return sizeof(float) * (2 * static_cast<size_t>(kC) * row_stride(dk) + kC * kLdA + kC * kC + 3 * kC + static_cast<size_t>(dk) * vc + kC * (vc + 1));
}

size_t cluster_smem_bytes(int dk) {
    return sizeof(float) * ((4 * kC + 8) * static_cast<size_t>(cluster_stride(dk)) + 4 * kC * kC + 2 * 8 * kC + 4 * kC + 8 * 2 * kC);
}
template <typename T, int CS>
cudaError_t launch_cluster(const GdnArgs &a, size_t smem, cudaStream_t s) {
    auto kernel = gdn_scan_fp32_cluster_kernel<T, CS>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kernel, dim3(a.H_v, a.n_seq, a.d_v / 8), 256, smem, s, a);
}

template <typename T, int VC>
cudaError_t launch(const GdnArgs &a, cudaStream_t s) {
    const size_t smem = smem_bytes(a.d_k, VC);
    auto kernel = gdn_scan_fp32_kernel<T, VC>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kernel, dim3(a.H_v, a.n_seq, a.d_v / VC), 256, smem, s, a);
}

// Shared memory of the CTAs of a call that goes to the clusters, or 0 for one that does not.
// - Where each CTA finds an SM.  The SMs of a cluster belong to one GPC, which leaves some without: 15, 33 and 74 clusters of 8, 4 and 2 are
//   resident at a time with one CTA an SM, 120, 132 and 148 of the 148 SMs (as numbers and not as a query, so that equal calls take the
//   same kernel, and give the same bits, whichever SMs a GPU has).  One cluster more and there is a second round: 64 tokens of 15,
//   16 heads of 176 x 64 15.9, 30.9 us against 24.4 without clusters.  CTAs that take less than half of an SM are packed two to an SM
//   although others are idle, so they ask for more: 64, 512 tokens of 15 heads of 64 x 64 12.6, 74 -> 9.9, 55 us (13.1, 87
//   without clusters).
// - Two to an SM a block takes longer, which only pays in long sequences and larger heads: 18 heads of 64 x 64 13.7 us (64 tokens), 23.9
//   (128), 43.0 (256), 95 (600) against 13.1, 23.6, 44.5, 102; 18 of 128 x 64 58, 130 (256, 600) against 67, 155; 16 of 32 x 64 38
//   (256) against 34.
// - Small heads have little to share: one head of 4 x 64 9.9 us (64 tokens) against 8.0; of 16 x 64 9.0, 25.4 (64, 256) against 9.0, 29.5.
constexpr size_t kOwnSmBytes = 116 * 1024;   // more than half of the 228 KB of an SM
size_t cluster_smem(const GdnArgs &a) {
    const long long ctas = static_cast<long long>(a.H_v) * a.n_seq * (a.d_v / 8);
    const size_t smem = cluster_smem_bytes(a.d_k);
    if (ctas > sm_count() || smem > 227 * 1024 || a.d_k < 16) return 0;
    const int without = a.d_v == 16 ? 0 : a.d_v == 32 ? 16 : 28;   // SMs
    const bool own = ctas <= sm_count() - without, longs = a.T_total >= 256LL * a.n_ranges;
    if (own && (a.d_k > 16 || longs)) return std::max(smem, kOwnSmBytes);
    return longs && a.d_k >= 64 && a.d_k % 16 == 0 && 2 * (smem + 1024) <= 228 * 1024 ? smem : 0;
}

// Columns per CTA: all of them when heads and sequences fill the GPU; otherwise halved as long as that still finds idle SMs.
// The coupling matrices are then computed once per part, side by side.
template <typename T>
cudaError_t dispatch(const GdnArgs &a, cudaStream_t s) {
    if (const size_t smem = cluster_smem(a))
        return a.d_v == 16 ? launch_cluster<T, 2>(a, smem, s) : a.d_v == 32 ? launch_cluster<T, 4>(a, smem, s) : launch_cluster<T, 8>(a, smem, s);
    int vc = a.d_v;
    const long long units = static_cast<long long>(a.H_v) * a.n_seq;
    while (vc > 16 && units * (a.d_v / vc) * 2 <= sm_count()) vc /= 2;
    switch (vc) {
        case 16: return launch<T, 16>(a, s);
        case 32: return launch<T, 32>(a, s);
        case 64: return launch<T, 64>(a, s);
        case 128: return launch<T, 128>(a, s);
        case 256: return launch<T, 256>(a, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Shapes this kernel takes: d_v a power of two in [16, 256], and the whole working set
// within the 227 KB of shared memory a CTA may use.
bool gdn_scan_fp32_supported(int dk, int dv) {
    const bool pow2 = dv >= 16 && dv <= 256 && (dv & (dv - 1)) == 0;
    return pow2 && dk >= 1 && smem_bytes(dk, dv) <= 227 * 1024;
}

cudaError_t launch_gdn_scan_fp32(const GdnArgs &a, bool io_bf16, cudaStream_t s) {
    return io_bf16 ? dispatch<__nv_bfloat16>(a, s) : dispatch<float>(a, s);
}

}  // namespace lkv
