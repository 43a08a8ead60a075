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
#include "common.cuh"

namespace lkv {

namespace {

constexpr int kC = 32;  // tokens per block

// row stride (floats) of the q and k tiles: 16-byte rows, successive rows four banks apart
__host__ __device__ constexpr int row_stride(int dk) { return (((dk + 3) / 4) | 1) * 4; }
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

size_t smem_bytes(int dk, int vc) {
    return sizeof(float) * (2 * static_cast<size_t>(kC) * row_stride(dk) + kC * kLdA + kC * kC + 3 * kC + static_cast<size_t>(dk) * vc + kC * (vc + 1));
}

template <typename T, int VC>
cudaError_t launch(const GdnArgs &a, cudaStream_t s) {
    const size_t smem = smem_bytes(a.d_k, VC);
    auto kernel = gdn_scan_fp32_kernel<T, VC>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kernel, dim3(a.H_v, a.n_seq, a.d_v / VC), 256, smem, s, a);
}

// Columns per CTA: all of them when heads and sequences fill the GPU; otherwise halved as long as that still finds idle SMs.
// The coupling matrices are then computed once per part, side by side.
template <typename T>
cudaError_t dispatch(const GdnArgs &a, cudaStream_t s) {
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
