// State-initialisation kernels (Eq. 4): single cached state, and exact composition
// (Eq. 6 as the chain of Eq. 5) for Mamba-2 (scalar decay, HBM-bound) and for GDN in
// plain fp32 FMA (the tight-tolerance / small-shape path; the tensor-core path for
// d_k = d_v = 128 lives in init_gdn_tensor.cu).
#include <algorithm>

#include <cooperative_groups.h>

#include "common.cuh"

namespace lkv {

namespace {

namespace cg = cooperative_groups;

// 16 bytes of pool state -> 4 (fp32 pool) or 8 (bf16 pool) floats.
template <bool BF16>
struct PoolVec;
template <>
struct PoolVec<false> {
    static constexpr int kElems = 4;
    __device__ static __forceinline__ void load(const void *base, size_t elem, float (&out)[4]) {
        const float4 v = __ldcs(reinterpret_cast<const float4 *>(static_cast<const float *>(base) + elem));
        out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
    }
};
template <>
struct PoolVec<true> {
    static constexpr int kElems = 8;
    __device__ static __forceinline__ void load(const void *base, size_t elem, float (&out)[8]) {
        const uint4 v = __ldcs(reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(base) + elem));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            out[2 * i] = __uint_as_float(w[i] << 16);
            out[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
};

template <int E>
__device__ __forceinline__ void store_vec(float *dst, const float (&v)[E]) {
#pragma unroll
    for (int i = 0; i < E; i += 4) __stcs(reinterpret_cast<float4 *>(dst + i), make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]));
}

// ---------------------------------------------------------------- single cached state
// S0[r] = states[ids[cu_k[r] + b_r]], b_r = sel[r] or the last position.  A pure copy: with
// an fp32 pool the bits are untouched.  grid = (vectors per state / 256, n_req).
template <bool BF16, class Args>
__global__ void __launch_bounds__(256) init_single_kernel(const __grid_constant__ Args a, size_t state_elems) {
    using PV = PoolVec<BF16>;
    pdl_launch();
    pdl_wait();
    const int r = blockIdx.y;
    const int k0 = a.cu_k(r), k1 = a.cu_k(r + 1);
    const size_t e = (static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x) * PV::kElems;
    if (e >= state_elems) return;
    float v[PV::kElems];
    if (k1 == k0) {
#pragma unroll
        for (int i = 0; i < PV::kElems; ++i) v[i] = 0.f;
    } else {
        const int b = a.sel(r, k1 - k0);
        const size_t chunk = static_cast<size_t>(a.id(k0 + b));
        PV::load(a.states, chunk * state_elems + e, v);
    }
    store_vec<PV::kElems>(a.S0 + static_cast<size_t>(r) * state_elems + e, v);
}

// ---------------------------------------------------------------- Mamba-2 exact composition
// S <- S_{c_1};  S <- exp(lambda_{c_j,h}) S + S_{c_j}.  Pure streaming: every thread owns
// one 16-byte vector of the state and walks the K chunks with kUnroll independent loads
// in flight; the decays are K scalars per head.  grid = (vectors per state / 256, n_req).
template <bool BF16>
__global__ void __launch_bounds__(256) init_mamba_exact_kernel(const __grid_constant__ InitArgs a, size_t state_elems, int head_elems) {
    using PV = PoolVec<BF16>;
    constexpr int E = PV::kElems;
    constexpr int kUnroll = 8;
    pdl_launch();
    pdl_wait();
    const int r = blockIdx.y;
    const int k0 = a.cu_k(r), K = a.cu_k(r + 1) - k0;
    const size_t e = (static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x) * E;
    if (e >= state_elems) return;
    const int h = static_cast<int>(e / head_elems);
    float acc[E];
#pragma unroll
    for (int i = 0; i < E; ++i) acc[i] = 0.f;
    int j = 0;
    if (K > 0) {
        PV::load(a.states, static_cast<size_t>(a.id(k0)) * state_elems + e, acc);
        j = 1;
    }
    for (; j < K; j += kUnroll) {
        float v[kUnroll][E];
        float dec[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            if (j + u < K) {
                const size_t c = static_cast<size_t>(a.id(k0 + j + u));
                PV::load(a.states, c * state_elems + e, v[u]);
                dec[u] = expf(__ldg(a.transitions + c * a.H + h));
            }
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            if (j + u < K) {
#pragma unroll
                for (int i = 0; i < E; ++i) acc[i] = fmaf(dec[u], acc[i], v[u][i]);
            }
        }
    }
    store_vec<E>(a.S0 + static_cast<size_t>(r) * state_elems + e, acc);
}

// ---------------------------------------------------------------- GDN exact composition, fp32 FMA
// One CTA owns TN columns of one head's state for one request: the chain
// S <- T_{c_j} S + S_{c_j} acts on the left, so columns never mix.  The current column
// block sits in shared memory; T_j streams through a ring in shared memory kTM rows at a time, copied asynchronously several
// tiles ahead (a step waited for global memory twice before;
// the measured figures stand at the scan, gdn_scan_fp32.cu).
constexpr int kTM = 32;        // transition rows per stage
constexpr int kMaxStages = 6;
// row stride (floats) of a staged transition: 16-byte rows, successive rows four banks apart
__host__ __device__ constexpr int t_stride(int dk) { return (((dk + 3) / 4) | 1) * 4; }

template <bool BF16, int TN>
__global__ void __launch_bounds__(256) init_gdn_exact_fp32_kernel(const __grid_constant__ InitArgs a, int stages) {
    constexpr int RG = 256 / TN, U = kTM / RG;   // thread (rg, c) has rows rg, rg + RG, ... of column c
    extern __shared__ __align__(16) float smem[];
    const int dk = a.d_k, dv = a.d_v, ts = t_stride(dk);
    float *Tt = smem;                           // stages x [kTM][ts]
    float *Scur = Tt + stages * kTM * ts;       // [dk][TN]
    float *Snew = Scur + dk * TN;               // [dk][TN]
    const int col0 = blockIdx.x * TN;
    const int h = blockIdx.y, r = blockIdx.z;
    pdl_launch();
    pdl_wait();
    const int k0 = a.cu_k(r), K = a.cu_k(r + 1) - k0;
    const size_t ss = static_cast<size_t>(dk) * dv;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = tid % TN;    // column inside the block
    const int rg = tid / TN;   // row group
    const bool col_ok = col0 + c < dv;

    auto load_state = [&](int chunk, int i) -> float {
        const size_t off = (static_cast<size_t>(chunk) * a.H + h) * ss + static_cast<size_t>(i) * dv + col0 + c;
        if (!col_ok) return 0.f;
        if (BF16) return __bfloat162float(static_cast<const __nv_bfloat16 *>(a.states)[off]);
        return static_cast<const float *>(a.states)[off];
    };
    // tile x of the sequence of all transitions, kTM rows each, into its stage: one asynchronous copy group per tile
    const int tiles = (dk + kTM - 1) / kTM, total = (K > 1 ? K - 1 : 0) * tiles;
    const bool vec = dk % 4 == 0;
    auto fetch = [&](int x) {
        if (x < total) {
            const int i0 = (x % tiles) * kTM;
            const float *Tj = a.transitions + (static_cast<size_t>(a.id(k0 + 1 + x / tiles)) * a.H + h) * dk * dk;
            float *st = Tt + (x % stages) * kTM * ts;
            for (int ii = warp; ii < kTM && i0 + ii < dk; ii += 8) {
                const float *src = Tj + static_cast<size_t>(i0 + ii) * dk;
                const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(st + ii * ts));
                if (vec)
                    for (int m = 4 * lane; m < dk; m += 128) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 4 * m), "l"(src + m) : "memory");
                else
                    for (int m = lane; m < dk; m += 32) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4 * m), "l"(src + m) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int x = 0; x < stages - 1; ++x) fetch(x);
#pragma unroll 4
    for (int i = rg; i < dk; i += RG) Scur[i * TN + c] = (K > 0) ? load_state(a.id(k0), i) : 0.f;
    for (int x = 0; x < total; ++x) {
        const int i0 = (x % tiles) * kTM, chunk = a.id(k0 + 1 + x / tiles);
        float acc[U], add[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {   // in flight while the tile is waited for
            const int i = i0 + rg + RG * u;
            add[u] = i < dk ? load_state(chunk, i) : 0.f;
            acc[u] = 0.f;
        }
        if (stages > 1) fetch(x + stages - 1);   // into the stage that every thread left at the end of the last round
        else fetch(x);
        switch (stages) {
            case 1: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
            case 2: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
            case 3: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
            case 4: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
            case 5: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
            default: asm volatile("cp.async.wait_group 5;" ::: "memory"); break;
        }
        __syncthreads();
        const float *st = Tt + (x % stages) * kTM * ts;
        const int dk4 = dk & ~3;
        for (int m = 0; m < dk4; m += 4) {
            float s[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] = Scur[(m + e) * TN + c];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float4 t = *reinterpret_cast<const float4 *>(st + (rg + RG * u) * ts + m);
                acc[u] = fmaf(t.x, s[0], acc[u]); acc[u] = fmaf(t.y, s[1], acc[u]);
                acc[u] = fmaf(t.z, s[2], acc[u]); acc[u] = fmaf(t.w, s[3], acc[u]);
            }
        }
        for (int m = dk4; m < dk; ++m)
#pragma unroll
            for (int u = 0; u < U; ++u) acc[u] = fmaf(st[(rg + RG * u) * ts + m], Scur[m * TN + c], acc[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + rg + RG * u;
            if (i < dk) Snew[i * TN + c] = acc[u] + add[u];
        }
        __syncthreads();
        if (x % tiles == tiles - 1) { float *t = Scur; Scur = Snew; Snew = t; }
    }
    if (total == 0) __syncthreads();
    if (col_ok)
#pragma unroll 4
        for (int i = rg; i < dk; i += RG)
            a.S0[(static_cast<size_t>(r) * a.H + h) * ss + static_cast<size_t>(i) * dv + col0 + c] = Scur[i * TN + c];
}

// The same for 8 columns a CTA, d_k a multiple of 8 up to 128 and whole groups of columns: what a small call runs, a chain of steps whose
// time is all that counts.  A stage holds all of T_j and the CTA's columns of S_j, copied asynchronously several steps ahead, so that
// nothing in a step waits for global memory and one barrier a step is enough.  A pair of lanes has two rows of two columns, a
// half of the products each (every other four channels): reads of 16 bytes along the contraction, four for sixteen products, with the
// eight different addresses of a warp in different banks.  Two heads of 64 x 64,
// K = 4, 8, 16: 12.9, 27.7, 57.5 -> 5.6, 10.9, 21.8 us.
constexpr int kNarrowMaxD = 128, kNarrowStages = 6;
template <bool BF16>
__global__ void __launch_bounds__(256) init_gdn_exact_narrow_kernel(const __grid_constant__ InitArgs a, int stages) {
    constexpr int TN = 8, kPasses = kNarrowMaxD / 64;
    constexpr int kElem = BF16 ? 2 : 4;
    extern __shared__ __align__(16) float smem[];
    const int dk = a.d_k, dv = a.d_v, ts = dk + 4, stage_floats = dk * ts + dk * TN;
    float *cur = smem;                       // the carried columns, [TN][ts], two copies
    float *next = cur + TN * ts;
    float *ring = next + TN * ts;            // stages x { T_j [dk][ts], the columns of S_j [dk][TN] as cached }
    const int col0 = blockIdx.x * TN, h = blockIdx.y, r = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int half = lane & 1, cp = 2 * ((lane >> 1) & 3), row0 = 2 * (4 * warp + (lane >> 3));   // of two columns, of two rows (and of row0 + 64)
    pdl_launch();
    pdl_wait();
    const int k0 = a.cu_k(r), K = a.cu_k(r + 1) - k0;
    const size_t ss = static_cast<size_t>(dk) * dv;
    auto async16 = [](float *dst, const void *src) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
    };
    // columns of chunk c as cached: rows of 32 (fp32) or 16 (bf16) bytes
    auto fetch_S = [&](float *dst, size_t c) {
        const char *src = static_cast<const char *>(a.states) + ((c * a.H + h) * ss + col0) * kElem;
        if (BF16)
            for (int i = tid; i < dk; i += 256) async16(dst + 4 * i, src + static_cast<size_t>(i) * dv * kElem);
        else
            for (int i = tid; i < 2 * dk; i += 256) async16(dst + 4 * i, src + static_cast<size_t>(i >> 1) * dv * kElem + 16 * (i & 1));
    };
    auto read_S = [&](const float *st, int row, int c) {
        return BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(st)[row * TN + c]) : st[row * TN + c];
    };
    auto fetch = [&](int j) {
        if (j < K) {
            const size_t c = a.id(k0 + j);
            float *st = ring + ((j - 1) % stages) * stage_floats;
            const float *Tj = a.transitions + (c * a.H + h) * dk * dk;
            const int per = dk / 4;
            for (int e = tid; e < dk * per; e += 256) {
                const int row = e / per;
                async16(st + row * ts + 4 * (e - row * per), Tj + 4 * static_cast<size_t>(e));
            }
            fetch_S(st + dk * ts, c);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float2 *out = reinterpret_cast<float2 *>(a.S0 + (static_cast<size_t>(r) * a.H + h) * ss + col0 + cp);
    // the first chunk's columns, through what is the second copy later; then as many transitions as there are stages but one
    if (K > 0) fetch_S(next, a.id(k0));
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int j = 1; j < stages; ++j) fetch(j);
    // all copies but the youngest n groups
    auto wait = [](int n) {
        switch (n) {
            case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
            case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
            case 3: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
            case 4: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
            default: asm volatile("cp.async.wait_group 5;" ::: "memory"); break;
        }
    };
    wait(stages - 1);
    __syncthreads();
    for (int p = 0; p < kPasses; ++p) {
        const int row = row0 + 64 * p + half;
        if (row >= dk) break;
#pragma unroll
        for (int c = 0; c < 2; ++c) cur[(cp + c) * ts + row] = K > 0 ? read_S(next, row, cp + c) : 0.f;
        if (K <= 1) out[static_cast<size_t>(row) * dv / 2] = make_float2(cur[cp * ts + row], cur[(cp + 1) * ts + row]);
    }
    for (int j = 1; j < K; ++j) {
        // T_{j + stages - 1} goes into the stage of T_{j - 1}, which everybody has left at the barrier
        wait(stages - 2);
        __syncthreads();
        fetch(j + stages - 1);
        const float *T = ring + ((j - 1) % stages) * stage_floats, *Sj = T + dk * ts;
        for (int p = 0; p < kPasses; ++p) {
            const int row = row0 + 64 * p;
            if (row >= dk) break;   // (the eight rows of a warp together)
            const float *t0 = T + row * ts + 4 * half, *s0 = cur + cp * ts + 4 * half;
            float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll 8
            for (int m = 0; m < dk; m += 8) {
                const float4 t[2] = {*reinterpret_cast<const float4 *>(t0 + m), *reinterpret_cast<const float4 *>(t0 + ts + m)};
                const float4 x[2] = {*reinterpret_cast<const float4 *>(s0 + m), *reinterpret_cast<const float4 *>(s0 + ts + m)};
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        acc[i][c] = fmaf(t[i].x, x[c].x, acc[i][c]);
                        acc[i][c] = fmaf(t[i].y, x[c].y, acc[i][c]);
                        acc[i][c] = fmaf(t[i].z, x[c].z, acc[i][c]);
                        acc[i][c] = fmaf(t[i].w, x[c].w, acc[i][c]);
                    }
            }
            // lane `half` keeps row + half
            float v[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float give = half ? acc[0][c] : acc[1][c], keep = half ? acc[1][c] : acc[0][c];
                v[c] = keep + __shfl_xor_sync(0xffffffffu, give, 1) + read_S(Sj, row + half, cp + c);
                next[(cp + c) * ts + row + half] = v[c];
            }
            if (j == K - 1) out[static_cast<size_t>(row + half) * dv / 2] = make_float2(v[0], v[1]);
        }
        float *x = cur; cur = next; next = x;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}
int narrow_stages(int dk) {   // 3 (d_k = 128) to 6
    const size_t carried = 2 * 8 * static_cast<size_t>(dk + 4) * sizeof(float), stage = (static_cast<size_t>(dk) * (dk + 4) + 8 * dk) * sizeof(float);
    return static_cast<int>(std::min<size_t>(kNarrowStages, (227 * 1024 - carried) / stage));
}
template <bool BF16>
cudaError_t launch_gdn_narrow(const InitArgs &a, cudaStream_t s) {
    const int stages = narrow_stages(a.d_k), d = a.d_k;
    const size_t smem = (2 * 8 * static_cast<size_t>(d + 4) + stages * (static_cast<size_t>(d) * (d + 4) + 8 * d)) * sizeof(float);
    auto kernel = init_gdn_exact_narrow_kernel<BF16>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kernel, dim3(a.d_v / 8, a.H, a.n_req), 256, smem, s, a, stages);
}

template <bool BF16, int TN>
cudaError_t launch_gdn_fp32(const InitArgs &a, cudaStream_t s) {
    const size_t state = 2 * static_cast<size_t>(a.d_k) * TN * sizeof(float), stage = static_cast<size_t>(kTM) * t_stride(a.d_k) * sizeof(float);
    const int stages = static_cast<int>(std::min<size_t>(kMaxStages, (227 * 1024 - state) / stage));
    const size_t smem = state + stages * stage;
    auto kernel = init_gdn_exact_fp32_kernel<BF16, TN>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kernel, dim3((a.d_v + TN - 1) / TN, a.H, a.n_req), 256, smem, s, a, stages);
}

}  // namespace

cudaError_t launch_init_single(const InitArgs &a, bool pool_bf16, cudaStream_t s) {
    const size_t elems = static_cast<size_t>(a.H) * a.d_k * a.d_v;
    const int per = pool_bf16 ? 8 : 4;
    dim3 grid(static_cast<unsigned>((elems / per + 255) / 256), a.n_req);
    auto launch = [&](const auto &x) {
        using Args = std::decay_t<decltype(x)>;
        return launch_chained(pool_bf16 ? init_single_kernel<true, Args> : init_single_kernel<false, Args>, grid, 256, 0, s, x, elems);
    };
    if (!a.idx.ptr && a.idx.n > kSmallIdxCap) return launch(a);
    InitArgsT<kSmallIdxCap> small;
    static_cast<InitArgsBase &>(small) = a;
    small.idx.ptr = a.idx.ptr;
    small.idx.n = a.idx.n;
    if (!a.idx.ptr) std::copy(a.idx.v, a.idx.v + a.idx.n, small.idx.v);
    return launch(small);
}

cudaError_t launch_init_mamba_exact(const InitArgs &a, bool pool_bf16, cudaStream_t s) {
    const size_t elems = static_cast<size_t>(a.H) * a.d_k * a.d_v;
    const int per = pool_bf16 ? 8 : 4;
    dim3 grid(static_cast<unsigned>((elems / per + 255) / 256), a.n_req);
    return launch_chained(pool_bf16 ? init_mamba_exact_kernel<true> : init_mamba_exact_kernel<false>, grid, 256, 0, s, a, elems, a.d_k * a.d_v);
}

// 32 columns of the state per CTA, or 8 where that many CTAs still find an SM each (a step is then a quarter of the work: what
// a small call waits for); 8 also where the rows are so long that two copies of 32 columns leave no room for a stage.
cudaError_t launch_init_gdn_exact_fp32(const InitArgs &a, bool pool_bf16, cudaStream_t s) {
    const long long narrow = static_cast<long long>((a.d_v + 7) / 8) * a.H * a.n_req;
    const bool wide_fits = (2 * static_cast<size_t>(a.d_k) * 32 + kTM * static_cast<size_t>(t_stride(a.d_k))) * sizeof(float) <= 227 * 1024;
    if (narrow <= sm_count() && a.d_k % 8 == 0 && a.d_k <= kNarrowMaxD && a.d_v % 8 == 0)
        return pool_bf16 ? launch_gdn_narrow<true>(a, s) : launch_gdn_narrow<false>(a, s);
    if (narrow <= sm_count() || !wide_fits) return pool_bf16 ? launch_gdn_fp32<true, 8>(a, s) : launch_gdn_fp32<false, 8>(a, s);
    return pool_bf16 ? launch_gdn_fp32<true, 32>(a, s) : launch_gdn_fp32<false, 32>(a, s);
}

namespace {

// Lanes walk consecutive heads, so every token's dt row is read with coalesced 128-byte accesses.  What bounds it is the latency of the
// loads, not their bytes.  A sequence of up to kDecayShort tokens is summed by one CTA of eight warps, a warp every eighth token,
// 16 loads in flight; a longer one in eight parts of its tokens, a part by eight warps with eight loads in flight.  The parts are
// side by side in a cluster or one after the other in a CTA: all sums are added in an order that the sequence's own length sets,
// whatever else is in the call.
// 80 heads: 1 x 16, 256, 512 tokens 1.4, 1.9, 2.6 us; 64 x 64 1.7, 256 x 64 3.6 (all in clusters 2.1, 2.2, 2.4, 7.7, 27.6; one load after
// the other in one CTA 1.6, 2.8, 4.4, 2.0, 3.2); 1 x 8192 18.5 and 32 x 2048 13.1 in clusters (144, 38).
constexpr int kDecayParts = 8, kDecayWarps = 8, kDecayLoads = 8, kDecayShort = 512;

__device__ __forceinline__ float decay_tree(const float (&x)[kDecayLoads]) {
    return ((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7]));
}
// dt of every eighth token, n of them, in eight running sums
__device__ __forceinline__ float decay_short(const float *dt, int H, int n) {
    const size_t step = static_cast<size_t>(kDecayWarps) * H;
    float acc[kDecayLoads];
#pragma unroll
    for (int i = 0; i < kDecayLoads; ++i) acc[i] = 0.f;
    for (; n > 0; n -= 2 * kDecayLoads, dt += 2 * kDecayLoads * step) {
        float v[2 * kDecayLoads];
#pragma unroll
        for (int i = 0; i < 2 * kDecayLoads; ++i) v[i] = i < n ? dt[i * step] : 0.f;
#pragma unroll
        for (int i = 0; i < 2 * kDecayLoads; ++i) acc[i % kDecayLoads] += v[i];
    }
    return decay_tree(acc);
}
// dt of every eighth of the tokens t .. end, in eight running sums
__device__ __forceinline__ float decay_part(const float *dt, int H, long long t, long long end) {
    float acc[kDecayLoads];
#pragma unroll
    for (int i = 0; i < kDecayLoads; ++i) acc[i] = 0.f;
    for (; t < end; t += kDecayWarps * kDecayLoads) {
        float v[kDecayLoads];
#pragma unroll
        for (int i = 0; i < kDecayLoads; ++i) v[i] = t + i * kDecayWarps < end ? dt[static_cast<size_t>(t + i * kDecayWarps) * H] : 0.f;
#pragma unroll
        for (int i = 0; i < kDecayLoads; ++i) acc[i] += v[i];
    }
    return decay_tree(acc);
}
__device__ __forceinline__ float decay_column(const float (*x)[32], int lane) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += x[i][lane];
    return s;
}

template <bool kCluster>
__device__ __forceinline__ void logdecay(const SsdArgs &a, float *__restrict__ out) {
    const int seq = blockIdx.y, part = kCluster ? blockIdx.x % kDecayParts : 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int h = (kCluster ? blockIdx.x / kDecayParts : blockIdx.x) * 32 + lane;
    __shared__ float red[kCluster ? 1 : kDecayParts][kDecayWarps][32], sum[kDecayParts][32];
    pdl_launch();
    pdl_wait();
    const int t0 = a.cu[seq], n = a.cu[seq + 1] - t0;
    const float *dt = a.dt + static_cast<size_t>(t0) * a.H + h;
    const bool in = h < a.H;
    if (n <= kDecayShort) {
        if (part > 0) return;   // (and so do the others of the cluster: nobody is waited for)
        sum[warp][lane] = in ? decay_short(dt + static_cast<size_t>(warp) * a.H, a.H, (n - warp + kDecayWarps - 1) / kDecayWarps) : 0.f;
        __syncthreads();
        if (warp == 0 && in) out[static_cast<size_t>(seq) * a.H + h] = a.A[h] * decay_column(sum, lane);
        return;
    }
    const long long per = (static_cast<long long>(n) + kDecayParts - 1) / kDecayParts;
    auto partial = [&](int p) { return in ? decay_part(dt, a.H, per * p + warp, min(per * (p + 1), static_cast<long long>(n))) : 0.f; };
    if (kCluster) {
        const cg::cluster_group cluster = cg::this_cluster();
        red[0][warp][lane] = partial(part);
        __syncthreads();
        if (warp == 0) sum[0][lane] = decay_column(red[0], lane);
        cluster.sync();
        if (part == 0 && warp == 0 && in) {
            float s = 0.f;
#pragma unroll
            for (int r = 0; r < kDecayParts; ++r) s += cluster.map_shared_rank(sum[0], r)[lane];
            out[static_cast<size_t>(seq) * a.H + h] = a.A[h] * s;
        }
        cluster.sync();   // the sums stay where they are until they have been read
    } else {
#pragma unroll 1
        for (int p = 0; p < kDecayParts; ++p) red[p][warp][lane] = partial(p);
        __syncthreads();
        sum[warp][lane] = decay_column(red[warp], lane);
        __syncthreads();
        if (warp == 0 && in) out[static_cast<size_t>(seq) * a.H + h] = a.A[h] * decay_column(sum, lane);
    }
}
__global__ void __cluster_dims__(kDecayParts, 1, 1) __launch_bounds__(32 * kDecayWarps)
mamba_logdecay_cluster_kernel(const __grid_constant__ SsdArgs a, float *__restrict__ out) { logdecay<true>(a, out); }
__global__ void __launch_bounds__(32 * kDecayWarps, 4)
mamba_logdecay_kernel(const __grid_constant__ SsdArgs a, float *__restrict__ out) { logdecay<false>(a, out); }

}  // namespace

cudaError_t launch_mamba_logdecay(const SsdArgs &a, float *logdecay, int longest, cudaStream_t s) {
    const int groups = (a.H + 31) / 32;
    // A launch of clusters costs 3.5 ns a CTA; in one CTA the longest sequence takes 4 (dt in L2) to 10 ns a token.  80 heads, clusters, CTAs:
    // 32 x 1024 tokens (768 CTAs in clusters) 8.7, 13.8 us; 64 x 1024 13.4, 14.5; 128 x 1024 22.8, 17.1; 400 x 1024 65, 40.
    if (longest > kDecayShort && static_cast<long long>(kDecayParts) * groups * a.n_seq <= 2LL * longest)
        return launch_chained(mamba_logdecay_cluster_kernel, dim3(kDecayParts * groups, a.n_seq), 32 * kDecayWarps, 0, s, a, logdecay);
    return launch_chained(mamba_logdecay_kernel, dim3(groups, a.n_seq), 32 * kDecayWarps, 0, s, a, logdecay);
}

namespace {

constexpr int kErrThreads = 256;
constexpr size_t kErrElemsPerCta = 16384;   // 64 KB of each input per CTA: 16 float4 per thread

// Squared norms of (x - r) and r over one slice of one state; one (num, den) pair per CTA, summed in a fixed order.
__global__ void state_err_partial_kernel(const float *__restrict__ x, const float *__restrict__ r, size_t elems, int parts,
                                         float *__restrict__ partials) {
    const int state = blockIdx.y, part = blockIdx.x;
    const size_t vecs = elems / 4;
    const size_t v0 = vecs * part / parts, v1 = vecs * (part + 1) / parts;
    const float4 *xv = reinterpret_cast<const float4 *>(x + static_cast<size_t>(state) * elems);
    const float4 *rv = reinterpret_cast<const float4 *>(r + static_cast<size_t>(state) * elems);
    float num = 0.f, den = 0.f;
    for (size_t i = v0 + threadIdx.x; i < v1; i += kErrThreads) {
        const float4 a = __ldcs(xv + i), b = __ldcs(rv + i);
        const float d0 = a.x - b.x, d1 = a.y - b.y, d2 = a.z - b.z, d3 = a.w - b.w;
        num += d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3;
        den += b.x * b.x + b.y * b.y + b.z * b.z + b.w * b.w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        num += __shfl_xor_sync(0xffffffffu, num, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    __shared__ float sn[kErrThreads / 32], sd[kErrThreads / 32];
    if ((threadIdx.x & 31) == 0) { sn[threadIdx.x >> 5] = num; sd[threadIdx.x >> 5] = den; }
    __syncthreads();
    if (threadIdx.x == 0) {
        float n = 0.f, d = 0.f;
        for (int w = 0; w < kErrThreads / 32; ++w) { n += sn[w]; d += sd[w]; }
        partials[2 * (static_cast<size_t>(state) * parts + part)] = n;
        partials[2 * (static_cast<size_t>(state) * parts + part) + 1] = d;
    }
}

__global__ void state_err_final_kernel(const float *__restrict__ partials, int parts, int n_states, float *__restrict__ rel_err) {
    const int state = blockIdx.x * blockDim.x + threadIdx.x;
    if (state >= n_states) return;
    float n = 0.f, d = 0.f;
    for (int p = 0; p < parts; ++p) {
        n += partials[2 * (static_cast<size_t>(state) * parts + p)];
        d += partials[2 * (static_cast<size_t>(state) * parts + p) + 1];
    }
    rel_err[state] = sqrtf(n) / sqrtf(d);
}

}  // namespace

int state_err_parts(size_t elems) {
    const size_t parts = (elems + kErrElemsPerCta - 1) / kErrElemsPerCta;
    return static_cast<int>(parts < 1 ? 1 : (parts > 4096 ? 4096 : parts));
}

cudaError_t launch_state_rel_error(const float *x, const float *r, float *rel_err, int n_states, size_t elems,
                                   float *partials, cudaStream_t s) {
    const int parts = state_err_parts(elems);
    state_err_partial_kernel<<<dim3(parts, n_states), kErrThreads, 0, s>>>(x, r, elems, parts, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    state_err_final_kernel<<<(n_states + 127) / 128, 128, 0, s>>>(partials, parts, n_states, rel_err);
    return cudaGetLastError();
}

}  // namespace lkv
