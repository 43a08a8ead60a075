// State and transition of cache chunks (Eq. 5 with Eq. 3) on the 5th-generation tensor cores, for d_k = d_v = 128 and bf16 k / v: one
// CTA owns one (chunk, value head) and carries both through the chunk's blocks of 64 tokens.
//
// The state S (from zero) and the transition T (from I, with v = 0) obey one recurrence, and all of a block that does not depend on what
// is carried is the same for both: loads, K K^T, A, its inverse, W = M diag(beta) K.  Notation, scaling, exact blocks and the order of
// all sums are those of the scan (gdn_scan_tensor.cu), which gives the same bits one by one:
//   (1) G    = K K^T;  A, M = (I + A)^{-1}, X1, X2                     tcgen05, mask and prep warps
//   (W) W^T  = K^T X2^T              -> bf16 tile                      tcgen05, W warps
//  (3a) U_S^T = V^T X1^T
//  (2W) U^T += C^T W^T for C = S, T; u -> bf16 pairs in place          tcgen05 (A = bf16 C^T in shared memory), chain warps
//   (5) C^T += u^T K; C^T -> bf16 tile for (2W) of the next block      tcgen05 (A from tensor memory), chain warps
// The two chains run in turn on the same warps: while one is in the tensor core the other is converted.
//
// Tensor memory holds both carried matrices in fp32 (256 columns), U of both, W and G, which fills it: the bf16 copies of S^T and T^T
// lie in shared memory (64 KB), where neither Q, Ps nor output tiles are needed.
//
// Bound: the chains, S and T in turn: (2W) 1.0 K cycles from issue to notice with a queue of other products before it, u 0.25 K, (5) 0.8 K,
// copy 0.7 K, of which one chain's products hide behind the other's conversions: 3.4 K a block, where the scan took 2 x 3.3 K for the two.
// 32 chunks x 2048 tokens, 32 heads: 785 -> 520 us (the scan kernel run twice per chunk; GPUs differ).  Slower: warps of their own
// for each chain (992 threads, 64 registers) 573, two groups of prep warps that take turns 537; level: five K stages, the loops over
// the two chains or the halves of a copy unrolled.
//
// Warps 0-7 chains (lane = column of the carried matrix, warpgroup = half of the tokens / rows), 8-9 mask, 10 TMA loads of K and the scalars,
// 11 TMA loads of V, 12-15 prep (the inverse), 16-19 W, 20 MMA issue of the chains, 21 MMA issue of (1) and (W).
#include <string.h>

#include "gdn_blocks.cuh"

namespace lkv {

namespace {

constexpr int kThreads = 704;

// shared-memory map (bytes, after 1024-byte alignment); operand tiles have 128-byte rows, 128-byte swizzle
constexpr int kKStage = 2 * kC * 128;                  // [K_kb0 | K_kb1], each [64 tokens x 128 B]
constexpr int kKStages = 4;
constexpr int kOffV = kKStages * kKStage;              // one V stage, [V_jb0 | V_jb1].  (Behind the K stages: (1) reads 128 rows from each half of a
                                                       // stage, of which the upper 64 are whatever follows and end in rows nobody looks at)
constexpr int kOffX = kOffV + 2 * kC * 128;            // X1 bf16 [64 rows t x 128 B], double-buffered
constexpr int kOffX2 = kOffX + 2 * kC * 128;           // X2 likewise, one buffer
constexpr int kOffW = kOffX2 + kC * 128;               // -W^T bf16 [128 rows d_k x 64 tokens]
constexpr int kOffC = kOffW + kD * 128;                // S^T, T^T as bf16: [2][128 rows j x 128 B] each, K-major operands of (2W)
constexpr int kCTile = 2 * kD * 128;
constexpr int kOffF = kOffC + 2 * kCTile;
constexpr int kOffD = kOffF + 2 * kFBytes;
constexpr int kOffGb = kOffD + kC * kLdD * 4;          // per-block scalars, four buffers
constexpr int kSmemBytes = kOffGb + 4 * kGbFloats * 4 + 1024;
static_assert(kSmemBytes + 512 <= 227 * 1024, "shared memory budget");

// tensor-memory map (columns)
constexpr uint32_t kTmC = 0;      // 2 x 128: S^T, T^T fp32
constexpr uint32_t kTmU = 256;    // 2 x 64: U^T fp32; in place u as bf16 pairs
constexpr uint32_t kTmW = 384;    // 64
constexpr uint32_t kTmG = 448;    // 64
constexpr uint32_t kTmemCols = 512;

struct Bars {   // index [2] where not said otherwise: the chain, S or T
    // single-arrival barriers: TMA transactions, tcgen05.commit, the scalar warp
    uint64_t full_k[kKStages], k_free[kKStages], full_v, v_free, g_done, w_done, w_free, x2_free, x1_free[2] /* block parity */, u_done[2], ds_done[2], gb_ready[4];
    // the two mask warps (block parity)
    uint64_t a_ready[2];
    // the four prep warps (block parity); the four W warps
    uint64_t m_ready[2], d_free, w_ready;
    // the eight chain warps
    uint64_t uw_ready[2], st_ready[2], chain_done[4];
};
constexpr int kBars1 = 2 * kKStages + 16, kBars2 = 2, kBars4 = 4, kBars8 = 8;
static_assert(sizeof(Bars) == 8 * (kBars1 + kBars2 + kBars4 + kBars8), "barrier table");

// Row t of A of block b from G (tensor memory, this thread's lane), two warps: fp16 into the tiles F0, the 16x16 diagonal blocks in fp32 into D0,
// their 8x8 blocks inverted
__device__ __forceinline__ void mask_a(Bars &bars, int b, uint32_t tm_g, const float *sc, unsigned char *F0, float *D0, int t, volatile int *dead, const GdnArgs &a) {
    const int row_hi = (t & 32) + 31;   // last row (token) of this warp
    const bool exact = sc[kGbExp + 3] != 0.f;
    // rows of A, strictly lower.  F is free once block b-2 has been inverted, D once the diagonal blocks of block b-1 are.
    if (b >= 2) mbar_wait(&bars.m_ready[b & 1], ((b - 2) >> 1) & 1, dead, a.status);
    if (b >= 1) mbar_wait(&bars.d_free, (b - 1) & 1, dead, a.status);
    mbar_wait(&bars.g_done, b & 1, dead, a.status);
    __syncwarp();
    tc_fence_after_sync();
    unsigned char *fb = F0 + (b & 1) * kFBytes + (t & 31) * kLdF;   // this row of the first tile
    float *drow = D0 + t * kLdD;
    const float bt = exact ? sc[kGbX1 + t] : -sc[kGbX2 + t];   // beta
    // Nothing is masked here: what lies above the 8x8 diagonal blocks is never read, and the substitution masks these
    // themselves.
#pragma unroll 1
    for (int q = 0; 32 * q <= row_hi; ++q) {
        const int i0 = 32 * q;
        unsigned char *frow = fb + (i0 + 31 == row_hi ? q : 2) * kFTile;
        uint32_t rr[32];
        tmem_ld32(tm_g + i0, rr);
        tmem_ld_wait();
        float v[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) v[c] = __uint_as_float(rr[c]) * bt;
        if (exact) apply_decay(v, sc + kGbL + i0, sc[kGbL + t]);
#pragma unroll
        for (int c = 0; c < 32; c += 8)
            *reinterpret_cast<uint4 *>(frow + 2 * c) =
                make_uint4(pack_f16(v[c], v[c + 1]), pack_f16(v[c + 2], v[c + 3]), pack_f16(v[c + 4], v[c + 5]), pack_f16(v[c + 6], v[c + 7]));
        if (i0 + 31 == row_hi) {
            if (t & 16) {
#pragma unroll
                for (int c = 0; c < 16; c += 4) *reinterpret_cast<float4 *>(drow + c) = make_float4(v[16 + c], v[17 + c], v[18 + c], v[19 + c]);
            } else {
#pragma unroll
                for (int c = 0; c < 16; c += 4) *reinterpret_cast<float4 *>(drow + c) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
            }
            __syncwarp();
        }
    }
    tc_fence_before_sync();
    // The 8x8 diagonal block of this row's group of eight, inverted by forward substitution in fp32: lane = row, the
    // rows that are final go around by shuffles.  d[i] is zero in the lanes up to row i, which keep their row.
    float d[8], xr[8];
    float *diag = drow + (t & 8);
#pragma unroll
    for (int c = 0; c < 8; c += 4) *reinterpret_cast<float4 *>(d + c) = *reinterpret_cast<const float4 *>(diag + c);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        d[c] = c < (t & 7) ? d[c] : 0.f;
        xr[c] = c == (t & 7) ? 1.f : -d[c];
    }
#pragma unroll
    for (int i = 1; i < 7; ++i)
#pragma unroll
        for (int c = 0; c < i; ++c) xr[c] = fmaf(-d[i], __shfl_sync(0xffffffffu, xr[c], i, 8), xr[c]);
#pragma unroll
    for (int c = 0; c < 8; c += 4) *reinterpret_cast<float4 *>(diag + c) = make_float4(xr[c], xr[c + 1], xr[c + 2], xr[c + 3]);
    warp_arrive(&bars.a_ready[b & 1]);
}
// The inverse of block b and its operands, four warps (wq): A from the mask warps in the fp16 tiles F0 (two buffers) and the diagonal
// blocks D0, column factors fx (those of X2 follow those of X1)
__device__ __forceinline__ void invert_block(Bars &bars, int b, unsigned char *F0, float *D0, unsigned char *xb1, unsigned char *xb2, const float *fx,
                                             int wq, int lane, volatile int *dead, const GdnArgs &a) {
    const int gid = lane >> 2, tig = lane & 3;
    const uint32_t Fs = smem_u32(F0 + (b & 1) * kFBytes);
    unsigned char *Ft = F0 + (b & 1) * kFBytes + (wq >> 1) * kFTile;   // the tile with this warp's diagonal block
    float *D = D0 + (16 * wq) * kLdD;                                  // the block itself
    // ---- A comes from the mask warpgroup (epilogue of (1)), its 8x8 diagonal blocks inverted; here the rest of it turns
    // into M = (I + A)^{-1} by doubling.
    mbar_wait(&bars.a_ready[b & 1], (b >> 1) & 1, dead, a.status);
    uint32_t a32[4];
    frag_a(a32, smem_u32(Ft) + 16 * kLdF, lane);
    // 8 -> 16 in fp32: warp w has the 16x16 diagonal block w, thread = (row i, column pair) of each of its three 8x8 blocks;
    // T = A21 inv(L1) passes through the block above the diagonal.
    {
        const int i = gid, j0 = 2 * tig;
        const float *d2 = D + (8 + i) * kLdD;
        float av[8], dv[8], t0 = 0.f, t1 = 0.f, m0 = 0.f, m1 = 0.f;
#pragma unroll
        for (int m = 0; m < 8; m += 4) *reinterpret_cast<float4 *>(av + m) = *reinterpret_cast<const float4 *>(d2 + m);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const float2 d = *reinterpret_cast<const float2 *>(D + m * kLdD + j0);   // zero where m < j: inv(L1) is lower triangular
            t0 = fmaf(av[m], d.x, t0);
            t1 = fmaf(av[m], d.y, t1);
        }
        *reinterpret_cast<float2 *>(D + i * kLdD + 8 + j0) = make_float2(t0, t1);
        const float2 d11 = *reinterpret_cast<const float2 *>(D + i * kLdD + j0), d22 = *reinterpret_cast<const float2 *>(d2 + 8 + j0);
#pragma unroll
        for (int m = 0; m < 8; m += 4) *reinterpret_cast<float4 *>(dv + m) = *reinterpret_cast<const float4 *>(d2 + 8 + m);
        __syncwarp();
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const float2 d = *reinterpret_cast<const float2 *>(D + m * kLdD + 8 + j0);   // dv is zero where m > i
            m0 = fmaf(-dv[m], d.x, m0);
            m1 = fmaf(-dv[m], d.y, m1);
        }
        warp_arrive(&bars.d_free);
        // X1 and X2 are written as the entries of M become final: the buffers were read by (3a) of block b-2 and by W of block b-1
        if (b >= 2) mbar_wait(&bars.x1_free[b & 1], ((b - 2) >> 1) & 1, dead, a.status);
        if (b >= 1) mbar_wait(&bars.x2_free, (b - 1) & 1, dead, a.status);
        unsigned char *fr = Ft + (16 * (wq & 1) + i) * kLdF + (16 * (wq & 1) + j0) * 2;
        *reinterpret_cast<uint32_t *>(fr) = pack_f16(d11.x, d11.y);
        *reinterpret_cast<uint32_t *>(fr + 16) = 0u;
        *reinterpret_cast<uint32_t *>(fr + 8 * kLdF) = pack_f16(m0, m1);
        *reinterpret_cast<uint32_t *>(fr + 8 * kLdF + 16) = pack_f16(d22.x, d22.y);
        const float acc[4] = {d11.x, d11.y, m0, m1}, acc2[4] = {0.f, 0.f, d22.x, d22.y};
        store_acc_x(xb1, xb2, fx, 16 * wq, 16 * wq, acc, 1.f, gid, tig);
        store_acc_x(xb1, xb2, fx, 16 * wq, 16 * wq + 8, acc2, 1.f, gid, tig);
    }
    uint32_t a64[2][2][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int kb = 0; kb < 2; ++kb) frag_a(a64[mt][kb], Fs + 2 * kFTile + (16 * mt) * kLdF + 32 * kb, lane);
    named_bar_sync(1, 128);
    // 16 -> 32: blocks (1, 0) and (3, 2), one half block per warp
    inv_merge32(a32, Ft, xb1, xb2, fx, wq & 2, wq & 1, lane);
    named_bar_sync(1, 128);
    // 32 -> 64: eight columns of the 32x32 result per warp
    inv_merge64(a64, Fs, xb1, xb2, fx, wq, lane);
    fence_async_smem();
    warp_arrive(&bars.m_ready[b & 1]);
}
// Scalars of a block, one warp: lane = tokens 2 lane, 2 lane + 1; R: exponent that the state is left with, before and after.
__device__ __forceinline__ void block_scalars(float *sc, float &R, float2 gv, float2 bv, const GdnArgs &a, int lane) {
    float run = gv.x + gv.y;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float up = __shfl_up_sync(0xffffffffu, run, o);
        if (lane >= o) run += up;
    }
    const float c0 = (run - gv.y) * kLog2e, c1 = run * kLog2e;
    const float last = __shfl_sync(0xffffffffu, c1, 31);
    const bool exact = __any_sync(0xffffffffu, fabsf(c0) > kMaxRange || fabsf(c1) > kMaxRange);
    float Rn = R;
    if (exact || fabsf(R - last) > kMaxScale) Rn = 0.f;
    const int t = 2 * lane;
    *reinterpret_cast<float2 *>(sc + kGbL + t) = make_float2(c0, c1);
    *reinterpret_cast<float2 *>(sc + kGbX1 + t) = exact ? bv : make_float2(bv.x * ex2(Rn - c0), bv.y * ex2(Rn - c1));
    *reinterpret_cast<float2 *>(sc + kGbX2 + t) = exact ? make_float2(-bv.x * ex2(c0), -bv.y * ex2(c1)) : make_float2(-bv.x, -bv.y);
    if (exact) *reinterpret_cast<float2 *>(sc + kGbW + t) = make_float2(ex2(last - c0), ex2(last - c1));
    const float in = Rn - R;
    R = exact ? 0.f : Rn - last;
    if (lane == 0) *reinterpret_cast<float4 *>(sc + kGbExp) = make_float4(in, exact ? in + last : in, -R, exact ? 1.f : 0.f);
}

// 64 values of row j of the bf16 tile from their columns in tensor memory, both times 2^exponent (the fp32 ones in place): rare
__device__ __noinline__ void rescale_carried(uint32_t tm_c, unsigned char *tile, int j, float copy_exp, float acc_exp) {
    const float fc = ex2(copy_exp), fa = ex2(acc_exp - copy_exp);
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
        uint32_t rr[16];
        float v[16];
        tmem_ld16(tm_c + 16 * q, rr);
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = __uint_as_float(rr[c]) * fc;
        store_row_chunks(tile, j, 2 * q, v);
#pragma unroll
        for (int c = 0; c < 16; ++c) rr[c] = __float_as_uint(v[c] * fa);
        tmem_st16(tm_c + 16 * q, rr);
    }
    tmem_st_wait();
}
// 64 rows of a carried matrix, this thread's column, times f^2 to memory
__device__ __noinline__ void store_carried(uint32_t tm_c, float *out, float f) {
#pragma unroll 1
    for (int q = 0; q < 4; ++q, out += 16 * kD) {
        uint32_t rr[16];
        tmem_ld16(tm_c + 16 * q, rr);
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < 16; ++c) out[c * kD] = __uint_as_float(rr[c]) * f * f;
    }
}

__global__ void __launch_bounds__(kThreads, 1)
gdn_build_tensor_kernel(const __grid_constant__ GdnArgs a, const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);   // an offset, not a cast: the compiler keeps shared-memory addressing
    __shared__ Bars bars;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int dead;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_launch();
    if (a.cu.ptr) pdl_wait();   // the index list is in global memory
    const int h = blockIdx.x, seq = a.cu[a.n_ranges + 1 + blockIdx.y];   // launch order: longest chunk first
    const int t_begin = a.cu[seq], t_end = a.cu[seq + 1];
    const int nblk = (t_end - t_begin + kC - 1) / kC;
    const size_t obase = (static_cast<size_t>(seq) * a.H_v + h) * kD * kD;

    if (nblk == 0) {  // empty chunk: zero state, the identity
        pdl_wait();
        hand_through(a.S_T, obase, 0, false, nullptr, nullptr);
        hand_through(a.tr_out, obase, 0, true, nullptr, nullptr);
        return;
    }
    if (tid == 0) {
        dead = 0;
        uint64_t *bp = &bars.full_k[0];
        for (int i = 0; i < kBars1; ++i) mbar_init(bp++, 1);
        for (int i = 0; i < kBars2; ++i) mbar_init(bp++, 2);
        for (int i = 0; i < kBars4; ++i) mbar_init(bp++, 4);
        for (int i = 0; i < kBars8; ++i) mbar_init(bp++, 8);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(&tmem_base, kTmemCols);
    pdl_wait();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tm = tmem_base;
    const uint32_t lane_base = tm + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    float *gb = reinterpret_cast<float *>(sm + kOffGb);

    if (warp == 10) {
        // ======================================================= TMA loads of the K tiles and the scalars of a block.  Here and in the
        // other single-issue roles the whole warp walks the loop and one elected lane issues.
        const int hk = h / (a.H_v / a.H_k);
        auto fetch_gb = [&](int b, float2 &gv, float2 &bv) {
            const int t = t_begin + b * kC + 2 * lane;
            gv = make_float2(0.f, 0.f); bv = make_float2(0.f, 0.f);
            if (t < t_end) {
                gv.x = a.g[static_cast<size_t>(t) * a.H_v + h];
                bv.x = a.beta[static_cast<size_t>(t) * a.H_v + h];
            }
            if (t + 1 < t_end) {
                gv.y = a.g[static_cast<size_t>(t + 1) * a.H_v + h];
                bv.y = a.beta[static_cast<size_t>(t + 1) * a.H_v + h];
            }
        };
        float2 gv_next = make_float2(0.f, 0.f), bv_next = gv_next;
        float R = 0.f;   // what is carried is held times 2^R
#pragma unroll 1
        for (int b = -1; b < nblk; ++b) {
            const float2 gv = gv_next, bv = bv_next;
            fetch_gb(b + 1, gv_next, bv_next);   // in flight while this block is prepared
            if (b < 0) continue;
            if (warp_dead(&dead)) break;   // a wait ran out: nothing more is issued
            const int s4 = b % kKStages, row = t_begin + b * kC;
            if (b >= kKStages) mbar_wait(&bars.k_free[s4], ((b - kKStages) / kKStages) & 1, &dead, a.status);
            __syncwarp();
            if (elect_one()) {
                mbar_expect_tx(&bars.full_k[s4], kKStage);
#pragma unroll 1
                for (int kb = 0; kb < 2; ++kb) {
                    tma_load_2d(sm + s4 * kKStage + kb * kC * 128, &mapK, hk * kD + kb * 64, row, &bars.full_k[s4]);
                    if (b + kKStages < nblk) tma_prefetch_l2_2d(&mapK, hk * kD + kb * 64, row + kKStages * kC);
                }
            }
            __syncwarp();
            // the buffer of block b was last read by the chains of block b-4
            if (b >= 4) mbar_wait(&bars.chain_done[b & 3], ((b - 4) >> 2) & 1, &dead, a.status);
            __syncwarp();
            block_scalars(gb + (b & 3) * kGbFloats, R, gv, bv, a, lane);
            warp_arrive(&bars.gb_ready[b & 3]);
        }
    } else if (warp == 11) {
        // ======================================================= TMA loads of V
#pragma unroll 1
        for (int b = 0; b < nblk; ++b) {
            if (warp_dead(&dead)) break;   // a wait ran out: nothing more is issued
            if (b >= 1) mbar_wait(&bars.v_free, (b - 1) & 1, &dead, a.status);
            __syncwarp();
            if (elect_one()) {
                const int row = t_begin + b * kC;
                mbar_expect_tx(&bars.full_v, 2 * kC * 128);
#pragma unroll 1
                for (int jb = 0; jb < 2; ++jb) {
                    tma_load_2d(sm + kOffV + jb * kC * 128, &mapV, h * kD + jb * 64, row, &bars.full_v);
                    if (b + 2 < nblk) tma_prefetch_l2_2d(&mapV, h * kD + jb * 64, row + 2 * kC);
                }
            }
            __syncwarp();
        }
    } else if (warp == 21) {
        // ======================================================= MMA issue of (1) and W
        constexpr uint32_t idG = umma_idesc(kFmtBF16, false, false, 128, 64);
        constexpr uint32_t idW = umma_idesc(kFmtBF16, true, false, 128, 64);   // A = K tile read MN-major
        const uint64_t dX2 = umma_desc(smem_u32(sm + kOffX2), 0, 1024);
#pragma unroll 1
        for (int b = 0; b <= nblk; ++b) {
            if (warp_dead(&dead)) break;   // a wait ran out: nothing more is issued
            if (b < nblk) {
                // (1) of block b: the mask warps have drained the G columns of block b-1
                if (b >= 1) mbar_wait(&bars.a_ready[(b - 1) & 1], ((b - 1) >> 1) & 1, &dead, a.status);
                mbar_wait(&bars.full_k[b % kKStages], (b / kKStages) & 1, &dead, a.status);
                __syncwarp();
                tc_fence_after_sync();
                const uint64_t dK = umma_desc(smem_u32(sm + (b % kKStages) * kKStage), 0, 1024);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const uint64_t off = ((k >> 2) * (kC * 128) + (k & 3) * 32) >> 4;
                        umma_bf16(tm + kTmG, dK + off, dK + off, idG, k > 0);
                    }
                    umma_commit(&bars.g_done);
                }
                __syncwarp();
            }
            if (b >= 1) {
                // -W^T of block b-1, once its inverse is there and the W warps have drained the W columns
                const int c = b - 1;
                if (c >= 1) mbar_wait(&bars.w_ready, (c - 1) & 1, &dead, a.status);
                mbar_wait(&bars.m_ready[c & 1], (c >> 1) & 1, &dead, a.status);
                __syncwarp();
                tc_fence_after_sync();
                const uint64_t dKm = umma_desc(smem_u32(sm + (c % kKStages) * kKStage), kC * 128, 1024);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) umma_bf16(tm + kTmW, dKm + ((k * 16 * 128) >> 4), dX2 + 2 * k, idW, k > 0);
                    umma_commit(&bars.w_done);
                    umma_commit(&bars.x2_free);
                }
                __syncwarp();
            }
        }
    } else if (warp == 20) {
        // ======================================================= MMA issue of (3a), (2W), (5), S before T
        constexpr uint32_t idV = umma_idesc(kFmtBF16, true, false, 128, 64);       // (3a): A = V tile read MN-major
        constexpr uint32_t id2W = umma_idesc(kFmtBF16, false, true, 128, 64);      // B = -W^T tile read MN-major
        constexpr uint32_t id5 = umma_idesc(kFmtBF16, false, true, 128, 128);      // B = K tile read MN-major
        const uint64_t dW = umma_desc(smem_u32(sm + kOffW), 0, 1024), dV = umma_desc(smem_u32(sm + kOffV), kC * 128, 1024);
#pragma unroll 1
        for (int b = 0; b < nblk; ++b) {
            if (warp_dead(&dead)) break;
            const uint32_t par = b & 1;
            const uint64_t dK = umma_desc(smem_u32(sm + (b % kKStages) * kKStage), kC * 128, 1024);
            // (3a): the U columns were read by (5) of block b-1, issued before
            mbar_wait(&bars.full_v, par, &dead, a.status);
            mbar_wait(&bars.m_ready[par], (b >> 1) & 1, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
            const uint64_t dX = umma_desc(smem_u32(sm + kOffX + par * (kC * 128)), 0, 1024);
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 4; ++k) umma_bf16(tm + kTmU, dV + ((k * 16 * 128) >> 4), dX + 2 * k, idV, k > 0);
                umma_commit(&bars.v_free);
                umma_commit(&bars.x1_free[par]);
            }
            __syncwarp();
            mbar_wait(&bars.w_ready, par, &dead, a.status);
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
                // (2W): needs the block's W tile and the bf16 copy
                mbar_wait(&bars.st_ready[c], par, &dead, a.status);
                __syncwarp();
                tc_fence_after_sync();
                const uint64_t dC = umma_desc(smem_u32(sm + kOffC + c * kCTile), 0, 1024);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        umma_bf16(tm + kTmU + 64 * c, dC + (((k >> 2) * (kD * 128) + (k & 3) * 32) >> 4), dW + ((k * 16 * 128) >> 4), id2W, c == 0 || k > 0);
                    umma_commit(&bars.u_done[c]);
                    if (c == 1) umma_commit(&bars.w_free);
                }
                __syncwarp();
            }
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
                // (5)
                mbar_wait(&bars.uw_ready[c], par, &dead, a.status);
                __syncwarp();
                tc_fence_after_sync();
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        umma_bf16_ts(tm + kTmC + 128 * c, tm + kTmU + 64 * c + 32 * (k >> 1) + 8 * (k & 1), dK + ((k * 16 * 128) >> 4), id5, true);
                    umma_commit(&bars.ds_done[c]);
                    if (c == 1) umma_commit(&bars.k_free[b % kKStages]);
                }
                __syncwarp();
            }
        }
    } else if (warp >= 16) {
        // ======================================================= W warps: -W^T -> bf16 tile [d_k][64 tokens], 128-byte rows: B operand of (2W)
        const int x = tid - 512;   // TMEM lane: key channel of W^T
#pragma unroll 1
        for (int b = 0; b < nblk; ++b) {
            mbar_wait(&bars.w_done, b & 1, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
#pragma unroll 1
            for (int q = 0; q < 2; ++q) {
                uint32_t rr[32], w[16];
                tmem_ld32(lane_base + kTmW + 32 * q, rr);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 16; ++e) w[e] = pack_bf16(__uint_as_float(rr[2 * e]), __uint_as_float(rr[2 * e + 1]));
                // the tile was read by (2W) of block b-1
                if (q == 0 && b >= 1) mbar_wait(&bars.w_free, (b - 1) & 1, &dead, a.status);
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    *reinterpret_cast<uint4 *>(sm + kOffW + sw128_offset(x, 4 * q + c)) = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
            }
            tc_fence_before_sync();
            fence_async_smem();
            warp_arrive(&bars.w_ready);
        }
    } else if (warp >= 12) {
        // ======================================================= prep warpgroup: the inverse and its operands, ahead of the chains
        // the X operands start as zeros: only entries on or below the block diagonal are ever written
        for (int e = tid - 384; e < 3 * kC * 128 / 16; e += 128) reinterpret_cast<uint4 *>(sm + kOffX)[e] = make_uint4(0u, 0u, 0u, 0u);
        named_bar_sync(1, 128);
#pragma unroll 1
        for (int b = 0; b < nblk; ++b)
            invert_block(bars, b, sm + kOffF, reinterpret_cast<float *>(sm + kOffD), sm + kOffX + (b & 1) * (kC * 128), sm + kOffX2,
                         gb + (b & 3) * kGbFloats + kGbX1, warp & 3, lane, &dead, a);
    } else if (warp >= 8) {
        // ======================================================= mask warps: thread = row of K K^T
#pragma unroll 1
        for (int b = 0; b < nblk; ++b) {
            mbar_wait(&bars.gb_ready[b & 3], (b >> 2) & 1, &dead, a.status);
            mask_a(bars, b, lane_base + kTmG, gb + (b & 3) * kGbFloats, sm + kOffF, reinterpret_cast<float *>(sm + kOffD), tid & 63, &dead, a);
        }
    } else {
        // ======================================================= chain warps: lane = column j of S and T, `half` = token / row half
        const int j = tid & 127, half = warp >> 2;
        unsigned char *tile = sm + kOffC + half * (kD * 128);   // columns 64 half .. of the bf16 tile of S
        // zero and the identity, times 2^R of block 0
        mbar_wait(&bars.gb_ready[0], 0, &dead, a.status);
        {
            const float fc = ex2(0.5f * gb[kGbExp]), fa = ex2(0.5f * gb[kGbExp + 1]);
#pragma unroll 1
            for (int q = 0; q < 8; ++q) {
                float v[16];
                uint32_t rr[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    v[c] = q >= 4 && 64 * half + 16 * (q & 3) + c == j ? 1.f : 0.f;
                    rr[c] = __float_as_uint(v[c] * fa * fa);
                    v[c] *= fc * fc;
                }
                tmem_st16(lane_base + kTmC + 128 * (q >> 2) + 64 * half + 16 * (q & 3), rr);
                store_row_chunks(tile + (q >> 2) * kCTile, j, 2 * (q & 3), v);
            }
            tmem_st_wait();
            tc_fence_before_sync();
            fence_async_smem();
            warp_arrive(&bars.st_ready[0]);
            warp_arrive(&bars.st_ready[1]);
        }
#pragma unroll 1
        for (int b = 0; b < nblk; ++b) {
            const uint32_t par = b & 1;
            const float *sc = gb + (b & 3) * kGbFloats;
            const bool exact = sc[kGbExp + 3] != 0.f;
            // u_t[j], tokens 32*half..+31 -> bf16 pairs over the first 16 of this thread's own 32 columns: the operand of (5)
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
                const uint32_t tu = lane_base + kTmU + 64 * c + 32 * half;
                mbar_wait(&bars.u_done[c], par, &dead, a.status);
                __syncwarp();
                tc_fence_after_sync();
                if (exact) {
                    u_operands_exact(tu, sc + kGbW + 32 * half, false);
                } else {
                    uint32_t rr[32], w[16];
                    tmem_ld32(tu, rr);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e) w[e] = pack_bf16(__uint_as_float(rr[2 * e]), __uint_as_float(rr[2 * e + 1]));
                    tmem_st16(tu, w);
                }
                tmem_st_wait();
                tc_fence_before_sync();
                warp_arrive(&bars.uw_ready[c]);
            }
            // new rows 64*half..+63: bf16 for the next block (the fp32 values stay as they are unless their scale has to change),
            // or the result at the end
            const bool last = b + 1 == nblk;
            float2 into = make_float2(0.f, 0.f);
            if (!last) {
                mbar_wait(&bars.gb_ready[(b + 1) & 3], ((b + 1) >> 2) & 1, &dead, a.status);
                into = *reinterpret_cast<const float2 *>(gb + ((b + 1) & 3) * kGbFloats + kGbExp);
            }
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
                const uint32_t tc_ = lane_base + kTmC + 128 * c + 64 * half;
                unsigned char *t = tile + c * kCTile;
                mbar_wait(&bars.ds_done[c], par, &dead, a.status);
                __syncwarp();
                tc_fence_after_sync();
                if (last) {
                    if (!dead) store_carried(tc_, (c ? a.tr_out : a.S_T) + obase + static_cast<size_t>(64 * half) * kD + j, ex2(0.5f * sc[kGbExp + 2]));
                    continue;
                }
                if (into.x == 0.f && into.y == 0.f) {
#pragma unroll 1
                    for (int q = 0; q < 2; ++q) {
                        uint32_t rr[32];
                        tmem_ld32(tc_ + 32 * q, rr);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            *reinterpret_cast<uint4 *>(t + sw128_offset(j, 4 * q + e)) =
                                make_uint4(pack_bf16(__uint_as_float(rr[8 * e]), __uint_as_float(rr[8 * e + 1])), pack_bf16(__uint_as_float(rr[8 * e + 2]), __uint_as_float(rr[8 * e + 3])),
                                           pack_bf16(__uint_as_float(rr[8 * e + 4]), __uint_as_float(rr[8 * e + 5])), pack_bf16(__uint_as_float(rr[8 * e + 6]), __uint_as_float(rr[8 * e + 7])));
                    }
                } else {
                    rescale_carried(tc_, t, j, into.x, into.y);
                }
                tc_fence_before_sync();
                fence_async_smem();
                warp_arrive(&bars.st_ready[c]);
            }
            warp_arrive(&bars.chain_done[b & 3]);
        }
    }
    grace_after_timeout(&dead);
    __syncwarp();
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tm, kTmemCols);
}

}  // namespace

cudaError_t launch_gdn_build_tensor(const GdnArgs &a, cudaStream_t s) {
    CUtensorMap mapK, mapV;
    const uint64_t rows = static_cast<uint64_t>(a.T_total);
    const uint64_t k_inner = static_cast<uint64_t>(a.H_k) * kD, v_inner = static_cast<uint64_t>(a.H_v) * kD;
    if (rows == 0) {
        // no token anywhere: no CTA touches a tile (and a map of zero rows cannot be encoded)
        memset(&mapK, 0, sizeof(mapK));
        mapV = mapK;
    } else if (!make_tensor_map_2d(&mapK, a.k, 2, k_inner, rows, k_inner * 2, 64, kC, true) ||
               !make_tensor_map_2d(&mapV, a.v, 2, v_inner, rows, v_inner * 2, 64, kC, true)) {
        return cudaErrorInvalidValue;
    }
    const cudaError_t e = cudaFuncSetAttribute(gdn_build_tensor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    return launch_chained(gdn_build_tensor_kernel, dim3(a.H_v, a.n_seq), kThreads, kSmemBytes, s, a, mapK, mapV);
}

}  // namespace lkv
