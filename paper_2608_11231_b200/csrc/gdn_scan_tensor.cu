// Chunkwise Gated DeltaNet scan on the 5th-generation tensor cores (Eq. 1 with Eq. 3), for
// d_k = d_v = 128 and bf16 q/k/v/o.  One CTA owns one (sequence, value head) and walks the
// sequence in blocks of 64 tokens, carrying the state on chip.
//
// Everything is held transposed so that every tensor-core tile has M = d_v = 128 rows (all 128
// TMEM lanes): lane j owns state column j.  The decays stay out of the contractions: with l_t the running sum of g of a block
// in log2 units and R the block's scale exponent, the state is carried as S^ = 2^R S and the pseudo-values as u^_t =
// 2^{R - l_t} u_t, which makes the recurrence of a block the plain delta rule on v^_t = 2^{R - l_t} v_t, and R moves to
// R - l_C from block to block without touching the state.  Per block:
//   (1) G    = [Q;K] K^T             rows 0..63: q_t.k_i, rows 64..127: k_t.k_i            tcgen05
//       Ps   = tril(Q K^T), A = beta tril(K K^T, -1), its 8x8 diagonal blocks inverted     mask warps
//       M    = (I + A)^{-1}          by doubling: 8 -> 16 in fp32, 16 -> 32 -> 64 by fp16 block products
//       X1   = M diag(beta 2^{R - l}), X2 = -M diag(beta)      bf16 operands               prep warps
//   (W) W^T  = K^T X2^T              -> bf16 tile                                          tcgen05, W / output warps
//  (3a) U^T  = V^T X1^T              the part of the solve that does not depend on S       tcgen05
//  (2W) U^T += S^T W^T               u^ = X1 V - M diag(beta) K S^                         tcgen05 (A = bf16 S^T in TMEM)
//       u^ -> bf16 pairs in place                                                          chain warps
//   (5) S^T += u^T K                 fp32 state accumulated in TMEM                        tcgen05 (A from TMEM)
//       S^T -> bf16 pairs in TMEM for (2W)/(2Q) of the next block                          chain warps
//  (2Q) O^T  = S^T Q^T,  (7) O^T += u^T Ps^T                                               tcgen05 (A from TMEM)
//       o_t  = scale 2^{l_t - R} O_t -> bf16 tile -> TMA store                             W / output warps
// The block-to-block chain is (2W) -> u -> (5) -> state copy: two tensor-memory to tensor-memory conversions, no
// multiplication, no shared memory and no proxy fence on it.  Everything else runs up to two blocks ahead of it ((1), mask,
// inverse, W, (3a)) or hangs off it ((2Q), (7), outputs).  A padded token (beyond the sequence end) has g = 0 and beta = 0: the
// identity step.
// R goes back to 0 when 2^R would leave its range (the state is rescaled then), and a block whose own decay is beyond 2^80 runs
// in an "exact" form: R = 0, A and Ps carry 2^{l_t - l_i} element by element, X2 takes 2^{l_i}, Q is scaled in its tile, and (5)
// and (7) get an operand each.  Same roles, same barriers.  What the mask warps add for it sits in their loops (the loads, packing and
// stores around it are shared: as functions beside the loops it cost instruction fetch, 740 -> 720 us on the case below), Q
// is scaled by the mask warps, off the chain.  32 sequences x 2048 tokens, 32 heads, log2 units of decay per token: 0.1 481 us, 0.5 503,
// 1.0 575, 1.3 (both forms in turn) 793, 4 758, 8 728; with the exact form written for rare use 485, 565, 639, 1382, 1438, 1438.
//
// Warps 0-7 chain (lane = state column, warpgroup = half of the tokens / state rows), 8-11 mask epilogue of (1), 12-15 prep
// (the inverse), 16 TMA loads of V and the stores of the output tiles, 17 MMA issue of the chain, 18 MMA issue of (1) and (W),
// 19 TMA loads of Q and K and the per-block scalars, 20-23 W and outputs.  All waits on mbarriers are bounded.
//
// What bounds it: neither a pipe (tensor 36 %, issue slots 39 % with every SM busy) nor one chain, but the latency of about
// 6 K instructions per block in ten programs that share an SM: mask 1.7 K cycles, inverse 3.0 K, chain 2.1 K of a block period of
// 3.3 K -- and instruction fetch: 7 KB less code in the issuing and scalar warps (each piece of code once, its loop started a
// block early instead of a copy before it) took 32 x 4096 tokens from 992 to 940 us.  Hence small rolled loops, fp16 storage of what
// is an fp16 operand, ldmatrix / movmatrix instead of fp32 round trips, and few warps: outputs in a warpgroup of their own, or the last
// merge of the inverse moved to the W warps, made every program slower (8 % and 17 % on one sequence).  Measured on B200, 32
// value heads: one sequence of 8192 tokens 311 -> 237 us as one chain, 32 x 4096 tokens 1172 -> 940 us against the form that gates
// the products and solves for u in the chain (three conversions).
#include <string.h>

#include "gdn_blocks.cuh"

namespace lkv {

namespace {

constexpr int kThreads = 768;

// shared-memory map (bytes, after 1024-byte alignment); operand tiles have 128-byte rows, 128-byte swizzle
constexpr int kQKStage = 4 * kC * 128;                 // [Q_kb0 | K_kb0 | Q_kb1 | K_kb1], each [64 tokens x 128 B]
                                                       // once (2Q) has read them the Q tiles hold the block's output tile,
                                                       // [2][64 tokens x 128 B] bf16, for the TMA store
constexpr int kQKStages = 4;                           // a stage is held from its load until that store: four block periods
constexpr int kVStage = 2 * kC * 128;                  // [V_jb0 | V_jb1], each [64 tokens x 128 B]
constexpr int kOffV = kQKStages * kQKStage;            // one V stage
constexpr int kOffX = kOffV + kVStage;                 // X1 bf16 [64 rows t x 128 B], double-buffered
constexpr int kOffX2 = kOffX + 2 * kC * 128;           // X2 likewise, one buffer
constexpr int kOffW = kOffX2 + kC * 128;               // -W^T bf16 [128 rows d_k x 64 tokens]
constexpr int kOffP = kOffW + kD * 128;                // Ps bf16 [64 rows t x 128 B], two buffers
constexpr int kOffF = kOffP + 2 * kC * 128;
constexpr int kOffD = kOffF + 2 * kFBytes;
constexpr int kOffGb = kOffD + kC * kLdD * 4;          // per-block scalars, four buffers
constexpr int kSmemUsed = kOffGb + 4 * kGbFloats * 4;  // from the 1024-byte aligned base
constexpr int kSmemBytes = kSmemUsed + 1024;
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");

// tensor-memory map (columns)
constexpr uint32_t kTmS = 0;      // 128: S^T fp32
constexpr uint32_t kTmSb = 128;   // 64: S^T as bf16 pairs (A operand of (2W), (2Q))
constexpr uint32_t kTmW = 192;    // 64: -W^T fp32
constexpr uint32_t kTmU = 256;    // 64: U^T fp32; in place u as bf16 pairs (columns 0..15 and 32..47; an exact block's second operand in 16..31 and 48..63)
constexpr uint32_t kTmO = 320;    // 2 x 64: O^T of the even / odd blocks
constexpr uint32_t kTmG = 448;    // 64
constexpr uint32_t kTmemCols = 512;

struct Bars {
    // single-arrival barriers: TMA transactions and tcgen05.commit
    uint64_t full_qk[4], full_v, v_free, g_done, w_done, w_free, x2_free, u_done, ds_done, o_mma_done[2], p_free[2], x1_free[2];
    // one arrival per warp: the four prep warps; the four output warps
    uint64_t m_ready[2], d_free, w_ready, o_done[4];
    // the two warps of a half of the mask warpgroup; (5) and the output store
    uint64_t a_ready[2], p_ready[2], tiles_free_qk[4];
    // the scalar warp
    uint64_t gb_ready[4];
    // the eight chain warps
    uint64_t uw_ready, st_ready, chain_done[4];
};
constexpr int kBars1 = 18, kBars4 = 8, kBars2 = 8, kBarsS = 4, kBars8 = 6;
static_assert(sizeof(Bars) == 8 * (kBars1 + kBars4 + kBars2 + kBarsS + kBars8), "barrier table");

// Exact block: row t of the Q tile multiplied in place by f.
static __device__ __noinline__ void scale_q_row(unsigned char *stage, int t, float f) {
    unsigned char *qt = stage + t * 128;
    const __nv_bfloat162 f2 = __float2bfloat162_rn(f);
#pragma unroll 1
    for (int kb = 0; kb < 2; ++kb, qt += 2 * kC * 128) {
        uint4 v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = *reinterpret_cast<uint4 *>(qt + ((c ^ (t & 7)) << 4));
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            __nv_bfloat162 *e = reinterpret_cast<__nv_bfloat162 *>(&v[c]);
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = __hmul2(e[i], f2);
            *reinterpret_cast<uint4 *>(qt + ((c ^ (t & 7)) << 4)) = v[c];
        }
    }
}

// Rows of a ragged last block go straight to global memory: 16 tokens of one state column per call, read from
// tensor memory and scaled here.
__device__ __noinline__ void store_o_partial(uint32_t taddr, const float *e, __nv_bfloat16 *orow, size_t tstride, int n_left) {
    uint32_t pu[16];
    tmem_ld16(taddr, pu);
    tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < 16; ++c)
        if (c < n_left) orow[c * tstride] = __float2bfloat16_rn(__uint_as_float(pu[c]) * e[c]);
}
// 64 rows of the state from row 64 half on: times 2^copy_exp as bf16 pairs beside them, times 2^acc_exp in place (2^copy_exp brings it back
// to a small scale, what an exact block takes off on top of that may vanish).  One block in several needs it.
__device__ __noinline__ void rescale_state(uint32_t tm_s, uint32_t tm_sb, float copy_exp, float acc_exp) {
    const float fc = ex2(copy_exp), fa = ex2(acc_exp - copy_exp);
#pragma unroll 1
    for (int q = 0; q < 2; ++q) {
        uint32_t rr[32], w[16];
        tmem_ld32(tm_s + 32 * q, rr);
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < 32; ++c) rr[c] = __float_as_uint(__uint_as_float(rr[c]) * fc);
#pragma unroll
        for (int e = 0; e < 16; ++e) w[e] = pack_bf16(__uint_as_float(rr[2 * e]), __uint_as_float(rr[2 * e + 1]));
        tmem_st16(tm_sb + 16 * q, w);
#pragma unroll
        for (int c = 0; c < 32; ++c) rr[c] = __float_as_uint(__uint_as_float(rr[c]) * fa);
        tmem_st32(tm_s + 32 * q, rr);
    }
}
__global__ void __launch_bounds__(kThreads, 1)
gdn_scan_tensor_kernel(const __grid_constant__ GdnArgs a, const __grid_constant__ CUtensorMap mapQ,
                       const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV,
                       const __grid_constant__ CUtensorMap mapO) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);   // an offset, not a cast: the compiler keeps shared-memory addressing
    __shared__ Bars bars;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int dead;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_launch();
    if (a.cu.ptr) pdl_wait();   // the index list is in global memory
    const int h = blockIdx.x, seq = a.cu[a.n_ranges + 1 + blockIdx.y];   // launch order: longest sequence first
    const bool tr = seq >= a.tr_first;                                    // transition sequence
    const int rg = tr ? seq - a.tr_first + a.tr_src0 : seq;
    const bool s0_id = a.s0_identity || tr;
    const int hk = h / (a.H_v / a.H_k);
    const int t_begin = a.cu[rg], t_end = a.cu[rg + 1];
    const int nblk = (t_end - t_begin + kC - 1) / kC;
    const size_t sbase = (static_cast<size_t>(seq) * a.H_v + h) * kD * kD;
    // this sequence's initial state (nullptr = zero), and where its final state goes (nullptr = nowhere; a transition sequence
    // may have a buffer of its own)
    auto initial_state = [&]() -> const float * {
        const float *p = seq < a.n_s0 ? a.S0 : a.S0_more;
        return p ? p + (static_cast<size_t>(seq < a.n_s0 ? seq : seq - a.n_s0) * a.H_v + h) * kD * kD : nullptr;
    };
    auto final_state = [&](size_t &base) -> float * {
        const bool own = tr && a.tr_out != nullptr;
        base = (static_cast<size_t>(own ? seq - a.tr_first : seq - a.st_first) * a.H_v + h) * kD * kD;
        return own ? a.tr_out : seq >= a.st_first ? a.S_T : nullptr;
    };
    const bool has_v = a.v != nullptr && !tr, has_o = a.o != nullptr && !tr;

    if (nblk == 0) {  // empty sequence: hand the state through untouched
        pdl_wait();
        size_t obase;
        float *ST = final_state(obase);
        const float *S0 = initial_state();
        if (ST && (ST != a.S0 || s0_id || a.S_add))
            hand_through(ST, obase, a.st_bf16, s0_id, s0_id ? nullptr : S0, a.S_add ? a.S_add + sbase : nullptr);
        return;
    }
    if (tid == 0) {
        dead = 0;
        uint64_t *bp = &bars.full_qk[0];
        for (int i = 0; i < kBars1; ++i) mbar_init(bp++, 1);
        for (int i = 0; i < kBars4; ++i) mbar_init(bp++, 4);
        for (int i = 0; i < kBars2; ++i) mbar_init(bp++, 2);
        for (int i = 0; i < kBarsS; ++i) mbar_init(bp++, 1);
        for (int i = 0; i < kBars8; ++i) mbar_init(bp++, 8);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(&tmem_base, kTmemCols);
    pdl_wait();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tm = tmem_base;
    float *gb = reinterpret_cast<float *>(sm + kOffGb);

    if (warp == 16) {
        // ======================================================= TMA loads of V and store of the output tiles.  Here and in the
        // other single-issue roles the whole warp walks the loop and one elected lane issues: the operands of these
        // instructions live in registers that the warp shares, so its lanes stay together.
#pragma unroll 1
        for (int b = -1; b <= nblk; ++b) {
            if (warp_dead(&dead)) break;   // a wait ran out: nothing more is issued
            const int row = t_begin + b * kC;
            // V of block b+1 as soon as (3a) of block b has read the stage; without v (read as zeros) nothing is loaded
            if (has_v && b + 1 < nblk) {
                if (b >= 0) mbar_wait(&bars.v_free, b & 1, &dead, a.status);
                __syncwarp();
                if (elect_one()) {
                    mbar_expect_tx(&bars.full_v, kVStage);
                    for (int jb = 0; jb < 2; ++jb) {
                        tma_load_2d(sm + kOffV + jb * kC * 128, &mapV, h * kD + jb * 64, row + kC, &bars.full_v);
                        if (b + 3 < nblk) tma_prefetch_l2_2d(&mapV, h * kD + jb * 64, row + 3 * kC);
                    }
                }
                __syncwarp();
            }
            // output tile of block b-1 (whole blocks only), staged over its Q tiles
            if (b >= 1) {
                const int s4 = (b - 1) % kQKStages;
                mbar_wait(&bars.o_done[(b - 1) & 3], ((b - 1) >> 2) & 1, &dead, a.status);
                const bool store = has_o && row <= t_end && !warp_dead(&dead);
                __syncwarp();
                if (elect_one()) {
                    if (store) {
                        for (int jb = 0; jb < 2; ++jb)
                            tma_store_2d(&mapO, sm + s4 * kQKStage + jb * 2 * kC * 128, h * kD + jb * 64, row - kC);
                        tma_store_commit();
                        tma_store_wait_read();
                    }
                    mbar_arrive(&bars.tiles_free_qk[s4]);
                }
                __syncwarp();
            }
        }
        if (elect_one()) tma_store_wait_all();
        __syncwarp();
    } else if (warp == 19) {
        // ======================================================= TMA loads of the Q and K tiles (four stages) and the scalars of a block:
        // lane = tokens 2 lane, 2 lane + 1
        auto fetch_gb = [&](int b, float2 &gv, float2 &bv) {
            const int t = t_begin + b * kC + 2 * lane;
            gv = make_float2(0.f, 0.f); bv = make_float2(0.f, 0.f);
            if (b < nblk && t < t_end) {
                gv.x = a.g[static_cast<size_t>(t) * a.H_v + h];
                bv.x = a.beta[static_cast<size_t>(t) * a.H_v + h];
            }
            if (b < nblk && t + 1 < t_end) {
                gv.y = a.g[static_cast<size_t>(t + 1) * a.H_v + h];
                bv.y = a.beta[static_cast<size_t>(t + 1) * a.H_v + h];
            }
        };
        float2 gv_next = make_float2(0.f, 0.f), bv_next = gv_next;
        float R = 0.f;   // the state is held times 2^R
#pragma unroll 1
        for (int b = -1; b < nblk; ++b) {
            const float2 gv = gv_next, bv = bv_next;
            fetch_gb(b + 1, gv_next, bv_next);   // in flight while this block is prepared
            if (b < 0) continue;
            if (warp_dead(&dead)) break;   // a wait ran out: nothing more is issued
            const int s4 = b % kQKStages;
            const int row = t_begin + b * kC;
            unsigned char *base = sm + s4 * kQKStage;
            // the tiles of block b go into the stage that (5) and the output store of block b-4 have released.  The ring
            // cannot hide the DRAM latency: the tiles of block b+4 are pulled into L2 now.
            if (b >= kQKStages) mbar_wait(&bars.tiles_free_qk[s4], ((b - kQKStages) / kQKStages) & 1, &dead, a.status);
            __syncwarp();
            if (elect_one()) {
                mbar_expect_tx(&bars.full_qk[s4], kQKStage);
#pragma unroll 1
                for (int kb = 0; kb < 2; ++kb) {
                    tma_load_2d(base + kb * 2 * kC * 128, &mapQ, hk * kD + kb * 64, row, &bars.full_qk[s4]);
                    tma_load_2d(base + kb * 2 * kC * 128 + kC * 128, &mapK, hk * kD + kb * 64, row, &bars.full_qk[s4]);
                    if (b + kQKStages < nblk) {
                        tma_prefetch_l2_2d(&mapQ, hk * kD + kb * 64, row + kQKStages * kC);
                        tma_prefetch_l2_2d(&mapK, hk * kD + kb * 64, row + kQKStages * kC);
                    }
                }
            }
            __syncwarp();
            // the buffer of block b was last read by the chain and the output epilogue of block b-4
            if (b >= 4) {
                mbar_wait(&bars.chain_done[b & 3], ((b - 4) >> 2) & 1, &dead, a.status);
                mbar_wait(&bars.o_done[b & 3], ((b - 4) >> 2) & 1, &dead, a.status);
            }
            __syncwarp();
            float *sc = gb + (b & 3) * kGbFloats;
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
            *reinterpret_cast<float2 *>(sc + kGbE + t) = exact ? make_float2(a.scale, a.scale) : make_float2(a.scale * ex2(c0 - Rn), a.scale * ex2(c1 - Rn));
            if (exact) *reinterpret_cast<float2 *>(sc + kGbW + t) = make_float2(ex2(last - c0), ex2(last - c1));
            const float in = Rn - R;
            R = exact ? 0.f : Rn - last;
            if (lane == 0) *reinterpret_cast<float4 *>(sc + kGbExp) = make_float4(in, exact ? in + last : in, -R, exact ? 1.f : 0.f);
            warp_arrive(&bars.gb_ready[b & 3]);
        }
    } else if (warp == 18) {
        // ======================================================= MMA issue of (1) and W
        constexpr uint32_t idG = umma_idesc(kFmtBF16, false, false, 128, 64);
        constexpr uint32_t idW = umma_idesc(kFmtBF16, true, false, 128, 64);   // A = K tile read MN-major
        const uint64_t dX2 = umma_desc(smem_u32(sm + kOffX2), 0, 1024);
        // -W^T = K^T X2^T of block b, once its inverse is there and the output warps have drained the W columns
        auto issue_w = [&](int b) {
            if (b >= 1) mbar_wait(&bars.w_ready, (b - 1) & 1, &dead, a.status);
            mbar_wait(&bars.m_ready[b & 1], (b >> 1) & 1, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
            const uint64_t dKm = umma_desc(smem_u32(sm + (b % kQKStages) * kQKStage + kC * 128), 2 * kC * 128, 1024);
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 4; ++k) umma_bf16(tm + kTmW, dKm + ((k * 16 * 128) >> 4), dX2 + 2 * k, idW, k > 0);
                umma_commit(&bars.w_done);
                umma_commit(&bars.x2_free);
            }
            __syncwarp();
        };
        auto issue_g = [&](int b) {
            const int s3 = b % kQKStages;
            // (1) of block b: the mask epilogue of block b-1 has drained the G columns
            if (b >= 1) {
                mbar_wait(&bars.a_ready[(b - 1) & 1], ((b - 1) >> 1) & 1, &dead, a.status);
                mbar_wait(&bars.p_ready[(b - 1) & 1], ((b - 1) >> 1) & 1, &dead, a.status);
            }
            mbar_wait(&bars.full_qk[s3], (b / kQKStages) & 1, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
            const uint64_t dQK = umma_desc(smem_u32(sm + s3 * kQKStage), 0, 1024);
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint64_t off = ((k >> 2) * (2 * kC * 128) + (k & 3) * 32) >> 4;
                    umma_bf16(tm + kTmG, dQK + off, dQK + off + ((kC * 128) >> 4), idG, k > 0);
                }
                umma_commit(&bars.g_done);
            }
            __syncwarp();
        };
#pragma unroll 1
        for (int b = 0; b <= nblk; ++b) {
            if (warp_dead(&dead)) break;   // a wait ran out: nothing more is issued
            if (b < nblk) issue_g(b);
            if (b >= 1) issue_w(b - 1);
        }
    } else if (warp == 17) {
        // ======================================================= MMA issue of (3a), (2W), (2Q), (5), (7)
        constexpr uint32_t idN64 = umma_idesc(kFmtBF16, false, false, 128, 64);    // (2Q), (7)
        constexpr uint32_t idW = umma_idesc(kFmtBF16, true, false, 128, 64);       // (3a): A = V tile read MN-major
        constexpr uint32_t id2W = umma_idesc(kFmtBF16, false, true, 128, 64);      // B = -W^T tile read MN-major
        constexpr uint32_t id5 = umma_idesc(kFmtBF16, false, true, 128, 128);      // B = K tile read MN-major
        const uint64_t dW = umma_desc(smem_u32(sm + kOffW), 0, 1024);
        // (3a) U^T = V^T X1^T of block b; the U columns were read by (5) and (7) of block b-1, issued before
        auto issue_3a = [&](int b) {
            if (!has_v) return;
            mbar_wait(&bars.full_v, b & 1, &dead, a.status);
            mbar_wait(&bars.m_ready[b & 1], (b >> 1) & 1, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
            const uint64_t dV = umma_desc(smem_u32(sm + kOffV), kC * 128, 1024);
            const uint64_t dX = umma_desc(smem_u32(sm + kOffX + (b & 1) * (kC * 128)), 0, 1024);
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 4; ++k) umma_bf16(tm + kTmU, dV + ((k * 16 * 128) >> 4), dX + 2 * k, idW, k > 0);
                umma_commit(&bars.v_free);
                umma_commit(&bars.x1_free[b & 1]);
            }
            __syncwarp();
        };
        auto chain_block = [&](int b) {
            const uint32_t par = b & 1;
            const uint32_t qk = smem_u32(sm + (b % kQKStages) * kQKStage);
            const uint64_t dQ = umma_desc(qk, 0, 1024), dKmn = umma_desc(qk + kC * 128, 2 * kC * 128, 1024);
            // (2W) U^T -= S^T W^T: needs the block's W tile and bf16 state
            mbar_wait(&bars.w_ready, par, &dead, a.status);
            mbar_wait(&bars.st_ready, par, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 8; ++k) umma_bf16_ts(tm + kTmU, tm + kTmSb + 8 * k, dW + ((k * 16 * 128) >> 4), id2W, has_v || k > 0);
                umma_commit(&bars.u_done);
                umma_commit(&bars.w_free);
            }
            __syncwarp();
            // (2Q) O = S^T Q^T while the chain warps work on U: O columns drained with the outputs of block b-2.  An exact
            // block has had its Q tile scaled.
            const bool exact = gb[(b & 3) * kGbFloats + kGbExp + 3] != 0.f;
            if (has_o) {
                if (exact) mbar_wait(&bars.p_ready[par], (b >> 1) & 1, &dead, a.status);   // with Ps its Q tile is ready
                if (b >= 2) mbar_wait(&bars.o_done[(b - 2) & 3], ((b - 2) >> 2) & 1, &dead, a.status);
                __syncwarp();
                tc_fence_after_sync();
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        umma_bf16_ts(tm + kTmO + 64 * par, tm + kTmSb + 8 * k, dQ + (((k >> 2) * (2 * kC * 128) + (k & 3) * 32) >> 4), idN64, k > 0);
                }
                __syncwarp();
            }
            // (5) S^T += u^T K
            mbar_wait(&bars.uw_ready, par, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    umma_bf16_ts(tm + kTmS, tm + kTmU + 32 * (k >> 1) + 8 * (k & 1), dKmn + ((k * 16 * 128) >> 4), id5, true);
                umma_commit(&bars.ds_done);
                umma_commit(&bars.tiles_free_qk[b % kQKStages]);
            }
            __syncwarp();
            // (7) O += u^T Ps^T; an exact block has an operand of its own here, behind that of (5)
            if (has_o) mbar_wait(&bars.p_ready[par], (b >> 1) & 1, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
            if (elect_one()) {
                if (has_o) {
                    const uint32_t u7 = tm + kTmU + (exact ? 16 : 0);
                    const uint64_t dP = umma_desc(smem_u32(sm + kOffP + par * (kC * 128)), 0, 1024);
#pragma unroll
                    for (int k = 0; k < 4; ++k) umma_bf16_ts(tm + kTmO + 64 * par, u7 + 32 * (k >> 1) + 8 * (k & 1), dP + 2 * k, idN64, true);
                    umma_commit(&bars.p_free[par]);
                }
                umma_commit(&bars.o_mma_done[par]);
            }
            __syncwarp();
        };
#pragma unroll 1
        for (int b = -1; b < nblk; ++b) {
            if (warp_dead(&dead)) break;
            if (b >= 0) chain_block(b);
            if (b + 1 < nblk) issue_3a(b + 1);
        }
    } else if (warp >= 20) {
        // ======================================================= W and output warpgroup
        const int x = tid - 640;   // TMEM lane: key channel of W^T, feature of O^T
        const uint32_t lane_base = tm + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        // outputs of block b: O^T (complete once (7) has run) -> bf16 tile [token][j], lane = j
        __nv_bfloat16 *o = static_cast<__nv_bfloat16 *>(a.o);
        const size_t tstride = static_cast<size_t>(a.H_v) * kD;
        auto o_epilogue = [&](int b) {
            mbar_wait(&bars.o_mma_done[b & 1], (b >> 1) & 1, &dead, a.status);
            tc_fence_after_sync();
            const int t0 = t_begin + b * kC;
            const int n = min(kC, t_end - t0);
            const float *ge = gb + (b & 3) * kGbFloats + kGbE;
            if (has_o && (n == kC || !dead)) {
                if (n != kC) {
                    // ragged last block: straight to global memory, 16 tokens of one state column per call
#pragma unroll 1
                    for (int q = 0; q < 4; ++q)
                        store_o_partial(lane_base + kTmO + 64 * (b & 1) + 16 * q, ge + 16 * q, o + (static_cast<size_t>(t0 + 16 * q) * a.H_v + h) * kD + x,
                                        tstride, n - 16 * q);
                } else {
                    // whole block: stage the tile over the Q tiles of this block, which (2Q) has finished reading, in the layout of
                    // the tensor map (two halves of 64 features, 128-byte rows, 128-byte swizzle); the store warp writes it out
                    // with TMA.  O^T leaves tensor memory in accumulator layout (thread = feature, register pair = two tokens) and
                    // is stored transposed, 16 features x 16 tokens per instruction.
                    unsigned char *os = sm + (b % kQKStages) * kQKStage + (warp & 2 ? 2 * kC * 128 : 0);
                    const int m = lane >> 3, i = lane & 7;
#pragma unroll 1
                    for (int lh = 0; lh < 2; ++lh) {
                        uint32_t pu[32];
                        tmem_ld_16x256b_x8(lane_base + (static_cast<uint32_t>(16 * lh) << 16) + kTmO + 64 * (b & 1), pu);
                        tmem_ld_wait();
                        const int chunk = 4 * (warp & 1) + 2 * lh + (m & 1);   // 16-byte piece of the 128-byte row: 8 features
                        const uint32_t row_addr = smem_u32(os) + (8 * (m >> 1) + i) * 128 + ((chunk ^ i) << 4);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {   // tokens 16 kk .. 16 kk + 15
                            uint32_t w[4];
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                const float2 e = *reinterpret_cast<const float2 *>(ge + 16 * kk + 8 * k + 2 * (lane & 3));
#pragma unroll
                                for (int u = 0; u < 2; ++u)
                                    w[2 * k + u] = pack_bf16(__uint_as_float(pu[8 * kk + 4 * k + 2 * u]) * e.x, __uint_as_float(pu[8 * kk + 4 * k + 2 * u + 1]) * e.y);
                            }
                            stmatrix_x4_trans(row_addr + 16 * kk * 128, w[0], w[1], w[2], w[3]);
                        }
                    }
                }
                fence_async_smem();
            }
            tc_fence_before_sync();
            warp_arrive(&bars.o_done[b & 3]);
        };
#pragma unroll 1
        for (int b = 0; b <= nblk; ++b) {
            if (b < nblk) {
                // -W^T of block b -> bf16 tile [d_k][64 tokens], 128-byte rows: B operand of (2W), read MN-major
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
            if (b >= 1) o_epilogue(b - 1);
        }
    } else if (warp >= 12) {
        // ======================================================= prep warpgroup: the inverse and its operand, ahead of the chain
        const int x = tid - 384;                 // 0..127
        const int wq = warp & 3, gid = lane >> 2, tig = lane & 3;
        // the X operands start as zeros: only entries on or below the block diagonal are ever written
        for (int e = x; e < 3 * kC * 128 / 16; e += 128) reinterpret_cast<uint4 *>(sm + kOffX)[e] = make_uint4(0u, 0u, 0u, 0u);
        unsigned char *xb2 = sm + kOffX2;
#pragma unroll 1
        for (int b = 0; b < nblk; ++b) {
            const float *fx = gb + (b & 3) * kGbFloats + kGbX1;   // factors of the columns of X1; those of X2 follow
            unsigned char *xb1 = sm + kOffX + (b & 1) * (kC * 128);
            const uint32_t Fs = smem_u32(sm + kOffF + (b & 1) * kFBytes);
            unsigned char *Ft = sm + kOffF + (b & 1) * kFBytes + (wq >> 1) * kFTile;   // the tile with this warp's diagonal block
            float *D = reinterpret_cast<float *>(sm + kOffD) + (16 * wq) * kLdD;       // the block itself
            // ---- A comes from the mask warpgroup (epilogue of (1)), its 8x8 diagonal blocks inverted; here the rest of it turns
            // into M = (I + A)^{-1} by doubling.
            mbar_wait(&bars.a_ready[b & 1], (b >> 1) & 1, &dead, a.status);
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
                if (b >= 2 && has_v) mbar_wait(&bars.x1_free[b & 1], ((b - 2) >> 1) & 1, &dead, a.status);
                if (b >= 1) mbar_wait(&bars.x2_free, (b - 1) & 1, &dead, a.status);
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
    } else if (warp >= 8) {
        // ======================================================= mask warpgroup: epilogue of (1), as far ahead of the chain as the
        // buffers allow
        const int x = tid - 256;   // TMEM lane: 0..63 rows of Q K^T (-> Ps), 64..127 rows of K K^T (-> A)
        const int t = x & 63;
        const uint32_t lane_base = tm + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const int row_hi = (t & 32) + 31;   // last row (token) of this warp
        if (x < 32) {
            // columns 32..63 of rows 0..31 lie above the diagonal in both Ps buffers: zero them once
            float z[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) z[c] = 0.f;
#pragma unroll 1
            for (int i = 0; i < 4; ++i) store_row_chunks(sm + kOffP + (i >> 1) * (kC * 128), t, 4 + 2 * (i & 1), z);
        }
#pragma unroll 1
        for (int b = 0; b < nblk; ++b) {
            const float *sc = gb + (b & 3) * kGbFloats;
            // (Without outputs the warps of Ps leave the scalars alone: nothing that frees their buffer would wait for that read.)
            if (x >= kC || has_o) mbar_wait(&bars.gb_ready[b & 3], (b >> 2) & 1, &dead, a.status);
            if (x < kC) {
                // rows of Ps, the diagonal included.  The buffer is free once (7) of block b-2 has read it.
                if (b >= 2 && has_o) mbar_wait(&bars.p_free[b & 1], ((b - 2) >> 1) & 1, &dead, a.status);
                mbar_wait(&bars.g_done, b & 1, &dead, a.status);
                __syncwarp();
                tc_fence_after_sync();
                unsigned char *ps = sm + kOffP + (b & 1) * (kC * 128);
                if (has_o) {
                    const bool exact = sc[kGbExp + 3] != 0.f;
                    // column groups above the diagonal for every row of this warp are never touched
#pragma unroll 1
                    for (int q = 0; 16 * q <= row_hi; ++q) {
                        const int i0 = 16 * q;
                        uint32_t rr[16];
                        tmem_ld16(lane_base + kTmG + i0, rr);
                        tmem_ld_wait();
                        float v[16];
#pragma unroll
                        for (int c = 0; c < 16; ++c) v[c] = __uint_as_float(rr[c]);
                        if (exact) apply_decay(v, sc + kGbL + i0, sc[kGbL + t]);
                        if (i0 + 31 >= row_hi) {   // the groups that the diagonal of this warp's rows passes through
#pragma unroll
                            for (int c = 0; c < 16; ++c) v[c] = (i0 + c <= t) ? v[c] : 0.f;
                        }
                        store_row_chunks(ps, t, 2 * q, v);
                    }
                    // an exact block's row of the Q tile times 2^l for (2Q), which waits for it; (1) has read the tile
                    if (exact) {
                        mbar_wait(&bars.full_qk[b % kQKStages], (b / kQKStages) & 1, &dead, a.status);   // this thread reads what the TMA wrote
                        scale_q_row(sm + (b % kQKStages) * kQKStage, t, ex2(sc[kGbL + t]));
                    }
                }
                tc_fence_before_sync();
                fence_async_smem();
                warp_arrive(&bars.p_ready[b & 1]);
            } else {
                const bool exact = sc[kGbExp + 3] != 0.f;
                // rows of A, strictly lower.  F is free once block b-2 has been inverted, D once the diagonal blocks of block b-1 are.
                if (b >= 2) mbar_wait(&bars.m_ready[b & 1], ((b - 2) >> 1) & 1, &dead, a.status);
                if (b >= 1) mbar_wait(&bars.d_free, (b - 1) & 1, &dead, a.status);
                mbar_wait(&bars.g_done, b & 1, &dead, a.status);
                __syncwarp();
                tc_fence_after_sync();
                unsigned char *fb = sm + kOffF + (b & 1) * kFBytes + (t & 31) * kLdF;   // this row of the first tile
                float *drow = reinterpret_cast<float *>(sm + kOffD) + t * kLdD;
                const float bt = exact ? sc[kGbX1 + t] : -sc[kGbX2 + t];   // beta
                // Nothing is masked here: what lies above the 8x8 diagonal blocks is never read, and the substitution masks these
                // themselves.
#pragma unroll 1
                for (int q = 0; 32 * q <= row_hi; ++q) {
                    const int i0 = 32 * q;
                    unsigned char *frow = fb + (i0 + 31 == row_hi ? q : 2) * kFTile;
                    uint32_t rr[32];
                    tmem_ld32(lane_base + kTmG + i0, rr);
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
        }
    } else {
        // ======================================================= chain warpgroups: lane = state column j, `half` = token / row half
        const int j = tid & 127, half = warp >> 2;
        const uint32_t lane_base = tm + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        // initial state: S0[m][j], m = 64*half..+63 -> TMEM (fp32, times 2^R of block 0) and bf16 pairs.  All of it is asked for at
        // once, and before the block's scalars are waited for: 16 values a thread in registers, the others into L2 (16 requests
        // of up to 128 tokens: 56.6 -> 55.4 us).
        {
            const float *S0 = s0_id ? nullptr : initial_state();
            if (S0) {
                S0 += static_cast<size_t>(64 * half) * kD;
                for (int i = j >> 2; i < 48; i += 32) prefetch_l2(S0 + (16 + i) * kD + 32 * (j & 3));
                S0 += j;
            }
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {
                float v[16];
                if (S0) {   // one branch for the sixteen loads: they are in flight together
#pragma unroll
                    for (int c = 0; c < 16; ++c) v[c] = S0[(16 * q + c) * kD];
                } else {
#pragma unroll
                    for (int c = 0; c < 16; ++c) v[c] = s0_id && 64 * half + 16 * q + c == j ? 1.f : 0.f;
                }
                if (q == 0) mbar_wait(&bars.gb_ready[0], 0, &dead, a.status);
                const float fc = ex2(0.5f * gb[kGbExp]), fa = ex2(0.5f * gb[kGbExp + 1]);
                uint32_t rr[16], w[8];
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    rr[c] = __float_as_uint(v[c] * fa * fa);
                    v[c] *= fc * fc;
                }
                tmem_st16(lane_base + kTmS + 64 * half + 16 * q, rr);
                pack16(v, w);
                tmem_st8(lane_base + kTmSb + 32 * half + 8 * q, w);
            }
            tmem_st_wait();
            tc_fence_before_sync();
            warp_arrive(&bars.st_ready);
        }
#pragma unroll 1
        for (int b = 0; b < nblk; ++b) {
            const uint32_t par = b & 1;
            const float *sc = gb + (b & 3) * kGbFloats;
            const bool exact = sc[kGbExp + 3] != 0.f;
            // u_t[j], tokens 32*half..+31 -> bf16 pairs over the first 16 of this thread's own 32 columns: the operand of (5) and (7)
            mbar_wait(&bars.u_done, par, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
            if (exact) {
                u_operands_exact(lane_base + kTmU + 32 * half, sc + kGbW + 32 * half, has_o);
            } else {
                uint32_t rr[32], w[16];
                tmem_ld32(lane_base + kTmU + 32 * half, rr);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 16; ++e) w[e] = pack_bf16(__uint_as_float(rr[2 * e]), __uint_as_float(rr[2 * e + 1]));
                tmem_st16(lane_base + kTmU + 32 * half, w);
            }
            tmem_st_wait();
            tc_fence_before_sync();
            warp_arrive(&bars.uw_ready);
            // new state rows m = 64*half..+63: bf16 pairs for the next block (the fp32 state stays as it is unless its scale has
            // to change), or S_T at the end
            const bool last = b + 1 == nblk;
            float2 into = make_float2(0.f, 0.f);
            if (!last) {
                mbar_wait(&bars.gb_ready[(b + 1) & 3], ((b + 1) >> 2) & 1, &dead, a.status);
                into = *reinterpret_cast<const float2 *>(gb + ((b + 1) & 3) * kGbFloats + kGbExp);
            }
            mbar_wait(&bars.ds_done, par, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
            if (last) {
                size_t obase;
                float *ST = final_state(obase);
                const float ff = ex2(0.5f * sc[kGbExp + 2]);
                if (ST && !dead) {
                    const size_t mine = static_cast<size_t>(64 * half) * kD + j;
                    const float *add = a.S_add ? a.S_add + sbase + mine : nullptr;
                    obase += mine;
#pragma unroll 1
                    for (int q = 0; q < 4; ++q, obase += 16 * kD) {
                        uint32_t rr[16];
                        tmem_ld16(lane_base + kTmS + 64 * half + 16 * q, rr);
                        tmem_ld_wait();
                        float v[16];
#pragma unroll
                        for (int c = 0; c < 16; ++c) v[c] = __uint_as_float(rr[c]) * ff * ff;
                        if (add) {
#pragma unroll
                            for (int c = 0; c < 16; ++c) v[c] += add[(16 * q + c) * kD];
                        }
                        if (a.st_bf16) {
#pragma unroll
                            for (int c = 0; c < 16; ++c) reinterpret_cast<__nv_bfloat16 *>(ST)[obase + c * kD] = __float2bfloat16_rn(v[c]);
                        } else {
#pragma unroll
                            for (int c = 0; c < 16; ++c) ST[obase + c * kD] = v[c];
                        }
                    }
                }
            } else {
                if (into.x == 0.f && into.y == 0.f) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint32_t rr[32], w[16];
                        tmem_ld32(lane_base + kTmS + 64 * half + 32 * q, rr);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 16; ++e) w[e] = pack_bf16(__uint_as_float(rr[2 * e]), __uint_as_float(rr[2 * e + 1]));
                        tmem_st16(lane_base + kTmSb + 32 * half + 16 * q, w);
                    }
                } else {
                    rescale_state(lane_base + kTmS + 64 * half, lane_base + kTmSb + 32 * half, into.x, into.y);
                }
                tmem_st_wait();
                tc_fence_before_sync();
                warp_arrive(&bars.st_ready);
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

bool gdn_scan_tensor_supported(const GdnArgs &a, bool io_bf16) {
    return io_bf16 && a.d_k == kD && a.d_v == kD;
}

cudaError_t launch_gdn_scan_tensor(const GdnArgs &a, cudaStream_t s) {
    CUtensorMap mapQ, mapK, mapV, mapO;
    const uint64_t rows = static_cast<uint64_t>(a.T_total);
    const uint64_t qk_inner = static_cast<uint64_t>(a.H_k) * kD, v_inner = static_cast<uint64_t>(a.H_v) * kD;
    if (rows == 0) {
        // no token anywhere: every CTA hands its state through and never touches a tile (and a map of zero rows
        // cannot be encoded)
        memset(&mapQ, 0, sizeof(mapQ));
        mapK = mapV = mapO = mapQ;
    } else if (!make_tensor_map_2d(&mapQ, a.q, 2, qk_inner, rows, qk_inner * 2, 64, kC, true) ||
        !make_tensor_map_2d(&mapK, a.k, 2, qk_inner, rows, qk_inner * 2, 64, kC, true) ||
        (a.v && !make_tensor_map_2d(&mapV, a.v, 2, v_inner, rows, v_inner * 2, 64, kC, true)) ||
        (a.o && !make_tensor_map_2d(&mapO, a.o, 2, v_inner, rows, v_inner * 2, 64, kC, true)))
        return cudaErrorInvalidValue;
    if (!a.v) mapV = mapK;   // never used by the kernel then
    if (!a.o) mapO = mapK;
    cudaError_t e = cudaFuncSetAttribute(gdn_scan_tensor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    return launch_chained(gdn_scan_tensor_kernel, dim3(a.H_v, a.n_seq), kThreads, kSmemBytes, s, a, mapQ, mapK, mapV, mapO);
}

}  // namespace lkv
