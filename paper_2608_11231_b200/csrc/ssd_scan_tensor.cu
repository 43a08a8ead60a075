// Chunkwise Mamba-2 (SSD) scan on the 5th-generation tensor cores (Eq. 1 with Eq. 2), for
// headdim P = 64, d_state N = 128 and bf16 x/B/C/y.  One CTA owns one sequence and TWO heads of one group and walks
// the sequence in tiles of 128 tokens with the heads' states carried on chip.  A tile is one block of the scan unless its decay
// is too strong (below).
//
// No decay appears inside a contraction.  With l the running sum of dt * A_h inside a block (in log2 units, n its last
// token) and R a scale exponent of the block,
//     y_t = 2^{l_t - R} [ sum_{i<=t} (C_t.B_i) X^_i  +  C_t S^ ],    X^_i = 2^{R - l_i} dt_i x_i,   S^ = 2^R S
//     S  <- 2^{l_n - R} [ S^ + B^T X^ ]
// so the token-by-token decay only scales the rows of X going in and the rows of y coming out,
// and the masked product G = tril(C B^T) is the same matrix for every head of the group: it is formed once per CTA, with
// nothing but the causal mask applied.  (The form with the decays inside, G'_ti = G_ti e^{l_t - l_i} dt_i, costs a mask of
// 128 x 128 / 2 products and exponent factors per head and block; that, not the tensor cores, set the pace of this scan.)
// The state as held, S^ + B^T X^, is the next block's S^ with R - l_n for R: it is multiplied by a power of two only when
// that would leave the window of kMaxScale, every block to every fifth with decays as strong as the benchmark's.
// Scaling by powers of two commutes with rounding, and fp32 and bf16 have the same exponent range, so nothing is lost
// while the exponents stay in range (see kMaxScale).
//
// Where |l| would pass kMaxRange inside a tile, in either head, the tile is scanned in several blocks, each with its own R, that end on
// multiples of 16 tokens: only the chain -- (Y2), (S), state pass -- runs once per block, 1.5 K cycles; loads, G, mask, X^ and
// outputs run once per tile as before.  Where 16 tokens are still too many (12 log2 units a token and more) a block of fewer
// tokens is a "unit" of its own, for which X^ is written and y read separately, 3 K cycles.  32 sequences x 2048 tokens x 80 heads, dt
// of 0.14 on average: A = -0.02 or -1 .. -7.4 375 / 382 us, A uniform in -1 .. -16 475 us; dt of 0.8: A = -4 737 us, A uniform in
// -1 .. -16 3200 us.  (Whole tiles loaded and scanned for every block: 370 / 378, 628, 1450, 3770 us.  The form with the decays
// inside the mask: 622 / 620, 650, 660, 960 us.)
//
// Everything is held transposed so that the tiles have M = 128 rows = 2 heads x 64 features (all 128 TMEM lanes):
//   (G)    G     = C B^T                     [128 t x 128 i], K = n        tcgen05; tril -> bf16 tile in shared memory (prep warps)
//   (Y2)   Y^T   = S^^T C^T                  [128 x 128 t], K = n          A = bf16 S^^T in tensor memory
//   (S)    S^^T += X^^T B                    [128 x 128 n], K = tokens     A = X^^T in tensor memory
//   (Y1)   Y^T  += X^^T G^T                  [128 x 128 t], K = tokens     A = X^^T in tensor memory (t < 64, i >= 64: skipped)
//   X^^T   ldmatrix.trans out of the X tile, scaled, stored to tensor memory                        prep warps
//   state  fp32 S^^T rescaled for the next block, bf16 copy beside it, both in tensor memory        state warps
//   y      Y^T scaled by 2^{l_t - r}, transposed by stmatrix into a tile that TMA stores            output warps
// X^ goes to tensor memory rather than back into its tile: the X tile is free for the next block at once, and the SM's
// shared-memory port (128 bytes per clock, the scarcest thing on chip here) is spared the write-back and three reads.
// The chain from block to block is (Y2), (S) -> state pass; X^, G and the outputs hang off it.
//
// Bound: per tile the CTA takes in 96 KB (B, C, two X tiles) and writes 32 KB; an SM takes in about 40 bytes per clock
// from L2, 2.4 K cycles, and the copy bandwidth of the memory gives 2.9 K for the X and y bytes alone.  Measured: 3.2 K
// cycles a tile on an idle GPU, 3.4 K on a full one, 2.0 K without outputs (one head per CTA and the decays inside the
// mask took 7.7 K for the same two heads).  32 sequences x 4096 tokens x 80 heads: 1370 -> 725 us.
//
// The hot loops are rolled where they repeat: eight programs run side by side, each once per tile, and fetched unrolled
// (60 KB of code) every role took three to five times as long as its instructions (the scalar warp 5300 cycles for 250).
//
// Warps 0-7 outputs (warpgroup = half of the tokens), 8-15 state (warpgroup = half of n), 16-23 X^ (warpgroup = half of the
// tokens) and then the mask, 24 TMA loads, 25 MMA issue of (S), 26 MMA issue of (G), (Y2), (Y1), 27 blocks and scalars.
// All waits on mbarriers are bounded.
#include <string.h>

#include "common.cuh"
#include "tc_common.cuh"

namespace lkv {

namespace {

using namespace tc;

constexpr int kP = 64;     // headdim
constexpr int kN = 128;    // d_state
constexpr int kQ = 128;    // tokens per tile
constexpr int kThreads = 896;

// shared-memory map (bytes, after 1024-byte alignment); every tile row is 128 bytes, 128-byte swizzle
constexpr int kTile = kQ * 128;                  // [128 rows x 64 bf16]
constexpr int kBCStage = 4 * kTile;              // [B_nb0 | B_nb1 | C_nb0 | C_nb1], each [128 tokens x 64 n]
constexpr int kOffX = 2 * kBCStage;              // X of the two heads, [128 tokens x 64 p] each
constexpr int kOffY = kOffX + 2 * kTile;         // y likewise, staged for the TMA store; an output warp writes 64 tokens x 32 p
constexpr int kOffG = kOffY + 2 * kTile;         // tril(G) bf16: columns i < 64 of all rows t (16 KB), then i >= 64 of rows t >= 64 (8 KB)
constexpr int kOffSlot = kOffG + kTile + kTile / 2;
constexpr int kSlots = 4;
constexpr int kMaxBlocks = kQ / 16;
// A unit: tokens o .. o + n - 1 of the tile that begins at token `row`, as a rule the whole tile.  It is scanned in nb blocks, block j
// in steps of 16 tokens from kb[j - 1] (k0) to kb[j]
struct Slot {            // its descriptor
    uint2 s[2][kQ / 2];  // 2^{R - l_t} dt_t of two tokens per head (0 outside the unit), as two bf16 parts: {high pair, low pair}
    float e[2][kQ];      // 2^{l_t - R}
    int fin, last;       // the last unit of its tile; of the sequence
    int row, o, n, k0, nb, pad;
    int kb[kMaxBlocks];
    float f2[2][kMaxBlocks], e2[2];   // exponents: R of a block minus the R that the one before left, l_n - R of the last one
    int pad2[2];
};
static_assert(sizeof(Slot) % 16 == 0, "vector stores");
constexpr int kSmemBytes = kOffSlot + kSlots * static_cast<int>(sizeof(Slot)) + 1024;
static_assert(kSmemBytes + 512 <= 227 * 1024, "shared memory budget");
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kMaxRange = 200.f;               // log2 units of decay inside one block of the scan
constexpr float kMaxScale = 64.f;                // R and R - l_n stay within -64 .. 64, or where the block's own decay leaves no other
                                                 // choice within -100 .. 100.  fp32 and bf16 then hold what lies between 2^-60 and 2^60, in
                                                 // those blocks 2^-25 and 2^25; a state that is only carried on has no upper limit
                                                 // (it decays as R grows)

// tensor-memory map (columns)
constexpr uint32_t kTmS = 0;        // 128: S^^T fp32
constexpr uint32_t kTmSb = 128;     // 64: S^^T as bf16 pairs (A operand of (Y2))
constexpr uint32_t kTmX = 192;      // 64: X^^T as bf16 pairs (A operand of (S) and (Y1))
constexpr uint32_t kTmY = 256;      // 128
constexpr uint32_t kTmG = 384;      // 128
constexpr uint32_t kTmemCols = 512;

struct Bars {
    // single-arrival barriers: TMA transactions and tcgen05.commit
    uint64_t full_bc[2], full_x, g_done, y2_done, y_done, h_done, xs_free, xy_free;
    // commits of (S) and (Y2) ((S) alone when no outputs are wanted)
    uint64_t bc_free[2];
    // one arrival per warp: the scalar warp
    uint64_t sc_ready[kSlots];
    // the eight output, state or prep warps
    uint64_t y_free, hb_ready, x_free, x2_ready, mask_done;
    // output and state warps (state warps alone when no outputs are wanted), the last readers of a descriptor: the others are done
    // before the products that these wait for
    uint64_t slot_free[kSlots];
};
constexpr int kBars1 = 9;
static_assert(sizeof(Bars) == 8 * (kBars1 + 2 + kSlots + 5 + kSlots), "barrier table");

__device__ __forceinline__ void named_bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
// barrier over n threads that also tells whether any of them passed true
__device__ __forceinline__ bool named_bar_or(int id, int n, bool p) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred a, b;\n\tsetp.ne.u32 a, %3, 0;\n\t"
        "bar.red.or.pred b, %1, %2, a;\n\tselp.u32 %0, 1, 0, b;\n\t}"
        : "=r"(r)
        : "r"(id), "r"(n), "r"(p ? 1u : 0u)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred P1;\n\telect.sync _|P1, %1;\n\tselp.u32 %0, 1, 0, P1;\n\t}" : "=r"(e) : "r"(0xffffffffu));
    return e;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 32 columns n0 .. n0+31 of the state of this thread's lane (feature p of head h) as bf16 pairs for (Y2)
__device__ __forceinline__ void copy_state32(uint32_t lane_base, int n0, const uint32_t (&rr)[32]) {
    uint32_t w[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) w[c] = pack_bf16(__uint_as_float(rr[2 * c]), __uint_as_float(rr[2 * c + 1]));
    tmem_st16(lane_base + kTmSb + n0 / 2, w);
}
// Scale exponent of a block of decay ln, R what the block before has left.  It is kept while it stays in the window, and then goes to the
// window's other end: the longest way until the state has to be scaled again.
__device__ __forceinline__ float scale_into(float R, float ln) {
    const float W = fmaxf(kMaxScale, ceilf(0.5f * fabsf(ln)));
    float Rn = R;
    if (fmaxf(fabsf(R), fabsf(R - ln)) > W) Rn = copysignf(W, ln);
    if (fabsf(ln) > kMaxRange) Rn = rintf(ln);   // a single token of violent decay: nothing of the state is left
    return Rn;
}
__device__ __forceinline__ void append_block(Slot &sl, int nb, int hd, float f2, float e2, int end) {
    sl.f2[hd][nb] = f2;
    sl.e2[hd] = e2;
    sl.kb[nb] = (end + 15) / 16;
}
// The blocks of a unit whose decay leaves the range.  A block ends before the first token that does, in either head, on a multiple of 16
// tokens: then the blocks of a unit share no step of the products, and X^ is written, G masked and y read once for all of
// them.  Where 16 tokens are too many, they end the unit too.  Per lane, eight tokens: l from the first token of the unit ->
// l - R of their block; dt and l zero beyond the unit.  Rare, and kept out of the scalar warp's loop.
struct Cut {
    float l[8], dt[8], keep[8];   // keep: dt of the tokens that the unit leaves
    float R, total;
    int o, end, nb;               // first token of the unit; end of the tile -> of the unit
};
__device__ __noinline__ void cut_unit(Slot &sl, Cut &c, int hd, int hl) {
    float l[8], base = 0.f, R = c.R, total = c.total;
    const int o = c.o, end = c.end;
    int cur = o, nb = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) l[j] = c.l[j];
#pragma unroll 1
    for (bool open = true; open;) {
        unsigned bad = end;
#pragma unroll
        for (int j = 7; j >= 0; --j)
            if (8 * hl + j >= cur && !(fabsf(l[j] - base) <= kMaxRange)) bad = min(bad, 8 * hl + j);
        int m = __reduce_min_sync(0xffffffffu, bad);
        open = m < end;
        if (open) {
            if ((m & ~15) > cur) {
                m &= ~15;
            } else {
                if (nb > 0) break;
                m = max(m, o + 1);
                open = false;
            }
        }
        float lm = 0.f;   // l of the block's last token
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j == ((m - 1) & 7)) lm = l[j];
        lm = __shfl_sync(0xffffffffu, lm, (m - 1) >> 3, 16);
        const float ln = lm - base, Rn = scale_into(R, ln);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (8 * hl + j >= cur && 8 * hl + j < m) l[j] -= base + Rn;   // (not looked at again)
        if (hl == 0) append_block(sl, nb, hd, Rn - R, ln - Rn, m);
        R = Rn - ln;
        total += ln;
        base = lm;
        cur = m;
        ++nb;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const bool out = 8 * hl + j >= cur;
        const float dt = c.dt[j];
        c.keep[j] = out ? dt : 0.f;
        c.dt[j] = out ? 0.f : dt;
        c.l[j] = out ? 0.f : l[j];
    }
    c.R = R;
    c.total = total;
    c.end = cur;
    c.nb = nb;
}

__global__ void __launch_bounds__(kThreads, 1)
ssd_scan_tensor_kernel(const __grid_constant__ SsdArgs a, const __grid_constant__ CUtensorMap mapX,
                       const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapC,
                       const __grid_constant__ CUtensorMap mapY) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);   // an offset, not a cast: the compiler keeps shared-memory addressing
    __shared__ Bars bars;
    __shared__ uint32_t tmem_base;
    __shared__ volatile int dead;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int per_grp = a.H / a.G, pairs = (per_grp + 1) / 2;
    const int grp = blockIdx.x / pairs, pr = blockIdx.x % pairs;
    const int h0 = grp * per_grp + 2 * pr;
    const bool two = 2 * pr + 1 < per_grp;   // the last head of an odd group is computed twice and stored once
    const int h1 = h0 + (two ? 1 : 0);
    pdl_launch();
    if (a.cu.ptr) pdl_wait();   // the index list is in global memory
    const int seq = a.cu[a.n_seq + 1 + blockIdx.y];   // launch order: longest sequence first
    const int t_begin = a.cu[seq], t_end = a.cu[seq + 1];
    // initial and final state of head h0; that of the other follows
    const float *S0 = seq < a.n_s0 ? a.S0 : a.S0_more;
    if (S0) S0 += (static_cast<size_t>(seq < a.n_s0 ? seq : seq - a.n_s0) * a.H + h0) * kN * kP;
    float *ST = seq < a.st_first ? nullptr : a.S_T;
    const size_t st_off = (static_cast<size_t>(seq - a.st_first) * a.H + h0) * kN * kP;
    const bool has_y = a.y != nullptr;

    if (t_begin == t_end) {  // empty sequence: hand the states through untouched
        pdl_wait();
        if (ST && a.S_T != a.S0)
            for (int e = tid; e < (two ? 2 : 1) * kN * kP; e += kThreads) store_state(ST, a.st_bf16, st_off + e, S0 ? S0[e] : 0.f);
        return;
    }
    if (tid == 0) {
        dead = 0;
        uint64_t *bp = &bars.full_bc[0];
        for (int i = 0; i < kBars1; ++i) mbar_init(bp++, 1);
        for (int i = 0; i < 2; ++i) mbar_init(bp++, has_y ? 2 : 1);
        for (int i = 0; i < kSlots; ++i) mbar_init(bp++, 1);
        for (int i = 0; i < 5; ++i) mbar_init(bp++, 8);
        for (int i = 0; i < kSlots; ++i) mbar_init(bp++, has_y ? 16 : 8);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(&tmem_base, kTmemCols);
    pdl_wait();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tm = tmem_base;
    Slot *slots = reinterpret_cast<Slot *>(sm + kOffSlot);
    const uint32_t lane_base = tm + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const int wg = warp >> 2, wq = warp & 3;

    if (warp == 27) {
        // ======================================================= scalar warp: half-warp = head, lane = 8 tokens
        const int hd = lane >> 4, hl = lane & 15;
        const float Ah = a.A[hd ? h1 : h0] * kLog2e;
        const float *dth = a.dt + (hd ? h1 : h0);
        // dt of the next tile and of the one after it (a load from DRAM takes as long as a block without outputs)
        float dt[8], dt2[8];
        auto fetch_dt = [&](float (&d)[8], int t0) {
            const float *p = dth + static_cast<size_t>(t0 + 8 * hl) * a.H;
#pragma unroll
            for (int j = 0; j < 8; ++j) d[j] = t0 + 8 * hl + j < t_end ? p[static_cast<size_t>(j) * a.H] : 0.f;
        };
        int t0 = t_begin, o = 0;   // tile, first token of the unit in it
        float R = 0.f, total = 0.f;
        fetch_dt(dt, t0);
        fetch_dt(dt2, t0 + kQ);
        // (never leaves the loop early: every pass advances whatever the waits say)
#pragma unroll 1
        for (int b = 0; t0 < t_end; ++b) {
            Slot &sl = slots[b % kSlots];
            float l2[8], run = 0.f, far = 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                run = fmaf(dt[j], Ah, run);   // (the tokens before the unit have been set to zero)
                l2[j] = run;
            }
            float tot = run;
#pragma unroll
            for (int k = 1; k < 16; k <<= 1) {
                const float up = __shfl_up_sync(0xffffffffu, tot, k, 16);
                if (hl >= k) tot += up;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                l2[j] += tot - run;
                far = fmaxf(far, fabsf(l2[j]));
            }
            if (b >= kSlots) mbar_wait(&bars.slot_free[b % kSlots], ((b - kSlots) / kSlots) & 1, &dead, a.status);
            __syncwarp();
            int cur = min(kQ, t_end - t0), nb = 1;
            Cut c;
            if (__builtin_expect(__any_sync(0xffffffffu, !(far <= kMaxRange)), 0)) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    c.l[j] = l2[j];
                    c.dt[j] = dt[j];
                }
                c.R = R;
                c.total = total;
                c.o = o;
                c.end = cur;
                cut_unit(sl, c, hd, hl);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    l2[j] = c.l[j];
                    dt[j] = c.dt[j];
                }
                R = c.R;
                total = c.total;
                nb = c.nb;
                cur = c.end;
            } else {
                const float ln = __shfl_sync(0xffffffffu, l2[7], 15, 16);   // tokens beyond the sequence have dt = 0
                const float Rn = scale_into(R, ln);
#pragma unroll
                for (int j = 0; j < 8; ++j) l2[j] -= Rn;
                if (hl == 0) append_block(sl, 0, hd, Rn - R, ln - Rn, cur);
                R = Rn - ln;
                total += ln;
            }
            const bool last = t0 + cur == t_end, fin = cur == kQ || last;
            if (lane == 0) {
                *reinterpret_cast<int4 *>(&sl.fin) = make_int4(fin, last, t0, o);
                *reinterpret_cast<int4 *>(&sl.n) = make_int4(cur - o, o / 16, nb, 0);
            }
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                const float s0 = dt[j] * ex2(-l2[j]), s1 = dt[j + 1] * ex2(-l2[j + 1]);
                hi[j / 2] = pack_bf16(s0, s1);
                lo[j / 2] = pack_bf16(s0 - __uint_as_float(hi[j / 2] << 16), s1 - __uint_as_float(hi[j / 2] & 0xFFFF0000u));
            }
#pragma unroll
            for (int j = 0; j < 8; j += 4) {
                *reinterpret_cast<uint4 *>(&sl.s[hd][4 * hl + j / 2]) = make_uint4(hi[j / 2], lo[j / 2], hi[j / 2 + 1], lo[j / 2 + 1]);
                if (has_y) *reinterpret_cast<float4 *>(&sl.e[hd][8 * hl + j]) = make_float4(ex2(l2[j]), ex2(l2[j + 1]), ex2(l2[j + 2]), ex2(l2[j + 3]));
            }
            warp_arrive(&bars.sc_ready[b % kSlots]);
            if (fin) {
                o = 0;
                t0 += kQ;
#pragma unroll
                for (int j = 0; j < 8; ++j) dt[j] = dt2[j];
                fetch_dt(dt2, t0 + kQ);
            } else {
                o = cur;
#pragma unroll
                for (int j = 0; j < 8; ++j) dt[j] = c.keep[j];
            }
        }
        if (a.lam && hl == 0 && (hd == 0 || two)) a.lam[static_cast<size_t>(seq) * a.H + h0 + hd] = total / kLog2e;
    } else if (warp >= 24) {
        // ======================================================= single-issue roles.  The whole warp walks the loop and one elected lane
        // issues: the operands of these instructions live in registers that the warp shares, so its lanes stay together.
        if (warp == 24) {
            // ---- TMA: one load brings both 64-column halves of B or C, or X of both heads
            int row = t_begin;
#pragma unroll 1
            for (int j = 0; row < t_end; ++j, row += kQ) {
                if (warp_dead(&dead)) break;   // a wait ran out: nothing more is issued
                const int st = j & 1;
                if (j >= 2) mbar_wait(&bars.bc_free[st], ((j - 2) >> 1) & 1, &dead, a.status);
                __syncwarp();
                if (elect_one()) {
                    unsigned char *bc = sm + st * kBCStage;
                    mbar_expect_tx(&bars.full_bc[st], has_y ? kBCStage : kBCStage / 2);
                    tma_load_3d(bc, &mapB, row, 2 * grp, &bars.full_bc[st]);
                    if (has_y) tma_load_3d(bc + 2 * kTile, &mapC, row, 2 * grp, &bars.full_bc[st]);
                    // the ring cannot hide the DRAM latency of the tile loads: pull the tiles after the next into L2 now
                    if (row + 2 * kQ < t_end) {
                        tma_prefetch_l2_3d(&mapX, row + 2 * kQ, h0);
                        tma_prefetch_l2_3d(&mapB, row + 2 * kQ, 2 * grp);
                        if (has_y) tma_prefetch_l2_3d(&mapC, row + 2 * kQ, 2 * grp);
                    }
                }
                __syncwarp();
                if (j >= 1) mbar_wait(&bars.x_free, (j - 1) & 1, &dead, a.status);
                __syncwarp();
                if (elect_one()) {
                    mbar_expect_tx(&bars.full_x, 2 * kTile);
                    tma_load_3d(sm + kOffX, &mapX, row, h0, &bars.full_x);
                }
                __syncwarp();
            }
        } else if (warp == 25) {
            // ---- MMA issue of (S)
            constexpr uint32_t idS = umma_idesc(kFmtBF16, false, true, 128, 128);
            bool last = false;
            uint32_t par = 0;   // of the block
#pragma unroll 1
            for (int b = 0, tile = 0; !last; ++b) {
                if (warp_dead(&dead)) break;
                mbar_wait(&bars.sc_ready[b % kSlots], (b / kSlots) & 1, &dead, a.status);
                const Slot &sl = slots[b % kSlots];
                const int nb = sl.nb, fin = sl.fin;
                last = sl.last;
                const int st = tile & 1;
                const uint64_t dB = umma_desc(smem_u32(sm + st * kBCStage), kTile, 1024);
                mbar_wait(&bars.full_bc[st], (tile >> 1) & 1, &dead, a.status);
                mbar_wait(&bars.x2_ready, b & 1, &dead, a.status);
                int k = sl.k0;
#pragma unroll 1
                for (int j = 0; j < nb; ++j, par ^= 1) {
                    const int k1 = sl.kb[j];
                    mbar_wait(&bars.hb_ready, par, &dead, a.status);
                    __syncwarp();
                    tc_fence_after_sync();
                    if (elect_one()) {
                        if (__builtin_expect(k1 - k == 8, 1)) {   // these instructions are on the chain: nothing is computed between them
#pragma unroll
                            for (int i = 0; i < 8; ++i) umma_bf16_ts(tm + kTmS, tm + kTmX + 8 * i, dB + ((i * 16 * 128) >> 4), idS, true);
                        } else {
#pragma unroll 1
                            for (int i = k; i < k1; ++i) umma_bf16_ts(tm + kTmS, tm + kTmX + 8 * i, dB + ((i * 16 * 128) >> 4), idS, true);
                        }
                        umma_commit(&bars.h_done);
                        if (j == nb - 1) {
                            umma_commit(&bars.xs_free);
                            if (fin) umma_commit(&bars.bc_free[st]);
                        }
                    }
                    k = k1;
                    __syncwarp();
                }
                tile += fin;
            }
        } else if (has_y) {
            // ---- MMA issue of (G) (both operands K-major; one tile ahead), (Y2), (Y1)
            constexpr uint32_t idG = umma_idesc(kFmtBF16, false, false, 128, 128);
            auto id_cols = [](int k) { return umma_idesc(kFmtBF16, false, false, 128, 16 * k); };   // 16 k columns
            const uint64_t dG = umma_desc(smem_u32(sm + kOffG), 0, 1024);
            int tile = 0;
            uint32_t par = 0;   // of the block
            bool last = false;
#pragma unroll 1
            for (int b = -1; !last; ++b) {
                if (warp_dead(&dead)) break;
                bool next = true;
                if (b >= 0) {
                    mbar_wait(&bars.sc_ready[b % kSlots], (b / kSlots) & 1, &dead, a.status);
                    const Slot &sl = slots[b % kSlots];
                    const int nb = sl.nb, fin = sl.fin;
                    last = sl.last;
                    next = fin && !last;
                    const uint64_t dC = umma_desc(smem_u32(sm + (tile & 1) * kBCStage + 2 * kTile), 0, 1024);
                    if (b >= 1) mbar_wait(&bars.y_free, (b - 1) & 1, &dead, a.status);
                    int k = sl.k0;
#pragma unroll 1
                    for (int j = 0; j < nb; ++j, par ^= 1) {
                        const int k1 = sl.kb[j];
                        mbar_wait(&bars.hb_ready, par, &dead, a.status);
                        __syncwarp();
                        tc_fence_after_sync();
                        if (elect_one()) {
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                umma_bf16_ts(tm + kTmY + 16 * k, tm + kTmSb + 8 * i, dC + ((16 * k * 128 + (i >> 2) * kTile + (i & 3) * 32) >> 4), id_cols(k1 - k), i > 0);
                            umma_commit(&bars.y2_done);
                            if (fin && j == nb - 1) umma_commit(&bars.bc_free[tile & 1]);
                        }
                        k = k1;
                        __syncwarp();
                    }
                    mbar_wait(&bars.x2_ready, b & 1, &dead, a.status);
                    mbar_wait(&bars.mask_done, tile & 1, &dead, a.status);
                    __syncwarp();
                    tc_fence_after_sync();
                    if (elect_one()) {
                        // tokens i < 64 onto all t of their block, those from 64 on onto t from 64 on
                        if (__builtin_expect(nb == 1 && k - sl.k0 == 8, 1)) {
                            constexpr uint32_t idY64 = umma_idesc(kFmtBF16, false, false, 128, 64);
#pragma unroll
                            for (int i = 0; i < 4; ++i) umma_bf16_ts(tm + kTmY, tm + kTmX + 8 * i, dG + ((i * 32) >> 4), idG, true);
#pragma unroll
                            for (int i = 4; i < 8; ++i)
                                umma_bf16_ts(tm + kTmY + 64, tm + kTmX + 8 * i, dG + ((kTile + (i - 4) * 32) >> 4), idY64, true);
                        } else {
                            k = sl.k0;
#pragma unroll 1
                            for (int j = 0; j < nb; ++j) {
                                const int k1 = sl.kb[j], q = max(k, 4);
#pragma unroll 1
                                for (int i = k; i < k1; ++i) {
                                    const int c = i < 4 ? k : q;
                                    const uint32_t tile_at = i < 4 ? 16 * k * 128 + i * 32 : kTile + 16 * (q - 4) * 128 + (i - 4) * 32;
                                    umma_bf16_ts(tm + kTmY + 16 * c, tm + kTmX + 8 * i, dG + (tile_at >> 4), id_cols(k1 - c), true);
                                }
                                k = k1;
                            }
                        }
                        umma_commit(&bars.y_done);
                        umma_commit(&bars.xy_free);
                    }
                    __syncwarp();
                    tile += next;
                }
                if (next) {   // (G) of the next tile: the mask warps have drained the G columns
                    const uint32_t bc = smem_u32(sm + (tile & 1) * kBCStage);
                    const uint64_t dB = umma_desc(bc, 0, 1024), dC = umma_desc(bc + 2 * kTile, 0, 1024);
                    mbar_wait(&bars.full_bc[tile & 1], (tile >> 1) & 1, &dead, a.status);
                    __syncwarp();
                    tc_fence_after_sync();
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const uint64_t off = ((k >> 2) * kTile + (k & 3) * 32) >> 4;
                            umma_bf16(tm + kTmG, dC + off, dB + off, idG, k > 0);
                        }
                        umma_commit(&bars.g_done);
                    }
                    __syncwarp();
                }
            }
        }
    } else if (wg >= 4) {
        // ======================================================= prep: X^^T of 64 tokens; this warp: 32 features of one head
        const int th = wg - 4, hd = wq >> 1;
        const int m = lane >> 3, i = lane & 7;
        // matrix m of a load: features 8 (m & 1) .., tokens 8 (m >> 1) ..
        const uint32_t xrow = smem_u32(sm + kOffX + hd * kTile) + (64 * th + 8 * (m >> 1) + i) * 128;
        // mask: row t of tril(G) -> bf16 operand tile, columns < 64 of row t and columns >= 64 of row t - 64
        const int t = tid & 127;
        unsigned char *g0 = sm + kOffG + t * 128, *g1 = g0 + kTile - 64 * 128;
        if ((wq & 1) == 0 && th == 0) {   // the 32 columns right of this warp's diagonal block: zeros, never written again
#pragma unroll
            for (int c8 = 4; c8 < 8; ++c8) *reinterpret_cast<uint4 *>((wq ? g1 : g0) + ((c8 ^ (t & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
        }
        bool last = false;
#pragma unroll 1
        for (int b = 0, tile = 0; !last; ++b) {
            if (warp_dead(&dead)) break;
            mbar_wait(&bars.sc_ready[b % kSlots], (b / kSlots) & 1, &dead, a.status);
            const Slot &sl = slots[b % kSlots];
            const bool first = sl.o == 0, fin = sl.fin;
            last = sl.last;
            mbar_wait(&bars.full_x, tile & 1, &dead, a.status);
            __syncwarp();
            uint32_t w[2][16];
#pragma unroll
            for (int lh = 0; lh < 2; ++lh)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    ldmatrix_x4_trans(xrow + 16 * j * 128 + (((4 * (wq & 1) + 2 * lh + (m & 1)) ^ i) << 4), w[lh][4 * j], w[lh][4 * j + 1],
                                      w[lh][4 * j + 2], w[lh][4 * j + 3]);
            // x s with s = high + low part: two packed operations and one rounding that counts, where unpacking, fp32 products and
            // packing take five
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint2 s2 = sl.s[hd][32 * th + 4 * k + (lane & 3)];
                const __nv_bfloat162 sh = *reinterpret_cast<const __nv_bfloat162 *>(&s2.x), sl2 = *reinterpret_cast<const __nv_bfloat162 *>(&s2.y);
#pragma unroll
                for (int lh = 0; lh < 2; ++lh)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        __nv_bfloat162 *x = reinterpret_cast<__nv_bfloat162 *>(&w[lh][2 * k + e]);
                        *x = __hfma2(*x, sh, __hmul2(*x, sl2));
                    }
            }
            // The tile may be overwritten once its loads have RETURNED, not once they are issued: the assembler may hold their first
            // use back past the arrival, and under load they have come back later than the next tile (seen: single rows of the
            // next block).  So which lane arrives depends on one result of every load of every lane.
            uint32_t any = 0;
#pragma unroll
            for (int j = 0; j < 16; j += 4) any |= w[0][j] | w[1][j];
            const uint32_t odd = __ballot_sync(0xffffffffu, any & 1u);
            if (fin && lane == (odd ? __ffs(odd) - 1 : 0)) mbar_arrive(&bars.x_free);
            if (b >= 1) {   // (S) and (Y1) have read the X^ before
                mbar_wait(&bars.xs_free, (b - 1) & 1, &dead, a.status);
                if (has_y) mbar_wait(&bars.xy_free, (b - 1) & 1, &dead, a.status);
            }
            __syncwarp();
            tc_fence_after_sync();
#pragma unroll
            for (int lh = 0; lh < 2; ++lh) tmem_st_16x128b_x8(lane_base + (static_cast<uint32_t>(16 * lh) << 16) + kTmX + 32 * th, w[lh]);
            tmem_st_wait();
            tc_fence_before_sync();
            warp_arrive(&bars.x2_ready);
            if (has_y && first) {
                // mask, 32 columns at a time: the two warps of a lane quarter take every other one; the last holds the diagonal.
                // ((Y1) of the block before has read the tile: waited for above.)
                mbar_wait(&bars.g_done, tile & 1, &dead, a.status);
                __syncwarp();
                tc_fence_after_sync();
#pragma unroll 1
                for (int q = th; q <= wq; q += 2) {
                    uint32_t rr[32], wm[16];
                    tmem_ld32(lane_base + kTmG + 32 * q, rr);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e) wm[e] = pack_bf16(__uint_as_float(rr[2 * e]), __uint_as_float(rr[2 * e + 1]));
                    if (q == wq) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) wm[e] = 2 * e + 1 <= lane ? wm[e] : (2 * e <= lane ? wm[e] & 0xffffu : 0u);
                    }
                    unsigned char *row = q < 2 ? g0 : g1;
#pragma unroll
                    for (int c8 = 0; c8 < 4; ++c8)
                        *reinterpret_cast<uint4 *>(row + (((4 * (q & 1) + c8) ^ (t & 7)) << 4)) = make_uint4(wm[4 * c8], wm[4 * c8 + 1], wm[4 * c8 + 2], wm[4 * c8 + 3]);
                }
                fence_async_smem();
                tc_fence_before_sync();
                warp_arrive(&bars.mask_done);
            }
            tile += fin;
        }
    } else if (wg >= 2) {
        // ======================================================= state: lane = (head, p), warpgroup = 64 columns n
        const int x = tid & 127, hd = x >> 6, n0 = 64 * (wg - 2);
        const size_t mine = (hd && two ? static_cast<size_t>(kN) * kP : 0) + static_cast<size_t>(n0) * kP + (x & 63);
        {
            // initial state, scaled by 2^R of the first block
#pragma unroll 1
            for (int q = 0; q < 2; ++q) {
                uint32_t rr[32];
#pragma unroll
                for (int c = 0; c < 32; ++c) rr[c] = S0 ? __float_as_uint(S0[mine + (32 * q + c) * kP]) : 0u;
                if (q == 0) mbar_wait(&bars.sc_ready[0], 0, &dead, a.status);
                __syncwarp();
                const float f = ex2(slots[0].f2[hd][0]);
#pragma unroll
                for (int c = 0; c < 32; ++c) rr[c] = __float_as_uint(__uint_as_float(rr[c]) * f);
                tmem_st32(lane_base + kTmS + n0 + 32 * q, rr);
                copy_state32(lane_base, n0 + 32 * q, rr);
            }
            tmem_st_wait();
            tc_fence_before_sync();
            warp_arrive(&bars.hb_ready);
        }
        bool last = false;
        int b = 0, j = 0;   // unit, block
#pragma unroll 1
        for (uint32_t par = 0; !last; par ^= 1) {
            if (warp_dead(&dead)) break;
            mbar_wait(&bars.sc_ready[b % kSlots], (b / kSlots) & 1, &dead, a.status);
            const Slot &sl = slots[b % kSlots];
            const bool done = j + 1 == sl.nb;   // with the unit
            last = done && sl.last;
            float ex = sl.e2[hd];
            if (!done) {
                ex = sl.f2[hd][j + 1];
            } else if (!last) {
                mbar_wait(&bars.sc_ready[(b + 1) % kSlots], ((b + 1) / kSlots) & 1, &dead, a.status);
                ex = slots[(b + 1) % kSlots].f2[hd][0];
            }
            const float f = ex2(0.5f * ex);   // in two steps: the factor may lie below the fp32 range where its product with the state does not
            const bool scale = __any_sync(0xffffffffu, ex != 0.f);
            mbar_wait(&bars.h_done, par, &dead, a.status);
            if (has_y) mbar_wait(&bars.y2_done, par, &dead, a.status);   // the bf16 copy has been read
            __syncwarp();
            tc_fence_after_sync();
            if (last) {
                const bool store = ST && (hd == 0 || two) && !warp_dead(&dead);
#pragma unroll 1
                for (int q = 0; q < 8; ++q) {
                    uint32_t rr[8];
                    tmem_ld8(lane_base + kTmS + n0 + 8 * q, rr);
                    tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        if (store) store_state(ST, a.st_bf16, st_off + mine + static_cast<size_t>(8 * q + c) * kP, __uint_as_float(rr[c]) * f * f);
                }
            } else {
#pragma unroll 1
                for (int q = 0; q < 2; ++q) {
                    uint32_t rr[32];
                    tmem_ld32(lane_base + kTmS + n0 + 32 * q, rr);
                    tmem_ld_wait();
                    if (scale) {
#pragma unroll
                        for (int c = 0; c < 32; ++c) rr[c] = __float_as_uint(__uint_as_float(rr[c]) * f * f);
                        tmem_st32(lane_base + kTmS + n0 + 32 * q, rr);
                    }
                    copy_state32(lane_base, n0 + 32 * q, rr);
                }
                tmem_st_wait();
                tc_fence_before_sync();
                warp_arrive(&bars.hb_ready);
            }
            ++j;
            if (done) {
                warp_arrive(&bars.slot_free[b % kSlots]);
                ++b;
                j = 0;
            }
        }
    } else if (has_y) {
        // ======================================================= outputs of 64 tokens; this warp: 32 features of one head
        const int th = wg, hd = wq >> 1;
        const int m = lane >> 3, i = lane & 7;
        // staging rows [token][128 bytes = 64 features], this warp's four 16-byte pieces of each;
        // matrix m of a store: features 8 (m & 1) .., tokens 8 (m >> 1) ..
        unsigned char *ys = sm + kOffY + hd * kTile + 64 * th * 128;
        const uint32_t srow = smem_u32(ys) + (8 * (m >> 1) + i) * 128;
        bool last = false;
#pragma unroll 1
        for (int b = 0; !last; ++b) {
            mbar_wait(&bars.sc_ready[b % kSlots], (b / kSlots) & 1, &dead, a.status);
            const Slot &sl = slots[b % kSlots];
            const int row = sl.row, o = sl.o, n = sl.n;
            last = sl.last;
            mbar_wait(&bars.y_done, b & 1, &dead, a.status);
            __syncwarp();
            tc_fence_after_sync();
            // all of Y leaves tensor memory (packed: 32 registers) before the stage is needed, which the store of the block before
            // may still be reading
            uint32_t w[2][16];
            const float *e0 = &sl.e[hd][64 * th + 2 * (lane & 3)];
#pragma unroll
            for (int lh = 0; lh < 2; ++lh) {
                uint32_t r[32];
                tmem_ld_16x256b_x8(lane_base + (static_cast<uint32_t>(16 * lh) << 16) + kTmY + 64 * th, r);
                tmem_ld_wait();
                if (lh == 1) {
                    tc_fence_before_sync();
                    warp_arrive(&bars.y_free);
                }
#pragma unroll
                for (int k = 0; k < 8; ++k) {   // 8 tokens
                    const float2 e = *reinterpret_cast<const float2 *>(e0 + 8 * k);
#pragma unroll
                    for (int u = 0; u < 2; ++u)   // (scalar multiplies: packed ones cost register moves here)
                        w[lh][2 * k + u] = pack_bf16(__uint_as_float(r[4 * k + 2 * u]) * e.x, __uint_as_float(r[4 * k + 2 * u + 1]) * e.y);
                }
            }
            warp_arrive(&bars.slot_free[b % kSlots]);
            // the eight warps leave together if a wait ran out
            if (warp == 0 && elect_one()) tma_store_wait_read();
            if (named_bar_or(1, 256, dead != 0)) break;
#pragma unroll
            for (int lh = 0; lh < 2; ++lh)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)   // 16 tokens
                    stmatrix_x4_trans(srow + 16 * kk * 128 + (((4 * (wq & 1) + 2 * lh + (m & 1)) ^ i) << 4), w[lh][4 * kk], w[lh][4 * kk + 1],
                                      w[lh][4 * kk + 2], w[lh][4 * kk + 3]);
            if (__builtin_expect(n == kQ && two, 1)) {
                fence_async_smem();
                named_bar_sync(2, 256);
                if (warp == 0 && elect_one()) {
                    tma_store_3d(&mapY, sm + kOffY, row, h0);
                    tma_store_commit();
                }
            } else if (hd == 0 || two) {
                // a block that is not a whole tile, or whose second head is not wanted: rows straight to global memory; lane = row i
                // of eight, piece m of this warp's four
                __syncwarp();
                const int lo = max(o - 64 * th, 0), hi = min(o + n - 64 * th, 64), row0 = (lo & ~7) + i;
                const size_t tstride = static_cast<size_t>(a.H) * kP;
                __nv_bfloat16 *dst = static_cast<__nv_bfloat16 *>(a.y) + static_cast<size_t>(row + 64 * th + row0) * tstride +
                                     static_cast<size_t>(h0 + hd) * kP + 32 * (wq & 1) + 8 * m;
                const unsigned char *src = ys + row0 * 128 + (((4 * (wq & 1) + m) ^ i) << 4);
#pragma unroll 1
                for (int r = row0; r < hi; r += 8, src += 8 * 128, dst += 8 * tstride)
                    if (r >= lo) *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(src);
                fence_async_smem();
            }
        }
        if (warp == 0 && elect_one()) tma_store_wait_all();
    }
    grace_after_timeout(&dead);
    __syncwarp();   // the warps of the single-thread roles come back together before the warp-aligned instructions below
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tm, kTmemCols);
}

}  // namespace

bool ssd_scan_tensor_supported(const SsdArgs &a, bool io_bf16) {
    return io_bf16 && a.P == kP && a.N == kN;
}

cudaError_t launch_ssd_scan_tensor(const SsdArgs &a, cudaStream_t s) {
    CUtensorMap mapX, mapB, mapC, mapY;
    const uint64_t rows = static_cast<uint64_t>(a.T_total);
    const uint64_t x_inner = static_cast<uint64_t>(a.H) * kP, bc_inner = static_cast<uint64_t>(a.G) * kN;
    if (rows == 0) {
        // no token anywhere: every CTA hands its state through and never touches a tile (and a map of zero rows
        // cannot be encoded)
        memset(&mapX, 0, sizeof(mapX));
        mapB = mapC = mapY = mapX;
    } else if (!make_tensor_map_cols64(&mapX, a.x, x_inner, rows, x_inner * 2, kQ, 2) ||
               !make_tensor_map_cols64(&mapB, a.B, bc_inner, rows, bc_inner * 2, kQ, 2) ||
               !make_tensor_map_cols64(&mapC, a.C, bc_inner, rows, bc_inner * 2, kQ, 2) ||
               !make_tensor_map_cols64(&mapY, a.y ? a.y : a.x, x_inner, rows, x_inner * 2, kQ, 2)) {
        return cudaErrorInvalidValue;
    }
    cudaError_t e = cudaFuncSetAttribute(ssd_scan_tensor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    const int pairs = (a.H / a.G + 1) / 2;
    return launch_chained(ssd_scan_tensor_kernel, dim3(a.G * pairs, a.n_seq), kThreads, kSmemBytes, s, a, mapX, mapB, mapC, mapY);
}

}  // namespace lkv
