// What the GDN kernels on the tensor cores share: the layout of a block's matrices and scalars, and the steps of the inverse of I + A.
// (The scan has the bodies of its roles in place: moved into functions that both kernels call its blocks took 1.3 % longer, 32 sequences of
// 2048 tokens 483 -> 489 us.)
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"
#include "tc_common.cuh"

namespace lkv {

namespace {

using namespace tc;

constexpr int kD = 128;   // d_k = d_v
constexpr int kC = 64;    // tokens per block

// A, inverted in place: fp16 tiles F, two buffers (rows and columns 0..31; 32..63; rows 32..63 of columns 0..31: the part below
// the 16x16 diagonal blocks, which only ever is an operand of fp16 MMAs, and M as it becomes final), and the 16x16 diagonal
// blocks D [t][i & 15] in fp32.  The row strides keep the eight rows of an 8x8 tile in different banks.
constexpr int kLdF = 80, kLdD = 20;                    // bytes; floats
constexpr int kFTile = 32 * kLdF, kFBytes = 3 * kFTile;
// arrays of a block's scalars (l = running sum of g in log2 units, R = the block's scale exponent), 64 floats each
constexpr int kGbL = 0;                                // l
constexpr int kGbX1 = kC, kGbX2 = 2 * kC;              // column factors of X1, X2: beta 2^{R - l}, -beta (exact block: beta, -beta 2^l)
constexpr int kGbE = 3 * kC, kGbW = 4 * kC;            // output factor scale 2^{l - R} (exact block: scale), 2^{l_C - l} (exact block only)
constexpr int kGbExp = 5 * kC;                         // exponents into the block: bf16 copy, fp32 state; exponent out of it; exact flag
constexpr int kGbFloats = 5 * kC + 4;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kMaxRange = 80.f;                      // log2 units of decay inside a block: beyond that the block is "exact"
constexpr float kMaxScale = 80.f;                      // R - l_C at most; then the state goes back to R = 0 (never below: a state that
                                                       // only decays, as a transition does, keeps the whole fp32 range).  fp32 and bf16
                                                       // then hold pseudo-values u up to 2^46; a state that is only carried on has no
                                                       // upper limit (it decays as R grows)

// Warp-level tensor-core MMA on fp16 operands (11-bit significands like tf32, but 16 k-elements per
// instruction): acc[16 x 8] += A[16 x 16] B[16 x 8], fp32 accumulation.  Fragments as the PTX ISA lays them out.
// Every operand here is an entry of A or of an inverse of I + A: of order one or smaller, far inside the fp16 range.
__device__ __forceinline__ void mma_f16_16x8x16(float (&acc)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
    const __half2 v = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}
// Operands from an fp16 matrix with row stride kLdF (shared address p of their first element): A, the 16 x 16 tile
__device__ __forceinline__ void frag_a(uint32_t (&a)[4], uint32_t p, int lane) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(p + (lane & 15) * kLdF + (lane >> 4) * 16)
                 : "memory");
}
// B, the 16 (k) x 8 (n) tile B[k][n]
__device__ __forceinline__ void frag_b(uint32_t (&b)[2], uint32_t p, int lane) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];"
                 : "=r"(b[0]), "=r"(b[1])
                 : "r"(p + (lane & 15) * kLdF)
                 : "memory");
}

// Byte offset of element (row m, column i) of a bf16 operand tile with 128-byte rows and the 128-byte swizzle
__device__ __forceinline__ uint32_t x_offset(int m, int i) { return m * 128u + ((((uint32_t)i >> 3) ^ (m & 7u)) << 4) + (i & 7) * 2u; }
// Final entries of M also go, times the factor of their column and rounded to bf16, into the operands X1 = M diag(f1) and
// X2 = M diag(f2): no second pass over M.  f1 and f2 are kC floats apart, xb1 and xb2 the two tiles.  Accumulator tile
// [16 x 8] at (m0, i0):
__device__ __forceinline__ void store_acc_x(unsigned char *xb1, unsigned char *xb2, const float *f, int m0, int i0, const float (&acc)[4], float sgn,
                                            int gid, int tig) {
    const int i = i0 + 2 * tig;
    const float2 f1 = *reinterpret_cast<const float2 *>(f + i), f2 = *reinterpret_cast<const float2 *>(f + kC + i);
    const uint32_t o0 = x_offset(m0 + gid, i), o1 = x_offset(m0 + gid + 8, i);
    const float v0 = sgn * acc[0], v1 = sgn * acc[1], v2 = sgn * acc[2], v3 = sgn * acc[3];
    *reinterpret_cast<uint32_t *>(xb1 + o0) = pack_bf16(v0 * f1.x, v1 * f1.y);
    *reinterpret_cast<uint32_t *>(xb1 + o1) = pack_bf16(v2 * f1.x, v3 * f1.y);
    *reinterpret_cast<uint32_t *>(xb2 + o0) = pack_bf16(v0 * f2.x, v1 * f2.y);
    *reinterpret_cast<uint32_t *>(xb2 + o1) = pack_bf16(v2 * f2.x, v3 * f2.y);
}

// The inverse M = (I + A)^{-1} of the unit lower triangular 64x64 matrix of a block is built by doubling:
// 8x8 diagonal blocks by forward substitution, then three merges
//     inv [[L1, 0], [A21, L2]] = [[inv L1, 0], [-inv(L2) A21 inv(L1), inv L2]]
// from 8 to 16 (fp32 FMAs), 16 to 32 and 32 to 64 (warp-level tensor-core MMA, fp16 operands rounded to nearest,
// fp32 accumulation).  What is an operand of these MMAs is stored in fp16 once, by whoever produces it; the inner product of a
// merge passes from accumulator to operand layout in registers (movmatrix), so that a merge is a few ldmatrix, two rounds of
// MMAs and the stores, and both merges together need two barriers between the warps.
// A product [16 x 8] (rows = k of the next product) as B operand: columns become the fragment's n
__device__ __forceinline__ void acc_to_b(uint32_t (&b)[2], const float (&acc)[4]) {
    const uint32_t p0 = pack_f16(acc[0], acc[1]), p1 = pack_f16(acc[2], acc[3]);
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(b[0]) : "r"(p0));
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(b[1]) : "r"(p1));
}
// 16 -> 32: half (8 columns from 8 nh) of the 16x16 block (r, c) = (c + 1, c): M_rc = -M_rr (A_rc M_cc); a32 = A_rc, Ft the
// tile of F with these blocks
__device__ __forceinline__ void inv_merge32(const uint32_t (&a32)[4], unsigned char *Ft, unsigned char *xb1, unsigned char *xb2, const float *f, int c, int nh,
                                            int lane) {
    const int r = c + 1, gid = lane >> 2, tig = lane & 3;
    const uint32_t Fs = smem_u32(Ft);
    uint32_t a[4], b[2];
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    frag_b(b, Fs + 16 * nh, lane);
    frag_a(a, Fs + 16 * kLdF + 32, lane);
    mma_f16_16x8x16(acc, a32, b[0], b[1]);
    acc_to_b(b, acc);
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = 0.f;
    mma_f16_16x8x16(acc, a, b[0], b[1]);
    unsigned char *out = Ft + (16 + gid) * kLdF + (8 * nh + 2 * tig) * 2;
    *reinterpret_cast<uint32_t *>(out) = pack_f16(-acc[0], -acc[1]);
    *reinterpret_cast<uint32_t *>(out + 8 * kLdF) = pack_f16(-acc[2], -acc[3]);
    store_acc_x(xb1, xb2, f, 16 * r, 16 * c + 8 * nh, acc, -1.f, gid, tig);
}
// 32 -> 64: columns 8 w .. 8 w + 7 of M[32.., 0..31] = -inv(L2) (A21 inv(L1)); a64[mt][kb] = A[32 + 16 mt, 16 kb].  Only the
// operands of the solve need this block: it is not stored in F.
__device__ __forceinline__ void inv_merge64(const uint32_t (&a64)[2][2][4], uint32_t Fs, unsigned char *xb1, unsigned char *xb2, const float *f, int w,
                                            int lane) {
    float acc[2][4];
    uint32_t b[2][2], a[4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[mt][i] = 0.f;
    frag_b(b[1], Fs + 16 * kLdF + 16 * w, lane);
    if (w < 2) {   // rows 0..15 of inv(L1) are zero right of its block diagonal
        frag_b(b[0], Fs + 16 * w, lane);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) mma_f16_16x8x16(acc[mt], a64[mt][0], b[0][0], b[0][1]);
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) mma_f16_16x8x16(acc[mt], a64[mt][1], b[1][0], b[1][1]);
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) acc_to_b(b[mt], acc[mt]);
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[mt][i] = 0.f;
#pragma unroll
        for (int kb = 0; kb <= mt; ++kb) {   // columns of inv(L2) right of its block diagonal are zero
            frag_a(a, Fs + kFTile + (16 * mt) * kLdF + 32 * kb, lane);
            mma_f16_16x8x16(acc[mt], a, b[kb][0], b[kb][1]);
        }
        store_acc_x(xb1, xb2, f, 32 + 16 * mt, 8 * w, acc[mt], -1.f, lane >> 2, lane & 3);
    }
}
__device__ __forceinline__ void named_bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred P1;\n\telect.sync _|P1, %1;\n\tselp.u32 %0, 1, 0, P1;\n\t}" : "=r"(e) : "r"(0xffffffffu));
    return e;
}
// 16 consecutive fp32 values -> bf16, written as 2 swizzled 16-byte chunks (chunk0, chunk0+1) of operand row `row`
__device__ __forceinline__ void store_row_chunks(unsigned char *tile, int row, int chunk0, const float (&v)[16]) {
#pragma unroll
    for (int c8 = 0; c8 < 2; ++c8) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) w[e] = pack_bf16(v[8 * c8 + 2 * e], v[8 * c8 + 2 * e + 1]);
        *reinterpret_cast<uint4 *>(tile + sw128_offset(row, chunk0 + c8)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}
// 16 fp32 values (as loaded from tensor memory) -> 8 columns of bf16 pairs, the even element in the low half
__device__ __forceinline__ void pack16(const float (&v)[16], uint32_t (&w)[8]) {
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = pack_bf16(v[2 * e], v[2 * e + 1]);
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Exact block: W entries of a row of G times 2^{l_t - l_i}, l = the columns' l in shared memory.  What lies above the diagonal may
// overflow; nobody reads it unmasked.
template <int W>
__device__ __forceinline__ void apply_decay(float (&v)[W], const float *l, float lt) {
#pragma unroll
    for (int c = 0; c < W; c += 4) {
        const float4 li = *reinterpret_cast<const float4 *>(l + c);
        v[c] *= ex2(lt - li.x); v[c + 1] *= ex2(lt - li.y); v[c + 2] *= ex2(lt - li.z); v[c + 3] *= ex2(lt - li.w);
    }
}
// Exact block: u_t[j] of 32 tokens -> Uw = w o u as bf16 pairs over the first 16 of these 32 columns, u (if wanted) over the rest
__device__ __noinline__ void u_operands_exact(uint32_t taddr, const float *w, bool both) {
    uint32_t rr[32], p[16];
    tmem_ld32(taddr, rr);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 16; e += 2) {
        const float4 f = *reinterpret_cast<const float4 *>(w + 2 * e);
        p[e] = pack_bf16(__uint_as_float(rr[2 * e]) * f.x, __uint_as_float(rr[2 * e + 1]) * f.y);
        p[e + 1] = pack_bf16(__uint_as_float(rr[2 * e + 2]) * f.z, __uint_as_float(rr[2 * e + 3]) * f.w);
    }
    tmem_st16(taddr, p);
    if (!both) return;
#pragma unroll
    for (int e = 0; e < 16; ++e) p[e] = pack_bf16(__uint_as_float(rr[2 * e]), __uint_as_float(rr[2 * e + 1]));
    tmem_st16(taddr + 16, p);
}

// Empty sequence: the initial state (the identity, S0, or zero) and what is to be added, as the final state
__device__ __noinline__ void hand_through(float *ST, size_t obase, int st_bf16, bool id, const float *S0, const float *add) {
#pragma unroll 1
    for (int e = threadIdx.x; e < kD * kD; e += blockDim.x)
        store_state(ST, st_bf16, obase + e, (id ? (e / kD == e % kD ? 1.f : 0.f) : (S0 ? S0[e] : 0.f)) + (add ? add[e] : 0.f));
}
}  // namespace

}  // namespace lkv
