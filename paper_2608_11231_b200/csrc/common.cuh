// Shared device/host helpers of the lkv CUDA library (sm_100a only).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <type_traits>

#include "../../include/lkv.h"

namespace lkv {

// First 256 bytes of every workspace: word 0 is the device status (0 = fine).
constexpr size_t kWsHeaderBytes = 256;
// Status values written by kernels whose bounded waits ran out.
constexpr int kDevTimeout = 1;

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

template <typename T>
__device__ __forceinline__ float to_f32(T x);
template <>
__device__ __forceinline__ float to_f32<float>(float x) { return x; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

template <typename T>
__device__ __forceinline__ T from_f32(float x);
template <>
__device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// Final-state store of the scans: element idx of S_T as fp32, or rounded to bf16 when the caller asked for that.
__device__ __forceinline__ void store_state(float *S_T, int st_bf16, size_t idx, float v) {
    if (st_bf16) reinterpret_cast<__nv_bfloat16 *>(S_T)[idx] = __float2bfloat16_rn(v);
    else S_T[idx] = v;
}

// Kernels of this library are launched so that the next one on the stream may start while this one runs (programmatic dependent
// launch): its launch latency and its set-up -- barriers, tensor memory -- then overlap this one's tail.  What such a kernel
// owes: every thread calls pdl_wait(), which returns when the kernels before it are complete and their writes visible, before it
// reads or writes global memory; pdl_launch() says that the next one may start as soon as SMs are free.
// Measured on B200: the two kernels of a request that continues from its cached state 14.3 -> 11.0 us, composition and scan of
// 1024 tokens 33.1 -> 27.9 us.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... Params, typename... Args>
cudaError_t launch_kernel(bool early, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const Args &...args) {
    static_assert((std::is_same<Params, Args>::value && ...), "the arguments are passed by address");
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s; cfg.attrs = attr; cfg.numAttrs = 1;
    void *p[] = {const_cast<void *>(static_cast<const void *>(&args))...};
    return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(kernel), p);
}
template <typename... Params, typename... Args>
cudaError_t launch_chained(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const Args &...args) {
    return launch_kernel(true, kernel, grid, block, smem, s, args...);
}

// Small host-checked index arrays travel to the device inside the kernel parameters
// (no copy, no extra stream operation); lists longer than CAP are copied into the
// caller's workspace instead and reached through `ptr`.
template <int CAP>
struct IndexBlock {
    const int32_t *ptr;  // device copy, or nullptr when the inline array is used
    int32_t n;           // entries of the inline array in use
    int32_t v[CAP];
    __device__ __forceinline__ int32_t operator[](int i) const { return ptr ? ptr[i] : v[i]; }
};
constexpr int kInitIdxCap = 4000;  // ints: cu_k | sel | ids
constexpr int kScanIdxCap = 1000;  // ints: cu_seqlens[n_seq + 1] | launch order[n_seq]
// A launch is the slower the more parameter bytes it carries.  It shows where the kernel is next to nothing and the kernel after it waits for
// no more than its launch: the copy of one cached state followed by the scan of a 37-token suffix takes 10.1 us with this short
// list and 10.9 with the long one (in turn on one GPU, twice); composition and the fp32 kernels take the same time with either.  So
// the copy exists with a short list too.
constexpr int kSmallIdxCap = 96;   // ints: 32 requests with one chunk each

// Launch-side records shared by the entry points and the kernels.  Passed by value as
// __grid_constant__ kernel parameters.
struct InitArgsBase {
    const void *states;        // pool
    const float *transitions;  // pool (log-decay or dense)
    float *S0;                 // [n_req, H, d_k, d_v]
    int32_t n_req, H, d_k, d_v, n_chunks;
    int32_t off_sel;           // offset of sel[n_req] in idx, or -1 (= last block)
    int32_t off_ids;           // offset of ids[total_K] in idx; cu_k[n_req + 1] sits at 0
    int32_t product = -1;      // GDN on the tensor cores: this request is the product of its chunks' transitions, with no states in it
    int32_t *status;           // device status word
};
template <int CAP>
struct InitArgsT : InitArgsBase {
    IndexBlock<CAP> idx;
    __device__ __forceinline__ int cu_k(int r) const { return idx[r]; }
    __device__ __forceinline__ int id(int i) const { return idx[off_ids + i]; }
    __device__ __forceinline__ int sel(int r, int K) const { return off_sel < 0 ? K - 1 : idx[off_sel + r]; }
};
using InitArgs = InitArgsT<kInitIdxCap>;

int sm_count();   // of the current device

struct GdnArgs {
    const void *q, *k, *v;
    const float *g, *beta, *S0;
    void *o;
    float *S_T;                  // final states, fp32 or (st_bf16) bf16 behind the same pointer
    const float *S_add;          // added to every final state before it is stored (Eq. 5: S_out = T_C S_in + S_local), or nullptr
    int32_t st_bf16;
    int32_t n_seq, T_total, H_k, H_v, d_k, d_v;
    float scale;
    int32_t s0_identity;         // start every sequence from S = I (d_k == d_v) instead of S0; with v == nullptr (read
                                 // as zeros) the final state is then the sequence's accumulated transition; o may be nullptr
    // Sequences tr_first .. n_seq-1 are "transition sequences": they run in that mode (S = I, v = 0, no outputs) whatever
    // the call's own mode is, over the token range of sequence (seq - tr_first + tr_src0).  cu has n_ranges + 1 entries
    // (the ranges of sequences 0 .. tr_first-1); a plain call has n_ranges = tr_first = n_seq.
    int32_t n_ranges, tr_first, tr_src0;
    float *tr_out;               // where transition sequence tr_first + i stores its final state (index i), or nullptr: S_T like the others
    // One sequence cut into segments that run side by side.  Sequences n_s0 .. start from S0_more (index
    // seq - n_s0; nullptr = zero), final states are wanted of sequences st_first .. only (index seq - st_first).  A plain call
    // has n_s0 = n_seq, st_first = 0.
    int32_t n_s0, st_first;
    const float *S0_more;
    int32_t *status;
    IndexBlock<kScanIdxCap> cu;  // cu_seqlens[n_seq + 1], then the launch order: sequence of grid row y at [n_seq + 1 + y]
};

struct SsdArgs {
    const void *x, *B, *C;
    const float *dt, *A, *S0;
    void *y;
    float *S_T;                  // final states, fp32 or (st_bf16) bf16 behind the same pointer
    int32_t st_bf16;
    // One sequence cut into segments that run side by side (tensor-core scan only).  Sequences n_s0 .. start from S0_more
    // (index seq - n_s0; nullptr = zero), final states are wanted of sequences st_first .. only (index seq - st_first), and
    // lam, where given, gets the log-decay of every sequence and head.  A plain call has n_s0 = n_seq, st_first = 0, lam = nullptr.
    int32_t n_s0, st_first;
    const float *S0_more;
    float *lam;
    int32_t n_seq, T_total, H, P, N, G;
    int32_t *status;
    IndexBlock<kScanIdxCap> cu;  // cu_seqlens[n_seq + 1]
};

// Kernel launchers (one translation unit each); all return a cudaError_t from the launch.
cudaError_t launch_init_single(const InitArgs &a, bool pool_bf16, cudaStream_t s);
cudaError_t launch_init_mamba_exact(const InitArgs &a, bool pool_bf16, cudaStream_t s);
// persistent streaming variant (head size a multiple of 16 KB of pool values); same results bit for bit
bool init_mamba_stream_supported(const InitArgs &a, bool pool_bf16);
cudaError_t launch_init_mamba_exact_stream(const InitArgs &a, bool pool_bf16, cudaStream_t s);
cudaError_t launch_init_gdn_exact_fp32(const InitArgs &a, bool pool_bf16, cudaStream_t s);
bool init_gdn_exact_tensor_supported(const InitArgs &a, bool pool_bf16);
// early = false: not before the kernel ahead of it on the stream has left the GPU; shared: the requests name the same chunks
cudaError_t launch_init_gdn_exact_tensor(const InitArgs &a, bool pool_bf16, cudaStream_t s, bool early = true, bool shared = false);

bool gdn_scan_fp32_supported(int d_k, int d_v);
cudaError_t launch_gdn_scan_fp32(const GdnArgs &a, bool io_bf16, cudaStream_t s);
bool gdn_scan_tensor_supported(const GdnArgs &a, bool io_bf16);
cudaError_t launch_gdn_scan_tensor(const GdnArgs &a, cudaStream_t s);
// states (S_T) and transitions (tr_out) of the n_seq sequences, from nothing; shapes as for the scan, v not null
cudaError_t launch_gdn_build_tensor(const GdnArgs &a, cudaStream_t s);

bool ssd_scan_fp32_supported(int N, int P);
cudaError_t launch_ssd_scan_fp32(const SsdArgs &a, bool io_bf16, cudaStream_t s);
bool ssd_scan_tensor_supported(const SsdArgs &a, bool io_bf16);
cudaError_t launch_ssd_scan_tensor(const SsdArgs &a, cudaStream_t s);
// lambda[c][h] = A[h] * sum of dt over sequence c (cu in the parameter block of `a`; only dt, A, H, n_seq, cu are read); longest: tokens of the longest sequence
cudaError_t launch_mamba_logdecay(const SsdArgs &a, float *logdecay, int longest, cudaStream_t s);
// rel_err[i] = ||x_i - r_i|| / ||r_i|| over n_states runs of `elems` floats; parts = CTAs per state, partial sums
// (2 floats per CTA) in `partials`
int state_err_parts(size_t elems);
cudaError_t launch_state_rel_error(const float *x, const float *r, float *rel_err, int n_states, size_t elems,
                                   float *partials, cudaStream_t s);

// one CTA waits on an mbarrier nobody arrives on, with the kernels' own bounded wait and a small poll limit
cudaError_t launch_selftest_bounded_wait(uint32_t poll_limit, int32_t *status, cudaStream_t s);

}  // namespace lkv
