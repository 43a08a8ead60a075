// C-ABI entry points: argument validation, index marshalling and kernel selection.
// Everything that can be wrong with a call is found here, on the host, before a launch.
#include <string.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "segments.h"

using namespace lkv;

int lkv::sm_count() {
    static int cached[64];   // per device; the same value whoever writes it
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return 148;
    }
    n = __atomic_load_n(&cached[dev], __ATOMIC_RELAXED);
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            n = 148;
        }
        __atomic_store_n(&cached[dev], n, __ATOMIC_RELAXED);
    }
    return n;
}

namespace {

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline bool dtype_ok(int d) { return d == LKV_DTYPE_F32 || d == LKV_DTYPE_BF16; }
inline bool compute_ok(int c) { return c == LKV_COMPUTE_AUTO || c == LKV_COMPUTE_FP32 || c == LKV_COMPUTE_TENSOR; }

// Byte ranges [p, p + n) and [q, q + m) share at least one byte (empty or NULL ranges never do).
inline bool overlaps(const void *p, size_t n, const void *q, size_t m) {
    if (!p || !q || n == 0 || m == 0) return false;
    const uintptr_t a = reinterpret_cast<uintptr_t>(p), b = reinterpret_cast<uintptr_t>(q);
    return a < b + m && b < a + n;
}

size_t ws_bytes_for(int n_ints, int cap) {
    return kWsHeaderBytes + (n_ints > cap ? align_up(sizeof(int32_t) * static_cast<size_t>(n_ints), 256) : 0);
}

// Puts `ints` where the kernels will find them: inline in the parameter block when they
// fit, otherwise one small async copy into the workspace behind its header.
template <int CAP>
int place_indices(IndexBlock<CAP> &blk, const std::vector<int32_t> &ints, void *workspace, cudaStream_t s) {
    if (static_cast<int>(ints.size()) <= CAP) {
        blk.ptr = nullptr;
        blk.n = static_cast<int32_t>(ints.size());
        if (!ints.empty()) memcpy(blk.v, ints.data(), sizeof(int32_t) * ints.size());
        return LKV_OK;
    }
    // The copy reads a host array that dies with this call: a stream capture would record the read, not do it.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
        cudaGetLastError();
        return LKV_ERR_CUDA;
    }
    if (cap != cudaStreamCaptureStatusNone) return LKV_ERR_UNSUPPORTED;
    int32_t *dst = reinterpret_cast<int32_t *>(static_cast<char *>(workspace) + kWsHeaderBytes);
    if (cudaMemcpyAsync(dst, ints.data(), sizeof(int32_t) * ints.size(), cudaMemcpyHostToDevice, s) != cudaSuccess) {
        cudaGetLastError();
        return LKV_ERR_CUDA;
    }
    blk.ptr = dst;
    blk.n = 0;
    return LKV_OK;
}

int check_init_desc(const lkv_init_desc *d) {
    if (!d) return LKV_ERR_NULL;
    if (d->family != LKV_FAMILY_MAMBA2 && d->family != LKV_FAMILY_GDN) return LKV_ERR_MODE;
    if (!dtype_ok(d->state_dtype) || !compute_ok(d->compute)) return LKV_ERR_MODE;
    if (d->H < 1 || d->d_k < 1 || d->d_v < 1 || d->n_chunks < 0) return LKV_ERR_DIM;
    return LKV_OK;
}

// Do the requests name the chunks 1.5 times on average or more, and is all that they name, repeats included and every state counted as
// fp32, more than L2 holds?  Then the order of the composition's CTAs matters (kMaxGroupLog2 in init_gdn_tensor.cu).  Below that
// many bytes it does not: 4 requests over 4 chunks (67 MB) 17.4 us in either order.
bool shares_chunks(const int32_t *ids, int total, const lkv_init_desc *d) {
    constexpr double kL2Bytes = 126e6;
    if (2.0 * sizeof(float) * total * d->H * d->d_k * d->d_v <= kL2Bytes) return false;
    std::vector<bool> seen(d->n_chunks, false);
    int distinct = 0;
    for (int i = 0; i < total; ++i) {
        distinct += !seen[ids[i]];
        seen[ids[i]] = true;
    }
    return 2LL * total >= 3LL * distinct;
}

// One request's chain of K steps in two halves side by side, where three CTAs a head find an SM each: the state A of the first half, and of
// the second the state B that it reaches from nothing and the product P of its transitions; then S0 = P A + B.  The second launch costs
// about four steps.  32 heads: K = 10 19.6 -> 17.1 us, 16 30.3 -> 22.8, 64 120.6 -> 69.7 (8 chunks are 16.2 as one chain); the error against
// 64 bits is that of the chain (7.3e-4 with transitions of norm 0.97).  Only lkv_init_state does this: a request of a batch is rounded as
// one chain, whatever else is in the batch and wherever the scratch lies.
constexpr int kSplitChunks = 10;
bool gdn_splits(const lkv_init_desc *d, int n_req, int total) {
    return n_req == 1 && total >= kSplitChunks && total + total <= kInitIdxCap - 4 && d->family == LKV_FAMILY_GDN && d->compute != LKV_COMPUTE_FP32 && d->d_k == 128 &&
           d->d_v == 128 && 3LL * d->H <= sm_count();
}
size_t gdn_split_scratch(const lkv_init_desc *d, int n_req, int total) {
    return gdn_splits(d, n_req, total) ? 3 * sizeof(float) * static_cast<size_t>(d->H) * d->d_k * d->d_v : 0;
}
int gdn_split(InitArgs a, const int32_t *ids, int K, bool pool_bf16, float *scratch, cudaStream_t s) {
    const int half = (K + 1) / 2;
    float *S0 = a.S0;
    const size_t slot = static_cast<size_t>(a.H) * a.d_k * a.d_v;
    a.S0 = scratch;   // A, B, P
    a.n_req = 3;
    a.product = 2;
    a.off_ids = 4;
    a.idx.ptr = nullptr;
    a.idx.n = 4 + half + 2 * (K - half);
    const int32_t cu[4] = {0, half, K, K + (K - half)};
    std::copy(cu, cu + 4, a.idx.v);
    std::copy(ids, ids + K, a.idx.v + 4);
    std::copy(ids + half, ids + K, a.idx.v + 4 + K);
    if (launch_init_gdn_exact_tensor(a, pool_bf16, s) != cudaSuccess) return LKV_ERR_CUDA;
    InitArgs b = a;   // chunks A, B of a pool whose second transition is P
    b.states = scratch; b.transitions = scratch + slot; b.S0 = S0; b.n_req = 1; b.n_chunks = 2; b.product = -1;
    const int32_t list[4] = {0, 2, 0, 1};
    b.off_ids = 2;
    b.idx.n = 4;
    std::copy(list, list + 4, b.idx.v);
    return launch_init_gdn_exact_tensor(b, false, s) == cudaSuccess ? LKV_OK : LKV_ERR_CUDA;
}

// may_split: lkv_init_state, whose one request may be composed in halves
int init_impl(const void *states, const void *transitions, const int32_t *chunk_ids, const int32_t *cu_k,
              int n_req, int mode, const int32_t *sel_index, void *S0, const lkv_init_desc *d, void *stream, bool may_split = false) {
    int st = check_init_desc(d);
    if (st != LKV_OK) return st;
    if (mode != LKV_INIT_LAST && mode != LKV_INIT_INDEX && mode != LKV_INIT_EXACT) return LKV_ERR_MODE;
    if (n_req < 0) return LKV_ERR_DIM;
    if (!cu_k) return LKV_ERR_NULL;
    if (cu_k[0] != 0) return LKV_ERR_INDEX;
    int max_k = 0;
    for (int r = 0; r < n_req; ++r) {
        if (cu_k[r + 1] < cu_k[r]) return LKV_ERR_INDEX;
        max_k = cu_k[r + 1] - cu_k[r] > max_k ? cu_k[r + 1] - cu_k[r] : max_k;
    }
    const int total = cu_k[n_req];
    if (total > 0 && !chunk_ids) return LKV_ERR_NULL;
    for (int i = 0; i < total; ++i)
        if (chunk_ids[i] < 0 || chunk_ids[i] >= d->n_chunks) return LKV_ERR_INDEX;
    if (mode == LKV_INIT_INDEX) {
        if (n_req > 0 && !sel_index) return LKV_ERR_NULL;
        for (int r = 0; r < n_req; ++r) {
            const int K = cu_k[r + 1] - cu_k[r];
            if (K > 0 && (sel_index[r] < 0 || sel_index[r] >= K)) return LKV_ERR_INDEX;
        }
    }
    if (n_req == 0) return LKV_OK;
    if (!S0) return LKV_ERR_NULL;
    if (total > 0 && !states) return LKV_ERR_NULL;
    const bool exact = mode == LKV_INIT_EXACT && max_k >= 2;
    if (exact && !transitions) return LKV_ERR_NULL;
    if (!aligned16(S0) || !aligned16(states) || (exact && !aligned16(transitions))) return LKV_ERR_ALIGN;
    const bool pool_bf16 = d->state_dtype == LKV_DTYPE_BF16;
    {
        const size_t state_elems = static_cast<size_t>(d->H) * d->d_k * d->d_v;
        const size_t out_bytes = sizeof(float) * state_elems * n_req;
        const size_t pool_bytes = (pool_bf16 ? 2 : 4) * state_elems * d->n_chunks;
        const size_t tr_bytes = sizeof(float) * static_cast<size_t>(d->n_chunks) * d->H *
                                (d->family == LKV_FAMILY_GDN ? static_cast<size_t>(d->d_k) * d->d_k : 1);
        if (overlaps(S0, out_bytes, states, total > 0 ? pool_bytes : 0) || (exact && overlaps(S0, out_bytes, transitions, tr_bytes)))
            return LKV_ERR_OVERLAP;
    }
    if (d->d_v % (pool_bf16 ? 8 : 4) != 0) return LKV_ERR_UNSUPPORTED;

    const int n_ints = (n_req + 1) + (mode == LKV_INIT_INDEX ? n_req : 0) + total;
    if (!d->workspace || d->workspace_bytes < ws_bytes_for(n_ints, kInitIdxCap)) return LKV_ERR_WORKSPACE;
    if (!aligned16(d->workspace)) return LKV_ERR_ALIGN;

    InitArgs a;
    a.states = states;
    a.transitions = static_cast<const float *>(transitions);
    a.S0 = static_cast<float *>(S0);
    a.n_req = n_req;
    a.H = d->H;
    a.d_k = d->d_k;
    a.d_v = d->d_v;
    a.n_chunks = d->n_chunks;
    a.status = static_cast<int32_t *>(d->workspace);
    std::vector<int32_t> ints;
    ints.reserve(n_ints);
    ints.insert(ints.end(), cu_k, cu_k + n_req + 1);
    a.off_sel = -1;
    if (mode == LKV_INIT_INDEX) {
        a.off_sel = static_cast<int32_t>(ints.size());
        ints.insert(ints.end(), sel_index, sel_index + n_req);
    }
    a.off_ids = static_cast<int32_t>(ints.size());
    if (total > 0) ints.insert(ints.end(), chunk_ids, chunk_ids + total);

    // kernel choice (no launch has happened yet: an unsupported request leaves everything untouched)
    enum { kSingle, kMamba, kGdnFp32, kGdnTensor } which;
    if (!exact) {
        which = kSingle;  // LAST, INDEX, and EXACT with K <= 1 everywhere are plain copies
        a.off_sel = (mode == LKV_INIT_INDEX) ? a.off_sel : -1;
    } else if (d->family == LKV_FAMILY_MAMBA2) {
        which = kMamba;
    } else {
        const bool tensor_fits = init_gdn_exact_tensor_supported(a, pool_bf16);
        if (d->compute == LKV_COMPUTE_TENSOR && !tensor_fits) return LKV_ERR_UNSUPPORTED;
        which = (d->compute != LKV_COMPUTE_FP32 && tensor_fits) ? kGdnTensor : kGdnFp32;
        if (which == kGdnFp32 && (2 * d->d_k * 32 + 32 * (d->d_k + 1)) * sizeof(float) > 227 * 1024) return LKV_ERR_UNSUPPORTED;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // (a caller whose workspace is smaller than lkv_workspace_bytes() asks for gets the chain in one)
    const size_t head = ws_bytes_for(n_ints, kInitIdxCap);
    if (may_split && which == kGdnTensor && gdn_splits(d, n_req, total) && d->workspace_bytes >= head + gdn_split_scratch(d, n_req, total))
        return gdn_split(a, chunk_ids, total, pool_bf16, reinterpret_cast<float *>(static_cast<char *>(d->workspace) + head), s);
    st = place_indices(a.idx, ints, d->workspace, s);
    if (st != LKV_OK) return st;
    cudaError_t e = cudaSuccess;
    switch (which) {
        case kSingle: e = launch_init_single(a, pool_bf16, s); break;
        case kMamba:
            e = init_mamba_stream_supported(a, pool_bf16) ? launch_init_mamba_exact_stream(a, pool_bf16, s)
                                                          : launch_init_mamba_exact(a, pool_bf16, s);
            break;
        case kGdnFp32: e = launch_init_gdn_exact_fp32(a, pool_bf16, s); break;
        case kGdnTensor: e = launch_init_gdn_exact_tensor(a, pool_bf16, s, true, shares_chunks(chunk_ids, total, d)); break;
    }
    return e == cudaSuccess ? LKV_OK : LKV_ERR_CUDA;
}

// Shared checks of the two scan descriptors' sequence layout; fills `cu` with the
// offsets the kernels will use.
int check_seqs(int T_total, int n_seq, const int32_t *cu_seqlens, std::vector<int32_t> &cu) {
    if (T_total < 0 || n_seq < 0) return LKV_ERR_DIM;
    if (!cu_seqlens) {
        if (n_seq != 1) return LKV_ERR_NULL;
        cu = {0, T_total};
        return LKV_OK;
    }
    if (cu_seqlens[0] != 0 || cu_seqlens[n_seq] != T_total) return LKV_ERR_INDEX;
    for (int i = 0; i < n_seq; ++i)
        if (cu_seqlens[i + 1] < cu_seqlens[i]) return LKV_ERR_INDEX;
    cu.assign(cu_seqlens, cu_seqlens + n_seq + 1);
    return LKV_OK;
}

// Appends to cu[n_seq + 1] the launch order of the sequences: longest first (ties by index), so that the CTAs of the
// long sequences, which are scheduled in grid order, start first and the short ones fill the tail of the launch.
void append_launch_order(std::vector<int32_t> &cu, int n_seq) {
    std::vector<int32_t> order(n_seq);
    for (int i = 0; i < n_seq; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(),
                     [&](int32_t x, int32_t y) { return cu[x + 1] - cu[x] > cu[y + 1] - cu[y]; });
    cu.insert(cu.end(), order.begin(), order.end());
}

// A single sequence fills (heads / 2) of the SMs (two heads per CTA) and is a chain of blocks.  Cut into segments, it runs as
// three launches: the states the first segments reach on their own (no outputs), the composition of every segment's initial
// state (Eq. 6), all segments with outputs side by side.
constexpr int kSsdBlock = 128, kGdnBlock = 64;   // tokens
std::vector<int32_t> segment_tokens(const Cut &c, int block, int T_total) {
    std::vector<int32_t> at(c.n + 1);
    for (int i = 0; i <= c.n; ++i) at[i] = std::min<long long>(static_cast<long long>(block) * c.at[i], T_total);
    return at;
}
Cut ssd_cut(const lkv_ssd_desc *d, int n_seq) {
    if (n_seq != 1 || d->io_dtype != LKV_DTYPE_BF16 || d->compute == LKV_COMPUTE_FP32 || d->H < 1 || d->G < 1 || d->H % d->G ||
        d->P != 64 || d->N != 128 || d->T_total < 1)
        return Cut{1, {0}};
    const int pairs = d->G * ((d->H / d->G + 1) / 2);
    return ssd_cut_blocks((d->T_total - 1) / kSsdBlock + 1, pairs, sm_count());
}
// local states and log-decays of the first segments, initial states of all but the first
size_t ssd_segment_scratch(const lkv_ssd_desc *d, int segs) {
    if (segs < 2) return 0;
    const size_t slot = sizeof(float) * static_cast<size_t>(d->H) * d->N * d->P;
    return 2 * (segs - 1) * slot + align_up(sizeof(float) * static_cast<size_t>(segs - 1) * d->H, 256);
}
int ssd_segmented(SsdArgs a, const Cut &cut, char *scratch, cudaStream_t s) {
    const int segs = cut.n;
    const size_t slot = static_cast<size_t>(a.H) * a.N * a.P;
    float *local = reinterpret_cast<float *>(scratch), *init = local + (segs - 1) * slot, *lam = init + (segs - 1) * slot;
    const std::vector<int32_t> tokens = segment_tokens(cut, kSsdBlock, a.T_total);
    auto bounds = [&](SsdArgs &b, int n) {
        b.n_seq = n;
        b.cu.ptr = nullptr;
        b.cu.n = 2 * n + 1;
        for (int i = 0; i <= n; ++i) b.cu.v[i] = tokens[i];
        for (int i = 0; i < n; ++i) b.cu.v[n + 1 + i] = i;
    };
    SsdArgs p1 = a;
    bounds(p1, segs - 1);
    p1.y = nullptr; p1.S_T = local; p1.st_bf16 = 0; p1.n_s0 = 1; p1.st_first = 0; p1.lam = lam;
    if (launch_ssd_scan_tensor(p1, s) != cudaSuccess) return LKV_ERR_CUDA;
    InitArgs c;
    c.states = local; c.transitions = lam; c.S0 = init; c.n_req = segs - 1; c.H = a.H; c.d_k = a.N; c.d_v = a.P; c.n_chunks = segs - 1;
    c.off_sel = -1; c.off_ids = segs; c.status = a.status; c.idx.ptr = nullptr;
    int at = segs;
    for (int r = 0; r < segs - 1; ++r) {
        c.idx.v[r] = at - segs;
        for (int j = 0; j <= r; ++j) c.idx.v[at++] = j;
    }
    c.idx.v[segs - 1] = at - segs;
    c.idx.n = at;
    if (launch_init_mamba_exact_stream(c, false, s) != cudaSuccess) return LKV_ERR_CUDA;
    SsdArgs p3 = a;
    bounds(p3, segs);
    p3.n_s0 = 1; p3.S0_more = init; p3.st_first = segs - 1;
    return launch_ssd_scan_tensor(p3, s) == cudaSuccess ? LKV_OK : LKV_ERR_CUDA;
}

// The same for the GDN scan (one head per CTA), where the first pass also computes the transitions of the segments between the
// first and the last.
Cut gdn_cut(const lkv_gdn_desc *d, int n_seq) {
    if (n_seq != 1 || d->io_dtype != LKV_DTYPE_BF16 || d->compute == LKV_COMPUTE_FP32 || d->d_k != 128 || d->d_v != 128 || d->T_total < 1)
        return Cut{1, {0}};
    return gdn_cut_blocks((d->T_total - 1) / kGdnBlock + 1, d->H_v, sm_count());
}
// local states and transitions of all segments but the last, initial states of all but the first
size_t gdn_segment_scratch(const lkv_gdn_desc *d, int n) {
    if (n < 2) return 0;
    return 3 * static_cast<size_t>(n - 1) * sizeof(float) * d->H_v * d->d_k * d->d_v;
}
// at: first tokens of the n segments and T_total, whole blocks.  tensor: the scans run on the tensor cores, and so does the
// composition unless the call asked for fp32 arithmetic.
// own_cut: the library chose the segments, so the passes fill the GPU.  A number of the caller's may leave a third of it idle: then
// the composition does not start early, because its waiting CTAs would hold the free SMs and leave the last pass packed onto
// neighbouring SMs, which share an instruction cache (3 segments of 16384 tokens, 32 heads: 339 us against 316; at the
// library's own cut, 4 segments there, 283 against 286).
int gdn_segmented(const GdnArgs &a, const lkv_gdn_desc *d, const std::vector<int32_t> &at, bool own_cut, bool tensor, void *scratch, cudaStream_t s) {
    const int n = static_cast<int>(at.size()) - 1, m = n - 1;
    const bool io_bf16 = d->io_dtype == LKV_DTYPE_BF16;
    const size_t slot = static_cast<size_t>(a.H_v) * a.d_k * a.d_v;
    float *local = static_cast<float *>(scratch), *trans = local + m * slot, *init = trans + m * slot;
    // the scan over the first k segments as sequences and n_tr transition sequences
    auto scan = [&](GdnArgs &b, int k, int n_tr) {
        b.n_ranges = b.tr_first = k;
        b.n_seq = k + n_tr;
        std::vector<int32_t> ints(at.begin(), at.begin() + k + 1), order(b.n_seq);
        auto len = [&](int sq) { const int r = sq < k ? sq : sq - k + b.tr_src0; return at[r + 1] - at[r]; };
        for (int i = 0; i < b.n_seq; ++i) order[i] = i;
        std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return len(x) > len(y); });
        ints.insert(ints.end(), order.begin(), order.end());
        const int st = place_indices(b.cu, ints, d->workspace, s);
        if (st != LKV_OK) return st;
        return (tensor ? launch_gdn_scan_tensor(b, s) : launch_gdn_scan_fp32(b, io_bf16, s)) == cudaSuccess ? LKV_OK : LKV_ERR_CUDA;
    };
    GdnArgs p1 = a;
    p1.tr_src0 = 1;
    p1.o = nullptr; p1.S_T = local; p1.st_bf16 = 0; p1.n_s0 = 1; p1.tr_out = trans + slot;   // transition of segment j at trans + j slots
    int st = scan(p1, m, std::max(m - 1, 0));
    if (st != LKV_OK) return st;
    InitArgs k;
    k.states = local; k.transitions = trans; k.S0 = init; k.n_req = m; k.H = a.H_v; k.d_k = a.d_k; k.d_v = a.d_v; k.n_chunks = m;
    k.off_sel = -1; k.off_ids = n; k.status = a.status;
    std::vector<int32_t> ints(n);
    for (int r = 0; r < m; ++r) {   // segment r + 1 starts from segments 0 .. r
        ints[r + 1] = ints[r] + r + 1;
        for (int j = 0; j <= r; ++j) ints.push_back(j);
    }
    st = place_indices(k.idx, ints, d->workspace, s);
    if (st != LKV_OK) return st;
    const bool tf32 = d->compute != LKV_COMPUTE_FP32 && init_gdn_exact_tensor_supported(k, false);
    if ((tf32 ? launch_init_gdn_exact_tensor(k, false, s, own_cut) : launch_init_gdn_exact_fp32(k, false, s)) != cudaSuccess) return LKV_ERR_CUDA;
    GdnArgs p3 = a;
    p3.n_s0 = 1; p3.S0_more = init; p3.st_first = n - 1;
    return scan(p3, n, 0);
}

}  // namespace

extern "C" {

int lkv_init_state(const void *states, const void *transitions, int K, int mode, void *S0,
                   const lkv_init_desc *d, void *stream) {
    if (!d) return LKV_ERR_NULL;
    if (K < 0) return LKV_ERR_DIM;
    std::vector<int32_t> ids;
    const int32_t *idp = d->chunk_ids;
    if (!idp) {
        ids.resize(K);
        for (int i = 0; i < K; ++i) ids[i] = i;
        idp = ids.data();
    }
    const int32_t cu_k[2] = {0, K};
    const int32_t sel[1] = {d->sel_index};
    return init_impl(states, transitions, idp, cu_k, 1, mode, sel, S0, d, stream, true);
}

int lkv_init_state_batched(const void *states, const void *transitions, const int32_t *chunk_ids,
                           const int32_t *cu_k, int n_req, int mode, const int32_t *sel_index, void *S0,
                           const lkv_init_desc *d, void *stream) {
    return init_impl(states, transitions, chunk_ids, cu_k, n_req, mode, sel_index, S0, d, stream);
}

// lkv_gdn_fwd, and with `transition` set the scan from S = I with v = 0 whose final state is the chunk transition
// what: 0 = scan, 1 = chunk transitions (start from S = I, v read as zeros), 2 = one step of the online fold (v read as
// zeros, S_add added to the final state), 3 = local states and transitions of every sequence in one launch: d->n_seq = 2 m
// sequences over the m ranges of d->cu_seqlens, the last m of them transition sequences that write to tr_out
// segments (of a scan of one sequence): cut there, with this scratch, instead of where gdn_cut says
static int gdn_impl(const void *q, const void *k, const void *v, const float *g, const float *beta,
                    const float *S0, void *o, void *S_T, const lkv_gdn_desc *d, void *stream, int what,
                    const float *S_add = nullptr, float *tr_out = nullptr, const std::vector<int32_t> *segments = nullptr,
                    bool own_cut = true, void *scratch = nullptr) {
    const bool transition = what == 1;
    if (!d) return LKV_ERR_NULL;
    if (!dtype_ok(d->io_dtype) || !compute_ok(d->compute) || !dtype_ok(d->state_dtype)) return LKV_ERR_MODE;
    const bool st_bf16 = d->state_dtype == LKV_DTYPE_BF16;
    if (st_bf16 && S_T && S_T == S0) return LKV_ERR_OVERLAP;   // an fp32 input cannot be a bf16 output
    if (d->H_k < 1 || d->H_v < 1 || d->d_k < 1 || d->d_v < 1 || d->H_v % d->H_k != 0) return LKV_ERR_DIM;
    std::vector<int32_t> cu;
    const int n_ranges = what == 3 ? d->n_seq / 2 : d->n_seq;
    int st = check_seqs(d->T_total, n_ranges, d->cu_seqlens, cu);
    if (st != LKV_OK) return st;
    if (d->n_seq == 0) return LKV_OK;
    if ((transition || what == 3) && d->d_k != d->d_v) return LKV_ERR_DIM;
    if (d->T_total > 0 && (!q || !k || !g || !beta)) return LKV_ERR_NULL;
    if (what == 0 && d->T_total > 0 && !v) return LKV_ERR_NULL;
    if (!o && !S_T) return LKV_ERR_NULL;   // nothing to compute
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(g) || !aligned16(beta) || !aligned16(S0) ||
        !aligned16(o) || !aligned16(S_T))
        return LKV_ERR_ALIGN;
    if (!d->workspace || d->workspace_bytes < ws_bytes_for(2 * d->n_seq + 1, kScanIdxCap)) return LKV_ERR_WORKSPACE;
    if (!aligned16(d->workspace)) return LKV_ERR_ALIGN;
    {
        // outputs may not overlap inputs (S_T == S0 exactly is the one allowed alias) nor each other
        const size_t es = d->io_dtype == LKV_DTYPE_BF16 ? 2 : 4, T = static_cast<size_t>(d->T_total);
        const size_t qk_b = es * T * d->H_k * d->d_k, v_b = es * T * d->H_v * d->d_v, gb_b = sizeof(float) * T * d->H_v;
        const size_t st_in = sizeof(float) * static_cast<size_t>(n_ranges) * d->H_v * d->d_k * d->d_v;
        const size_t st_b = st_bf16 ? st_in / 2 : st_in;
        const void *in[6] = {q, k, v, g, beta, S0};
        const size_t in_b[6] = {qk_b, qk_b, v ? v_b : 0, gb_b, gb_b, S0 ? st_in : 0};
        for (int i = 0; i < 6; ++i) {
            if (overlaps(o, o ? v_b : 0, in[i], in_b[i])) return LKV_ERR_OVERLAP;
            if (!(i == 5 && S_T == S0) && overlaps(S_T, S_T ? st_b : 0, in[i], in_b[i])) return LKV_ERR_OVERLAP;
        }
        if (overlaps(o, o ? v_b : 0, S_T, S_T ? st_b : 0)) return LKV_ERR_OVERLAP;
    }

    GdnArgs a;
    a.q = q; a.k = k; a.v = v; a.g = g; a.beta = beta; a.S0 = S0; a.o = o; a.S_T = static_cast<float *>(S_T);
    a.S_add = S_add; a.st_bf16 = st_bf16 ? 1 : 0;
    a.n_seq = d->n_seq; a.T_total = d->T_total; a.H_k = d->H_k; a.H_v = d->H_v; a.d_k = d->d_k; a.d_v = d->d_v;
    a.scale = d->scale != 0.f ? d->scale : 1.0f / sqrtf(static_cast<float>(d->d_k));
    a.s0_identity = transition ? 1 : 0;
    a.n_ranges = n_ranges; a.tr_first = n_ranges; a.tr_src0 = 0; a.tr_out = tr_out;
    a.n_s0 = d->n_seq; a.st_first = 0; a.S0_more = nullptr;
    a.status = static_cast<int32_t *>(d->workspace);
    const bool io_bf16 = d->io_dtype == LKV_DTYPE_BF16;
    const bool tensor_fits = gdn_scan_tensor_supported(a, io_bf16);
    const bool fp32_fits = gdn_scan_fp32_supported(d->d_k, d->d_v);
    bool use_tensor;
    if (d->compute == LKV_COMPUTE_TENSOR) {
        if (!tensor_fits) return LKV_ERR_UNSUPPORTED;
        use_tensor = true;
    } else if (d->compute == LKV_COMPUTE_FP32) {
        if (!fp32_fits) return LKV_ERR_UNSUPPORTED;
        use_tensor = false;
    } else {
        if (!tensor_fits && !fp32_fits) return LKV_ERR_UNSUPPORTED;
        use_tensor = tensor_fits;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (segments) {
        // S_T on top of S0 is written while S0 is read: it goes through the scratch, behind what gdn_segmented uses of it
        const bool alias = S_T && S_T == S0;
        const size_t st_elems = static_cast<size_t>(d->H_v) * d->d_k * d->d_v;
        if (alias) a.S_T = static_cast<float *>(scratch) + 3 * (segments->size() - 2) * st_elems;
        st = gdn_segmented(a, d, *segments, own_cut, use_tensor, scratch, s);
        if (st == LKV_OK && alias && cudaMemcpyAsync(S_T, a.S_T, sizeof(float) * st_elems, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
            st = LKV_ERR_CUDA;
        return st;
    }
    // A long sequence that leaves SMs idle runs in segments (a caller whose workspace is smaller than
    // lkv_workspace_bytes() asked for gets the plain scan; S_T on top of S0 would be written while S0 is read)
    const Cut cut = use_tensor && what == 0 && S_T != S0 && o ? gdn_cut(d, d->n_seq) : Cut{1, {0}};
    const size_t head = ws_bytes_for(2 * d->n_seq + 1, kScanIdxCap);
    if (cut.n > 1 && d->workspace_bytes >= head + gdn_segment_scratch(d, cut.n))
        return gdn_segmented(a, d, segment_tokens(cut, kGdnBlock, d->T_total), true, true, static_cast<char *>(d->workspace) + head, s);
    // States and transitions: one CTA for both of a chunk and head, once two CTAs would no longer find an SM each (32 heads, 3 x 1024 tokens
    // 57 -> 39 us); up to there they are faster side by side (2 x 2048 tokens 55 us, in one CTA 67).  Without v, read as zeros, or
    // in fp32 arithmetic the scan runs twice.
    const bool both = what == 3 && use_tensor && v && static_cast<long long>(a.n_seq) * a.H_v > sm_count();
    if (both) {
        a.n_seq = n_ranges;
        append_launch_order(cu, n_ranges);
    } else if (what == 3) {
        // launch order over all sequences, longest first; transition sequence j runs over range j - m
        std::vector<int32_t> order(d->n_seq);
        auto len = [&](int sq) { const int r = sq % n_ranges; return cu[r + 1] - cu[r]; };
        for (int i = 0; i < d->n_seq; ++i) order[i] = i;
        std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return len(x) > len(y); });
        cu.insert(cu.end(), order.begin(), order.end());
    } else {
        append_launch_order(cu, d->n_seq);
    }
    st = place_indices(a.cu, cu, d->workspace, s);
    if (st != LKV_OK) return st;
    const cudaError_t e = both ? launch_gdn_build_tensor(a, s) : use_tensor ? launch_gdn_scan_tensor(a, s) : launch_gdn_scan_fp32(a, io_bf16, s);
    return e == cudaSuccess ? LKV_OK : LKV_ERR_CUDA;
}

int lkv_gdn_fwd(const void *q, const void *k, const void *v, const float *g, const float *beta,
                const float *S0, void *o, void *S_T, const lkv_gdn_desc *d, void *stream) {
    return gdn_impl(q, k, v, g, beta, S0, o, S_T, d, stream, 0);
}

int lkv_gdn_chunk_transition(const void *k, const float *g, const float *beta, float *transitions,
                             const lkv_gdn_desc *d, void *stream) {
    if (d && d->n_seq > 0 && !transitions) return LKV_ERR_NULL;
    // q is not needed for the state: the key tensor stands in for it (its read-outs are not written)
    if (d && d->state_dtype != LKV_DTYPE_F32) return LKV_ERR_MODE;   // transitions are fp32
    return gdn_impl(k, k, nullptr, g, beta, nullptr, nullptr, transitions, d, stream, 1);
}

int lkv_init_state_fold(const void *states, const void *k, const float *g, const float *beta,
                        const int32_t *cu_tokens, int K, void *S0, const lkv_init_desc *d, int H_k, int io_dtype,
                        void *stream) {
    int st = check_init_desc(d);
    if (st != LKV_OK) return st;
    if (d->family != LKV_FAMILY_GDN || !dtype_ok(io_dtype)) return LKV_ERR_MODE;
    if (d->state_dtype != LKV_DTYPE_F32) return LKV_ERR_UNSUPPORTED;   // the cached states are added in fp32
    if (K < 0 || H_k < 1 || d->H % H_k != 0 || d->d_k != d->d_v) return LKV_ERR_DIM;
    if (!states || !S0 || !cu_tokens) return LKV_ERR_NULL;
    if (K > 0 && !d->chunk_ids && K > d->n_chunks) return LKV_ERR_INDEX;
    if (cu_tokens[0] != 0) return LKV_ERR_INDEX;
    for (int c = 0; c < d->n_chunks; ++c)
        if (cu_tokens[c + 1] < cu_tokens[c]) return LKV_ERR_INDEX;
    std::vector<int32_t> ids(K);
    for (int j = 0; j < K; ++j) {
        ids[j] = d->chunk_ids ? d->chunk_ids[j] : j;
        if (ids[j] < 0 || ids[j] >= d->n_chunks) return LKV_ERR_INDEX;
    }
    if (K >= 2 && cu_tokens[d->n_chunks] > 0 && (!k || !g || !beta)) return LKV_ERR_NULL;
    // the first chunk's state (or the zero state) through the single-state path, then one scan per later chunk
    lkv_init_desc first = *d;
    first.sel_index = 0;
    st = lkv_init_state(states, nullptr, K, LKV_INIT_INDEX, S0, &first, stream);
    if (st != LKV_OK) return st;
    const size_t es = io_dtype == LKV_DTYPE_BF16 ? 2 : 4;
    const size_t state_elems = static_cast<size_t>(d->H) * d->d_k * d->d_v;
    for (int j = 1; j < K; ++j) {
        const int c = ids[j], t0 = cu_tokens[c], len = cu_tokens[c + 1] - t0;
        lkv_gdn_desc sd{};
        sd.T_total = len; sd.n_seq = 1; sd.cu_seqlens = nullptr; sd.H_k = H_k; sd.H_v = d->H; sd.d_k = d->d_k; sd.d_v = d->d_v;
        sd.io_dtype = io_dtype; sd.compute = d->compute; sd.scale = 0.f; sd.state_dtype = LKV_DTYPE_F32;
        sd.workspace = d->workspace; sd.workspace_bytes = d->workspace_bytes;
        const char *kc = static_cast<const char *>(k) + es * static_cast<size_t>(t0) * H_k * d->d_k;
        const float *gc = g ? g + static_cast<size_t>(t0) * d->H : nullptr;
        const float *bc = beta ? beta + static_cast<size_t>(t0) * d->H : nullptr;
        st = gdn_impl(kc, kc, nullptr, gc, bc, static_cast<const float *>(S0), nullptr, S0, &sd, stream, 2,
                      static_cast<const float *>(states) + static_cast<size_t>(c) * state_elems);
        if (st != LKV_OK) return st;
    }
    return LKV_OK;
}

// Where the sequence is cut.  n_segments == 0: as lkv_gdn_fwd cuts it; what runs in fp32 arithmetic into as many segments as keep
// both scanning passes within one round of CTAs on this GPU -- (2 n - 3) H_v and n H_v CTAs, one per SM -- and none shorter
// than 512 tokens.
static std::vector<int32_t> segments_of(const lkv_gdn_desc *d, int n_segments) {
    if (n_segments == 0) {
        if (d->io_dtype == LKV_DTYPE_BF16 && d->compute != LKV_COMPUTE_FP32 && d->d_k == 128 && d->d_v == 128)
            return segment_tokens(gdn_cut(d, 1), kGdnBlock, d->T_total);
        n_segments = std::max(1, std::min((sm_count() / d->H_v + 3) / 2, d->T_total / 512));
    }
    // equal, on multiples of 64 tokens: every block of the segmented scan is a block of the plain one
    const long long per = (static_cast<long long>(d->T_total) + n_segments - 1) / n_segments;
    std::vector<int32_t> at(n_segments + 1);
    for (int i = 0; i <= n_segments; ++i) at[i] = static_cast<int32_t>(std::min<long long>(i * ((per + 63) / 64 * 64), d->T_total));
    return at;
}

size_t lkv_gdn_segmented_scratch_bytes(const lkv_gdn_desc *d, int n_segments) {
    if (!d || n_segments < 0 || d->T_total < 0 || d->H_v < 1 || d->d_k < 1 || d->d_v < 1) return 0;
    if (n_segments == 0) n_segments = static_cast<int>(segments_of(d, 0).size()) - 1;
    if (n_segments < 2) return 0;
    return sizeof(float) * (4 * static_cast<size_t>(n_segments) - 3) * d->H_v * d->d_k * d->d_v;
}

int lkv_gdn_fwd_segmented(const void *q, const void *k, const void *v, const float *g, const float *beta,
                          const float *S0, void *o, void *S_T, const lkv_gdn_desc *d, int n_segments,
                          void *scratch, size_t scratch_bytes, void *stream) {
    if (!d) return LKV_ERR_NULL;
    if (n_segments < 0) return LKV_ERR_DIM;
    std::vector<int32_t> at;
    if (n_segments == 0) {
        if (d->H_v < 1 || d->T_total < 0) return LKV_ERR_DIM;
        at = segments_of(d, 0);
        n_segments = static_cast<int>(at.size()) - 1;
    }
    if (n_segments == 1) return lkv_gdn_fwd(q, k, v, g, beta, S0, o, S_T, d, stream);
    if (d->n_seq != 1 || d->state_dtype != LKV_DTYPE_F32) return LKV_ERR_UNSUPPORTED;   // one sequence, fp32 final state
    if (d->d_k != d->d_v) return LKV_ERR_DIM;                                            // transitions are d_k x d_k
    if (d->T_total < 0) return LKV_ERR_DIM;
    if (d->cu_seqlens && (d->cu_seqlens[0] != 0 || d->cu_seqlens[1] != d->T_total)) return LKV_ERR_INDEX;
    if (!scratch || scratch_bytes < lkv_gdn_segmented_scratch_bytes(d, n_segments)) return LKV_ERR_WORKSPACE;
    if (!aligned16(scratch)) return LKV_ERR_ALIGN;
    // the longest index lists of the three launches
    const int n = n_segments;
    if (n > (1 << 15) || !d->workspace || d->workspace_bytes < ws_bytes_for(2 * (2 * n - 3) + 1, kScanIdxCap) ||
        d->workspace_bytes < ws_bytes_for(n + n * (n - 1) / 2, kInitIdxCap))
        return LKV_ERR_WORKSPACE;
    const bool own_cut = !at.empty();
    if (!own_cut) at = segments_of(d, n);
    return gdn_impl(q, k, v, g, beta, S0, o, S_T, d, stream, 0, nullptr, nullptr, &at, own_cut, scratch);
}

int lkv_stage_chunks(const void *host_states, const void *host_transitions, const int32_t *chunk_ids, int n_ids,
                     void *dev_states, void *dev_transitions, int capacity, int32_t *staged_ids, int32_t *n_staged,
                     const lkv_init_desc *d, void *stream) {
    int st = check_init_desc(d);
    if (st != LKV_OK) return st;
    if (n_ids < 0 || capacity < 0) return LKV_ERR_DIM;
    if (!n_staged) return LKV_ERR_NULL;
    *n_staged = 0;
    if (n_ids == 0) return LKV_OK;
    if (!host_states || !dev_states || !chunk_ids || !staged_ids) return LKV_ERR_NULL;
    if ((host_transitions == nullptr) != (dev_transitions == nullptr)) return LKV_ERR_NULL;   // both pools or neither
    if (!aligned16(dev_states) || !aligned16(dev_transitions)) return LKV_ERR_ALIGN;
    // slots in order of first appearance; everything is checked before the first copy is queued
    std::vector<int32_t> slot_of(d->n_chunks, -1), order;
    for (int i = 0; i < n_ids; ++i) {
        const int32_t c = chunk_ids[i];
        if (c < 0 || c >= d->n_chunks) return LKV_ERR_INDEX;
        if (slot_of[c] < 0) {
            slot_of[c] = static_cast<int32_t>(order.size());
            order.push_back(c);
        }
    }
    if (static_cast<long long>(order.size()) > capacity) return LKV_ERR_WORKSPACE;
    const size_t es = d->state_dtype == LKV_DTYPE_BF16 ? 2 : 4;
    const size_t state_b = es * static_cast<size_t>(d->H) * d->d_k * d->d_v;
    const size_t trans_b = sizeof(float) * static_cast<size_t>(d->H) * (d->family == LKV_FAMILY_GDN ? static_cast<size_t>(d->d_k) * d->d_k : 1);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    for (size_t k = 0; k < order.size(); ++k) {
        const size_t c = static_cast<size_t>(order[k]);
        if (cudaMemcpyAsync(static_cast<char *>(dev_states) + k * state_b, static_cast<const char *>(host_states) + c * state_b,
                            state_b, cudaMemcpyHostToDevice, s) != cudaSuccess ||
            (host_transitions &&
             cudaMemcpyAsync(static_cast<char *>(dev_transitions) + k * trans_b, static_cast<const char *>(host_transitions) + c * trans_b,
                             trans_b, cudaMemcpyHostToDevice, s) != cudaSuccess)) {
            cudaGetLastError();
            return LKV_ERR_CUDA;
        }
    }
    for (int i = 0; i < n_ids; ++i) staged_ids[i] = slot_of[chunk_ids[i]];
    *n_staged = static_cast<int32_t>(order.size());
    return LKV_OK;
}

int lkv_gdn_chunk_artifacts(const void *k, const void *v, const float *g, const float *beta, float *states,
                            float *transitions, const lkv_gdn_desc *d, void *stream) {
    if (!d) return LKV_ERR_NULL;
    if (d->state_dtype != LKV_DTYPE_F32) return LKV_ERR_MODE;
    if (d->n_seq > 0 && (!states || !transitions)) return LKV_ERR_NULL;
    if (d->n_seq < 0 || d->n_seq > (1 << 29)) return LKV_ERR_DIM;
    if (!aligned16(transitions)) return LKV_ERR_ALIGN;
    {
        const size_t st_b = sizeof(float) * static_cast<size_t>(d->n_seq > 0 ? d->n_seq : 0) * d->H_v * d->d_k * d->d_v;
        if (overlaps(states, st_b, transitions, st_b)) return LKV_ERR_OVERLAP;
    }
    lkv_gdn_desc d2 = *d;
    d2.n_seq = 2 * d->n_seq;   // every chunk twice: once as a scan from the empty state, once as a transition sequence
    // q is not needed for the states: the key tensor stands in for it (its read-outs are not written)
    return gdn_impl(k, k, v, g, beta, nullptr, nullptr, states, &d2, stream, 3, nullptr, transitions);
}

int lkv_mamba_chunk_logdecay(const float *dt, const float *A, float *logdecay, const lkv_ssd_desc *d, void *stream) {
    if (!d) return LKV_ERR_NULL;
    if (d->H < 1) return LKV_ERR_DIM;
    std::vector<int32_t> cu;
    int st = check_seqs(d->T_total, d->n_seq, d->cu_seqlens, cu);
    if (st != LKV_OK) return st;
    if (d->n_seq == 0) return LKV_OK;
    if (!A || !logdecay || (d->T_total > 0 && !dt)) return LKV_ERR_NULL;
    if (!aligned16(dt) || !aligned16(A) || !aligned16(logdecay)) return LKV_ERR_ALIGN;
    if (!d->workspace || d->workspace_bytes < ws_bytes_for(d->n_seq + 1, kScanIdxCap)) return LKV_ERR_WORKSPACE;
    if (!aligned16(d->workspace)) return LKV_ERR_ALIGN;
    SsdArgs a{};
    a.dt = dt; a.A = A; a.n_seq = d->n_seq; a.T_total = d->T_total; a.H = d->H; a.P = d->P; a.N = d->N; a.G = d->G;
    a.status = static_cast<int32_t *>(d->workspace);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int longest = 0;
    for (int i = 0; i < d->n_seq; ++i) longest = std::max(longest, cu[i + 1] - cu[i]);
    st = place_indices(a.cu, cu, d->workspace, s);
    if (st != LKV_OK) return st;
    return launch_mamba_logdecay(a, logdecay, longest, s) == cudaSuccess ? LKV_OK : LKV_ERR_CUDA;
}

size_t lkv_state_rel_error_workspace_bytes(int n_states, size_t state_elems) {
    if (n_states < 0 || state_elems == 0) return 0;
    return align_up(sizeof(float) * 2 * static_cast<size_t>(n_states) * state_err_parts(state_elems) + 16, 256);
}

int lkv_state_rel_error(const float *S_init, const float *S_ref, float *rel_err, int n_states, size_t state_elems,
                        void *workspace, size_t workspace_bytes, void *stream) {
    if (n_states < 0 || state_elems == 0 || state_elems % 4 != 0 || n_states > 65535) return LKV_ERR_DIM;
    if (n_states == 0) return LKV_OK;
    if (!S_init || !S_ref || !rel_err) return LKV_ERR_NULL;
    if (!aligned16(S_init) || !aligned16(S_ref) || !aligned16(workspace)) return LKV_ERR_ALIGN;
    if (!workspace || workspace_bytes < lkv_state_rel_error_workspace_bytes(n_states, state_elems)) return LKV_ERR_WORKSPACE;
    const cudaError_t e = launch_state_rel_error(S_init, S_ref, rel_err, n_states, state_elems,
                                                 static_cast<float *>(workspace), static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? LKV_OK : LKV_ERR_CUDA;
}

int lkv_ssd_fwd(const void *x, const float *dt, const float *A, const void *B, const void *C,
                const float *S0, void *y, void *S_T, const lkv_ssd_desc *d, void *stream) {
    if (!d) return LKV_ERR_NULL;
    if (!dtype_ok(d->io_dtype) || !compute_ok(d->compute) || !dtype_ok(d->state_dtype)) return LKV_ERR_MODE;
    const bool st_bf16 = d->state_dtype == LKV_DTYPE_BF16;
    if (st_bf16 && S_T && S_T == S0) return LKV_ERR_OVERLAP;   // an fp32 input cannot be a bf16 output
    if (d->H < 1 || d->P < 1 || d->N < 1 || d->G < 1 || d->H % d->G != 0) return LKV_ERR_DIM;
    std::vector<int32_t> cu;
    int st = check_seqs(d->T_total, d->n_seq, d->cu_seqlens, cu);
    if (st != LKV_OK) return st;
    if (d->n_seq == 0) return LKV_OK;
    if (!A) return LKV_ERR_NULL;
    if (d->T_total > 0 && (!x || !dt || !B || !C)) return LKV_ERR_NULL;
    if (!y && !S_T) return LKV_ERR_NULL;   // nothing to compute
    if (!aligned16(x) || !aligned16(dt) || !aligned16(A) || !aligned16(B) || !aligned16(C) || !aligned16(S0) ||
        !aligned16(y) || !aligned16(S_T))
        return LKV_ERR_ALIGN;
    if (!d->workspace || d->workspace_bytes < ws_bytes_for(2 * d->n_seq + 1, kScanIdxCap)) return LKV_ERR_WORKSPACE;
    if (!aligned16(d->workspace)) return LKV_ERR_ALIGN;
    {
        // outputs may not overlap inputs (S_T == S0 exactly is the one allowed alias) nor each other
        const size_t es = d->io_dtype == LKV_DTYPE_BF16 ? 2 : 4, T = static_cast<size_t>(d->T_total);
        const size_t x_b = es * T * d->H * d->P, bc_b = es * T * d->G * d->N, dt_b = sizeof(float) * T * d->H;
        const size_t st_in = sizeof(float) * static_cast<size_t>(d->n_seq) * d->H * d->N * d->P;
        const size_t st_b = st_bf16 ? st_in / 2 : st_in;
        const void *in[6] = {x, dt, A, B, C, S0};
        const size_t in_b[6] = {x_b, dt_b, sizeof(float) * d->H, bc_b, bc_b, S0 ? st_in : 0};
        for (int i = 0; i < 6; ++i) {
            if (overlaps(y, y ? x_b : 0, in[i], in_b[i])) return LKV_ERR_OVERLAP;
            if (!(i == 5 && S_T == S0) && overlaps(S_T, S_T ? st_b : 0, in[i], in_b[i])) return LKV_ERR_OVERLAP;
        }
        if (overlaps(y, y ? x_b : 0, S_T, S_T ? st_b : 0)) return LKV_ERR_OVERLAP;
    }

    SsdArgs a;
    a.x = x; a.dt = dt; a.A = A; a.B = B; a.C = C; a.S0 = S0; a.y = y; a.S_T = static_cast<float *>(S_T);
    a.st_bf16 = st_bf16 ? 1 : 0;
    a.n_seq = d->n_seq; a.T_total = d->T_total; a.H = d->H; a.P = d->P; a.N = d->N; a.G = d->G;
    a.status = static_cast<int32_t *>(d->workspace);
    const bool io_bf16 = d->io_dtype == LKV_DTYPE_BF16;
    const bool tensor_fits = ssd_scan_tensor_supported(a, io_bf16);
    const bool fp32_fits = ssd_scan_fp32_supported(d->N, d->P);
    bool use_tensor;
    if (d->compute == LKV_COMPUTE_TENSOR) {
        if (!tensor_fits) return LKV_ERR_UNSUPPORTED;
        use_tensor = true;
    } else if (d->compute == LKV_COMPUTE_FP32) {
        if (!fp32_fits) return LKV_ERR_UNSUPPORTED;
        use_tensor = false;
    } else {
        if (!tensor_fits && !fp32_fits) return LKV_ERR_UNSUPPORTED;
        use_tensor = tensor_fits;
    }
    a.n_s0 = d->n_seq; a.st_first = 0; a.S0_more = nullptr; a.lam = nullptr;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const Cut cut = use_tensor && S_T != S0 && y ? ssd_cut(d, d->n_seq) : Cut{1, {0}};
    const size_t head = ws_bytes_for(2 * d->n_seq + 1, kScanIdxCap);
    if (cut.n > 1 && d->workspace_bytes >= head + ssd_segment_scratch(d, cut.n))
        return ssd_segmented(a, cut, static_cast<char *>(d->workspace) + head, s);
    append_launch_order(cu, d->n_seq);
    st = place_indices(a.cu, cu, d->workspace, s);
    if (st != LKV_OK) return st;
    const cudaError_t e = use_tensor ? launch_ssd_scan_tensor(a, s) : launch_ssd_scan_fp32(a, io_bf16, s);
    return e == cudaSuccess ? LKV_OK : LKV_ERR_CUDA;
}

size_t lkv_workspace_bytes(int which, const void *desc, int n_units, int n_index) {
    if (!desc || n_units < 0 || n_index < 0) return 0;
    switch (which) {
        case LKV_WS_INIT_LIST:
        case LKV_WS_INIT: {
            const lkv_init_desc *d = static_cast<const lkv_init_desc *>(desc);
            const long long ints = 2LL * n_units + 1 + n_index;
            if (check_init_desc(d) != LKV_OK || ints > INT32_MAX) return 0;
            return ws_bytes_for(static_cast<int>(ints), kInitIdxCap) + (which == LKV_WS_INIT ? gdn_split_scratch(d, n_units, n_index) : 0);
        }
        case LKV_WS_GDN: {
            const lkv_gdn_desc *d = static_cast<const lkv_gdn_desc *>(desc);
            return ws_bytes_for(2 * n_units + 1, kScanIdxCap) + gdn_segment_scratch(d, gdn_cut(d, n_units).n);
        }
        case LKV_WS_SSD: {
            const lkv_ssd_desc *d = static_cast<const lkv_ssd_desc *>(desc);
            return ws_bytes_for(2 * n_units + 1, kScanIdxCap) + ssd_segment_scratch(d, ssd_cut(d, n_units).n);
        }
        default: return 0;
    }
}

int lkv_device_status(const void *workspace, void *stream) {
    if (!workspace) return LKV_ERR_NULL;
    int32_t word = 0;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(&word, workspace, sizeof(word), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        cudaGetLastError();
        return LKV_ERR_CUDA;
    }
    return word == 0 ? LKV_OK : LKV_ERR_DEVICE_TIMEOUT;
}

int lkv_selftest_bounded_wait(int poll_limit, void *workspace, void *stream) {
    if (!workspace) return LKV_ERR_NULL;
    if (poll_limit < 1 || poll_limit > (1 << 20)) return LKV_ERR_DIM;
    if (!aligned16(workspace)) return LKV_ERR_ALIGN;
    return launch_selftest_bounded_wait(static_cast<uint32_t>(poll_limit), static_cast<int32_t *>(workspace),
                                        static_cast<cudaStream_t>(stream)) == cudaSuccess ? LKV_OK : LKV_ERR_CUDA;
}

const char *lkv_status_string(int status) {
    switch (status) {
        case LKV_OK: return "ok";
        case LKV_ERR_NULL: return "a required pointer is NULL";
        case LKV_ERR_DIM: return "bad dimension";
        case LKV_ERR_MODE: return "unknown mode, family, dtype or compute value";
        case LKV_ERR_INDEX: return "index out of range or offsets not monotone";
        case LKV_ERR_ALIGN: return "pointer not 16-byte aligned";
        case LKV_ERR_UNSUPPORTED: return "no kernel for this shape or dtype";
        case LKV_ERR_WORKSPACE: return "workspace missing or too small";
        case LKV_ERR_CUDA: return "CUDA runtime call failed";
        case LKV_ERR_DEVICE_TIMEOUT: return "a bounded device-side wait ran out";
        case LKV_ERR_OVERLAP: return "an output buffer overlaps an input or another output";
        default: return "unknown status";
    }
}

int lkv_version(void) { return LKV_VERSION; }

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// Batched state initialisation for callers that cannot allocate device memory and therefore
// have no workspace to pass (an engine whose allocator is closed on the request path, a
// plugin running inside another component's memory budget).  The scratch is this fixed array,
// part of the library image on every GPU that loads it.
//
// In host code the name `g_static_scratch` is only a handle for the runtime, NOT a device
// address: the address a kernel may use has to be asked for with cudaGetSymbolAddress, once
// per device and with that device current.
static __device__ __align__(256) unsigned char g_static_scratch[LKV_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
void *g_static_scratch_addr[kMaxDevices];  // per device, filled on the first call there

// Device address of the static scratch on the current device (nullptr on failure).
void *static_scratch_for_current_device() {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return nullptr;
    }
    void *p = __atomic_load_n(&g_static_scratch_addr[dev], __ATOMIC_ACQUIRE);
    if (!p) {
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return nullptr;
        }
        __atomic_store_n(&g_static_scratch_addr[dev], p, __ATOMIC_RELEASE);
    }
    return p;
}
}  // namespace

// Status word of the static scratch on the current device: read, and cleared if it was set (nobody else can).
extern "C" int lkv_device_status_static(void *stream) {
    void *scratch = static_scratch_for_current_device();
    if (!scratch) return LKV_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int32_t word = 0;
    if (cudaMemcpyAsync(&word, scratch, sizeof(word), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        cudaGetLastError();
        return LKV_ERR_CUDA;
    }
    if (word == 0) return LKV_OK;
    if (cudaMemsetAsync(scratch, 0, sizeof(word), s) != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) {
        cudaGetLastError();
        return LKV_ERR_CUDA;
    }
    return LKV_ERR_DEVICE_TIMEOUT;
}

extern "C" int lkv_init_state_batched_static(const void *states, const void *transitions, const int32_t *chunk_ids,
                                             const int32_t *cu_k, int n_req, int mode, const int32_t *sel_index,
                                             void *S0, const lkv_init_desc *d, void *stream) {
    if (!d) return LKV_ERR_NULL;
    if (n_req < 0) return LKV_ERR_DIM;
    if (!cu_k) return LKV_ERR_NULL;
    // size check first: beyond the fixed array there is nowhere to put the index list
    const long long n_ints = 2LL * n_req + 1 + (cu_k[n_req] > 0 ? cu_k[n_req] : 0);
    if (n_ints > LKV_STATIC_MAX_INDEX) return LKV_ERR_WORKSPACE;
    void *scratch = static_scratch_for_current_device();
    if (!scratch) return LKV_ERR_CUDA;
    lkv_init_desc local = *d;
    local.workspace = scratch;
    local.workspace_bytes = LKV_STATIC_SCRATCH_BYTES;
    return init_impl(states, transitions, chunk_ids, cu_k, n_req, mode, sel_index, S0, &local, stream);
}
