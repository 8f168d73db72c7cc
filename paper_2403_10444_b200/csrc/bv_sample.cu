// The drafting step of Algorithm 3 for rows of logits: one token per row drawn from
// softmax(logits / T) by inverse CDF in vocabulary-index order with a supplied uniform, and the
// row's log-normaliser (what the verification needs of a draft row besides the logits).
//
// Persistent CTAs take rows round-robin.  Each of 16 warps streams its contiguous sixteenth of the
// row once, in eight sub-segments, and leaves each sub-segment's {integer reference, sum 2^{z k - M}}
// in shared memory; a seventeenth warp, a row behind, combines the 128 pairs (fp64 for the
// normaliser and for the sampler's prefix sums), finds the sub-segment that holds u * Z and rescans
// that one - a few KB still in L2 - in index order for the token.  Each logit is read from HBM once.
#include <cmath>
#include <cstdint>

#include "bv_sample_row.cuh"

#include "../../include/bv.h"

namespace bv {

template <int DT, bool SHORT>
__global__ void __launch_bounds__(kSAllThreads, 2)
sample_rows_kernel(const char* logits, const float* uni, int rows, int V, float kf, int32_t* tokens, float* lse) {
    using R = Raw<DT>;
    constexpr int EPV = R::EPV;
    constexpr size_t ESZ = (DT == kF32) ? 4 : 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int units = V / EPV;
    const size_t row_bytes = static_cast<size_t>(V) * ESZ;
    __shared__ SubSegment<SHORT> seg[2][kSSegs];

    // The streaming warps sweep the CTA's rows one after the other and leave each row's pairs in one of
    // two buffers; the sampling warp follows, a row behind or so, and draws each row's token from them.
    // Two named barriers per buffer order the two sides, producer and consumer: "full" (the 16 streaming
    // warps arrive when the row's pairs are written, the sampling warp waits) and "empty" (the sampling
    // warp arrives when it has read them, the streaming warps wait before they write that buffer again,
    // two rows later).  The streaming warps never wait for one another: there is no barrier across a row.
    // Every wait ends: the row count is the same for all warps of the CTA, each row has exactly one
    // arrival and one wait per side, and the streaming side waits for row `it - 2` only from row 2 on.
    const int nmine = rows > static_cast<int>(blockIdx.x) ? (rows - 1 - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x) + 1 : 0;
    if (warp < kSWarps) {
        for (int it = 0; it < nmine; ++it) {
            if (it >= 2) named_bar_sync(kBarEmpty + (it & 1), kSAllThreads);
            const int r = blockIdx.x + it * gridDim.x;
            s_sweep_row<DT, SHORT>(logits + static_cast<size_t>(r) * row_bytes, units, kf, warp, lane, seg[it & 1]);
            __threadfence_block();
            named_bar_arrive(kBarFull + (it & 1), kSAllThreads);
        }
    } else {
        for (int it = 0; it < nmine; ++it) {
            named_bar_sync(kBarFull + (it & 1), kSAllThreads);
            const int r = blockIdx.x + it * gridDim.x;
            double norm[2];
            // (row it + 2 waits for the release of this buffer; the last two rows have nobody waiting)
            const int found = s_draw_row<DT, SHORT>(logits + static_cast<size_t>(r) * row_bytes, units, kf, seg[it & 1], uni[r],
                                             lane, it + 2 < nmine ? kBarEmpty + (it & 1) : -1, norm);
            if (lane == 0) {
                tokens[r] = found;
                if (lse) lse[r] = s_lse(found, norm);
            }
        }
    }
}

// The drafting step of Algorithm 3 as a whole for a model whose next-token logits depend on the last
// token only (a table [V, V], row t = logits after token t): X_1 .. X_gamma one after the other, each
// from the row of the token before it.  One CTA per sequence; a step is the sweep of one row by the
// 16 streaming warps, a barrier, the draw by the sampling warp, a barrier.  A token that is not in
// [0, V) (a first token out of range, or a step whose row could not be sampled) ends the sequence's
// chain: the remaining tokens are -1 and their normalisers NaN.
// Before that, where the chain belongs to the decoding loop (loop.out_len), the sequence is extended by what the verification
// of the iteration before has emitted, and the chain starts from the last of it.
struct LoopState {
    const int32_t* out;       // [B, gamma+1], out_len [B]: the last verification's outputs; out_len null: none yet
    const int32_t* out_len;
    int32_t* cur;             // [B] last token of every sequence
    int32_t* seq;             // [B, width] tokens generated so far, lengths [B] of them
    long long* lengths;
    int32_t* tau;             // [B] accepted drafts of that iteration
    int32_t* fault;           // set if a sequence reported a data fault
    int width;
};
__device__ __forceinline__ void extend_sequence(const LoopState& loop, int b, int gamma, int lane) {
    const int32_t* out = loop.out + static_cast<size_t>(b) * (gamma + 1);
    const int len = loop.out_len[b], n = len < 1 ? 1 : len;
    const long long pos = loop.lengths[b];
    for (int i = lane; i < n; i += 32)
        if (pos + i < loop.width) loop.seq[static_cast<size_t>(b) * loop.width + pos + i] = out[i];
    __syncwarp();
    if (lane == 0) {
        loop.cur[b] = out[n - 1];
        loop.lengths[b] = pos + n;
        loop.tau[b] = len - 1;
        if (len < 1) atomicExch(loop.fault, 1);
    }
}
__global__ void extend_kernel(const LoopState loop, int B, int gamma) {
    const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (b < B) extend_sequence(loop, b, gamma, threadIdx.x & 31);
}

template <int DT, bool SHORT>
__global__ void __launch_bounds__(kSAllThreads, 2)
draft_chain_kernel(const char* table, const int32_t* first, const float* uni, int B, int gamma, int V, float kf,
                   int32_t* tokens, float* lse, const LoopState loop) {
    using R = Raw<DT>;
    constexpr int EPV = R::EPV;
    constexpr size_t ESZ = (DT == kF32) ? 4 : 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int units = V / EPV;
    const size_t row_bytes = static_cast<size_t>(V) * ESZ;
    __shared__ SubSegment<SHORT> seg[kSSegs];
    __shared__ int s_next[2];
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        if (loop.out_len != nullptr) {
            if (warp == 0) extend_sequence(loop, b, gamma, lane);
            __syncthreads();
        }
        int last = first[b];
        for (int i = 0; i < gamma; ++i) {
            const bool ok = last >= 0 && last < V;
            const char* row = table + static_cast<size_t>(ok ? last : 0) * row_bytes;
            if (warp < kSWarps && ok) s_sweep_row<DT, SHORT>(row, units, kf, warp, lane, seg);
            const float u = uni[static_cast<size_t>(i) * B + b];
            __syncthreads();
            int found = -1;
            double norm[2] = {0.0, 0.0};
            if (warp == kSWarps) {
                if (ok) found = s_draw_row<DT, SHORT>(row, units, kf, seg, u, lane, -1, norm);
                if (lane == 0) s_next[i & 1] = found;
            }
            __syncthreads();
            last = s_next[i & 1];     // (written again two steps on, after another barrier)
            // the streaming warps are on the next row already
            if (warp == kSWarps && lane == 0) {
                tokens[static_cast<size_t>(b) * gamma + i] = found;
                if (lse) lse[static_cast<size_t>(b) * gamma + i] = s_lse(found, norm);
            }
        }
    }
}

}  // namespace bv

namespace {
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) % 16) == 0; }
}  // namespace

extern "C" int bv_sample_draft(const void* logits, const float* uniforms, int rows, int V, int dtype,
                               float temperature, int32_t* out_tokens, float* out_lse, void* stream) {
    if (!logits || !uniforms || !out_tokens) return BV_ERR_INVALID_ARG;
    if (rows < 0 || V < 1) return BV_ERR_INVALID_ARG;
    if (!(temperature > 0.f) || !std::isfinite(temperature)) return BV_ERR_INVALID_ARG;
    if (dtype != BV_DTYPE_F32 && dtype != BV_DTYPE_BF16) return BV_ERR_INVALID_ARG;
    const size_t row_bytes = static_cast<size_t>(V) * (dtype == BV_DTYPE_F32 ? 4 : 2);
    if (row_bytes % 16 != 0 || !aligned16(logits)) return BV_ERR_UNSUPPORTED;
    bv::note_launches(0);
    if (rows == 0) return BV_OK;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return bv::note_cuda_error(e);
    const int grid = rows < 2 * sms ? rows : 2 * sms;
    const float kf = static_cast<float>(1.4426950408889634 / static_cast<double>(temperature));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool f32 = dtype == BV_DTYPE_F32, brief = bv::s_short(row_bytes);
    const auto kernel = f32 ? (brief ? bv::sample_rows_kernel<bv::kF32, true> : bv::sample_rows_kernel<bv::kF32, false>)
                            : (brief ? bv::sample_rows_kernel<bv::kBF16, true> : bv::sample_rows_kernel<bv::kBF16, false>);
    kernel<<<grid, bv::kSAllThreads, 0, st>>>(static_cast<const char*>(logits), uniforms, rows, V, kf, out_tokens, out_lse);
    e = cudaGetLastError();
    if (e != cudaSuccess) return bv::note_cuda_error(e);
    bv::note_launches(1);
    return BV_OK;
}

namespace {
// One launch of the drafting chain; the arguments have been checked.
cudaError_t launch_chain(const void* table, const int32_t* first, const float* uni, int B, int gamma, int V, int dtype, float temperature,
                         int32_t* tokens, float* lse, const bv::LoopState& loop, cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int grid = B < 2 * sms ? B : 2 * sms;
    const float kf = static_cast<float>(1.4426950408889634 / static_cast<double>(temperature));
    const bool f32 = dtype == BV_DTYPE_F32, brief = bv::s_short(static_cast<size_t>(V) * (f32 ? 4 : 2));
    const auto kernel = f32 ? (brief ? bv::draft_chain_kernel<bv::kF32, true> : bv::draft_chain_kernel<bv::kF32, false>)
                            : (brief ? bv::draft_chain_kernel<bv::kBF16, true> : bv::draft_chain_kernel<bv::kBF16, false>);
    kernel<<<grid, bv::kSAllThreads, 0, st>>>(static_cast<const char*>(table), first, uni, B, gamma, V, kf, tokens, lse, loop);
    return cudaGetLastError();
}
}  // namespace

extern "C" int bv_draft_chain(const void* draft_table, const int32_t* first_tokens, const float* uniforms, int B, int gamma,
                              int V, int dtype, float temperature, int32_t* out_tokens, float* out_lse, void* stream) {
    if (!draft_table || !first_tokens || !uniforms || !out_tokens) return BV_ERR_INVALID_ARG;
    if (B < 0 || gamma < 1 || V < 1) return BV_ERR_INVALID_ARG;
    if (!(temperature > 0.f) || !std::isfinite(temperature)) return BV_ERR_INVALID_ARG;
    if (dtype != BV_DTYPE_F32 && dtype != BV_DTYPE_BF16) return BV_ERR_INVALID_ARG;
    const size_t row_bytes = static_cast<size_t>(V) * (dtype == BV_DTYPE_F32 ? 4 : 2);
    if (row_bytes % 16 != 0 || !aligned16(draft_table)) return BV_ERR_UNSUPPORTED;
    bv::note_launches(0);
    if (B == 0) return BV_OK;
    const cudaError_t e = launch_chain(draft_table, first_tokens, uniforms, B, gamma, V, dtype, temperature, out_tokens, out_lse,
                                       bv::LoopState{}, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return bv::note_cuda_error(e);
    bv::note_launches(1);
    return BV_OK;
}

extern "C" int bv_decode_loop(const void* target_table, const void* draft_table, const int32_t* first_tokens, const float* u_draft,
                              const float* u_verify, int iterations, int B, int gamma, int V, int dtype, float temperature, int algo,
                              int32_t* out_tokens, int64_t* out_lengths, int32_t* out_tau, int32_t* out_drafted, int32_t* out_fault,
                              int32_t* work, void* stream) {
    if (!target_table || !draft_table || !first_tokens || !u_draft || !u_verify || !out_tokens || !out_lengths || !out_tau ||
        !out_drafted || !out_fault || !work) return BV_ERR_INVALID_ARG;
    if (iterations < 1 || B < 1 || gamma < 1 || V < 1 || algo < 0 || algo > 3) return BV_ERR_INVALID_ARG;
    if (!(temperature > 0.f) || !std::isfinite(temperature)) return BV_ERR_INVALID_ARG;
    if (dtype != BV_DTYPE_F32 && dtype != BV_DTYPE_BF16) return BV_ERR_INVALID_ARG;
    const size_t row_bytes = static_cast<size_t>(V) * (dtype == BV_DTYPE_F32 ? 4 : 2);
    if (row_bytes % 16 != 0 || !aligned16(draft_table) || !aligned16(target_table) || gamma > BV_MAX_GAMMA || B > bv::kPhaseMaxB) return BV_ERR_UNSUPPORTED;
    const size_t b = static_cast<size_t>(B), width = static_cast<size_t>(iterations) * (gamma + 1);
    if (width > 0x7fffffffu) return BV_ERR_UNSUPPORTED;
    bv::note_launches(0);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e;
    int dev = 0, sms = 0;
    const int how = bv::loop_option();
    if (how == 0 && ((e = cudaGetDevice(&dev)) != cudaSuccess || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess))
        return bv::note_cuda_error(e);
    const bool fits = bv::loop_fits(V, dtype);
    auto one_kernel = [&]() -> int {
        const double kd = 1.4426950408889634073599246810019 / static_cast<double>(temperature);
        // (a last target row that is not wanted: the small-batch kernel sweeps every row and faults the sequence, the phase kernel does
        // not look; of a loop's calls, which of them takes it decides)
        const int last_counts = !(algo & 1) && bv::small_takes_tables(bv::kBlockVerify, algo < 2, B, gamma, row_bytes);
        const bv::LoopArgs args{target_table, draft_table, first_tokens, u_draft, u_verify, iterations, B, gamma, V, static_cast<int>(width),
                                static_cast<float>(kd), kd, algo & 1, last_counts, algo < 2, out_tokens, reinterpret_cast<long long*>(out_lengths),
                                out_tau, out_drafted, out_fault};
        if ((e = cudaMemsetAsync(out_fault, 0, 4, st)) != cudaSuccess || (e = bv::launch_loop(args, dtype, st)) != cudaSuccess) return bv::note_cuda_error(e);
        bv::note_launches(1);
        return BV_OK;
    };
    if (fits && (how == 1 || (how == 0 && bv::loop_pays(V, dtype, B, gamma, algo & 1, sms)))) return one_kernel();
    // work: last tokens, the last verification's outputs, the draft rows' normalisers
    int32_t* cur = work;
    int32_t* out = cur + b;
    int32_t* out_len = out + b * (gamma + 1);
    float* lse = reinterpret_cast<float*>(out_len + b);
    auto verify = [&](int n, bool probe) {
        return bv::run_tables(algo & 1 ? bv::kTokenVerify : bv::kBlockVerify, target_table, draft_table, cur, out_drafted + n * b * gamma,
                              u_verify + n * b * (gamma + 2), algo < 2 ? lse : nullptr, B, gamma, V, dtype, temperature, out, out_len, probe, st);
    };
    int rc = verify(0, true);
    const bool other = fits && how == 0;      // (where too few SMs can be had for the verification's kernels, the one kernel needs none at once)
    if (rc == BV_ERR_UNSUPPORTED && other) return one_kernel();
    if (rc != BV_OK) return rc;               // (before anything is enqueued)
    if ((e = cudaMemcpyAsync(cur, first_tokens, b * 4, cudaMemcpyDeviceToDevice, st)) != cudaSuccess ||
        (e = cudaMemsetAsync(out_tokens, 0xff, b * width * 4, st)) != cudaSuccess ||      // (-1)
        (e = cudaMemsetAsync(out_lengths, 0, b * 8, st)) != cudaSuccess ||
        (e = cudaMemsetAsync(out_fault, 0, 4, st)) != cudaSuccess)
        return bv::note_cuda_error(e);
    bv::LoopState loop{out, nullptr, cur, out_tokens, reinterpret_cast<long long*>(out_lengths), nullptr, out_fault, static_cast<int>(width)};
    int launches = 0;
    for (int n = 0; n < iterations; ++n) {
        if ((e = launch_chain(draft_table, cur, u_draft + n * b * gamma, B, gamma, V, dtype, temperature, out_drafted + n * b * gamma, lse, loop, st)) != cudaSuccess)
            return bv::note_cuda_error(e);
        rc = verify(n, false);
        if (rc == BV_ERR_UNSUPPORTED && other && n == 0) return one_kernel();      // (it writes all outputs anew)
        if (rc != BV_OK) return rc;
        loop.out_len = out_len;
        loop.tau = out_tau + n * b;
        launches += 2;
    }
    bv::extend_kernel<<<(B + 7) / 8, 256, 0, st>>>(loop, B, gamma);
    if ((e = cudaGetLastError()) != cudaSuccess) return bv::note_cuda_error(e);
    bv::note_launches(launches + 1);
    return BV_OK;
}
