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

#include "bv_flow_common.cuh"

#include "../../include/bv.h"

namespace bv {

constexpr int kSThreads = 512;                    // streaming threads; one more warp draws the samples
constexpr int kSWarps = kSThreads / 32;
constexpr int kSAllThreads = kSThreads + 32;
constexpr int kSSub = 8;                          // sub-segments per warp
constexpr int kSSegs = kSWarps * kSSub;           // 128: four per lane of warp 0
constexpr int kSInFlight = 8;                     // 16-byte loads a thread has in flight

// named barriers of a CTA (hardware barriers 1 .. 15; 0 is __syncthreads): all lanes of a warp take part,
// `threads` is the number of threads that arrive or wait at the barrier per use
constexpr int kBarFull = 1, kBarEmpty = 3;        // ids kBarFull + buffer, kBarEmpty + buffer
__device__ __forceinline__ void named_bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_bar_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// A warp's part of a row of `units` vectors is cut into sub-segments of whole runs of 32 vectors, one load of a warp: at most
// kSSub of them, `runs` runs each (the last ones of a short part are empty).
// vectors [a0, a1) of sub-segment `sub` of warp `warp`
__device__ __forceinline__ void s_part(int units, int warp, int& u0, int& u1, int& runs) {
    u0 = static_cast<int>(static_cast<long long>(units) * warp / kSWarps);
    u1 = static_cast<int>(static_cast<long long>(units) * (warp + 1) / kSWarps);
    runs = ((u1 - u0 + 31) / 32 + kSSub - 1) / kSSub;
    if (runs < 1) runs = 1;
}
__device__ __forceinline__ void s_range(int units, int warp, int sub, int& a0, int& a1) {
    int u0, u1, runs;
    s_part(units, warp, u0, u1, runs);
    a0 = min(u0 + sub * runs * 32, u1);
    a1 = min(a0 + runs * 32, u1);
}

// What a sub-segment leaves: its reference and its sum, in two parts that are added in double where the pairs are combined.
// The vectors that are joined in fp32 decide the precision of a normaliser.  In rows of 2048 vectors and more the parts are the
// sums of sixteen lanes each (of at most 32 vectors below 8192); in shorter ones (SHORT), of few vectors to a sub-segment, the
// lanes are joined in double.  (All 32 lanes joined in fp32: relative error of the normaliser of rows with a flat law 5.8e-9 on
// average at 1024 vectors, 4.1e-9 at 5000, where equal sub-segments of 8 and 39 vectors gave 2.5e-9 and 2.8e-9; like this 1.0e-9
// and 2.7e-9.  The double costs a step of a drafting chain at 128 vectors a row 0.2 of 3.1 us, nothing from 1024 vectors on.)
template <bool SHORT> struct alignas(16) SubSegment { float2 a, b; };                  // {sum of lanes 0 .. 15, M}, {of lanes 16 .. 31, M}
template <> struct alignas(16) SubSegment<true> { double z; float2 b; };              // {sum}, {M, -}
constexpr bool s_short(size_t row_bytes) { return row_bytes < static_cast<size_t>(2048) * 16; }
// (sub-segment `sub` of warp `warp` lies where lane (8 warp + sub) / 4 of the sampling warp finds it without bank conflicts)
__device__ __forceinline__ int s_place(int warp, int sub) { return (sub & 3) * 32 + warp * (kSSub / 4) + (sub >> 2); }
template <bool SHORT>
__device__ __forceinline__ void s_put(float M, float s, int lane, SubSegment<SHORT>* to) {
    float2 v = make_float2(s, M);
    if (SHORT) {
        const double z = warp_sum_d(static_cast<double>(s));
        v = lane == 0 ? make_float2(__int_as_float(__double2loint(z)), __int_as_float(__double2hiint(z))) : make_float2(M, 0.f);
    } else {
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
    }
    if ((lane & 15) == 0) reinterpret_cast<float2*>(to)[lane >> 4] = v;
}
__device__ __forceinline__ SubSegment<true> s_empty(SubSegment<true>*) { return {0.0, make_float2(kNoRef, 0.f)}; }
__device__ __forceinline__ SubSegment<false> s_empty(SubSegment<false>*) { return {make_float2(0.f, kNoRef), make_float2(0.f, kNoRef)}; }
template <bool SHORT>
__device__ __forceinline__ void s_get(const SubSegment<SHORT>& from, float& M, double& z, float& za, float& zb) {
    if constexpr (SHORT) { M = from.b.x; z = from.z; }
    else { M = from.a.y; za = from.a.x; zb = from.b.x; }
}

// One streaming warp's pass over its sixteenth of a row: the {reference, sum} pair of each of its
// sub-segments goes to `seg`.  The loads of kSInFlight runs are issued together whatever sub-segments they
// belong to.  (With one sub-segment's loads at a time a row of 2048 vectors, 16 to a sub-segment, waited for memory eight
// times: a step of a drafting chain, B = 128 sequences of 16384 bf16 logits, 13 us, now 5 us; 2048 rows of 128256 logits,
// 125 vectors to a sub-segment, 140 us, now 113 us: 4.7 TB/s.)
template <int DT, bool SHORT>
__device__ __forceinline__ void s_sweep_row(const char* row, int units, float kf, int warp, int lane, SubSegment<SHORT>* seg) {
    using R = Raw<DT>;
    constexpr int EPV = R::EPV;
    // (the warp's reference carries over from one sub-segment to the next: a sub-segment's pair is
    // its sum against the reference as it stood at its end, and only the first one has to find one)
    float M = kNoRef, s = 0.f;
    int u0, u1, runs;
    s_part(units, warp, u0, u1, runs);
    const uint4 ninf = make_uint4(R::kNegInf, R::kNegInf, R::kNegInf, R::kNegInf);
    int sub = 0, left = runs;
    for (int base = u0; base < u1; base += 32 * kSInFlight) {
        uint4 raw[kSInFlight];                    // all loads of the round are issued before any is used
#pragma unroll
        for (int j = 0; j < kSInFlight; ++j) {
            const int i = base + 32 * j + lane;
            raw[j] = i < u1 ? ld_stream_v4(row + static_cast<size_t>(i) * 16) : ninf;
        }
#pragma unroll
        for (int j = 0; j < kSInFlight; ++j) {
            if (base + 32 * j < u1) {
                float v[EPV];
                R::unpack(raw[j], v);
                f_accumulate<EPV>(v, kf, M, s);
                if (--left == 0) {                // the end of a sub-segment
                    s_put<SHORT>(M, s, lane, seg + s_place(warp, sub));
                    ++sub;
                    left = runs;
                    s = 0.f;
                }
            }
        }
    }
    if (left < runs) {
        s_put<SHORT>(M, s, lane, seg + s_place(warp, sub));
        ++sub;
    }
    if (lane >= sub && lane < kSSub) seg[s_place(warp, lane)] = s_empty(seg);
}

// The sampling warp's part: the row's normaliser from the 128 pairs and the token that the uniform u
// selects (inverse CDF in index order; -1 and a NaN normaliser for a row with a NaN or +inf logit or
// without a finite one).  release_pairs >= 0: a named barrier at which the warp arrives once it has
// read the pairs.
template <int DT, bool SHORT>
__device__ __forceinline__ int s_draw_row(const char* row, int units, float kf, const SubSegment<SHORT>* seg, float u,
                                          int lane, int release_pairs, double* norm) {
    // ---- normaliser and the sampled sub-segment (fp64 prefix sums, index order) ----
    float m[4], za[4], zb[4];
    double w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) s_get<SHORT>(seg[32 * j + lane], m[j], w[j], za[j], zb[j]);
    const float Mrow = warp_max(fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])));
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float to = ref_scale(m[j], Mrow);
        w[j] = SHORT ? w[j] * static_cast<double>(to) : static_cast<double>(za[j] * to) + static_cast<double>(zb[j] * to);
    }
    double Z = (w[0] + w[1]) + (w[2] + w[3]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) Z += shfl_xor_d(Z, off);
    // (the sums over sub-segments that locate the sample are formed in double: a token's cell can
    // be far narrower than fp32 resolves next to the mass before it)
    const double l1 = w[0], l2 = l1 + w[1], l3 = l2 + w[2], l4 = l3 + w[3];
    double inc = l4;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double o = shfl_up_d(inc, off);
        if (lane >= off) inc += o;
    }
    const double total = shfl_d(inc, 31);
    // a row with a NaN or +inf logit has a NaN / infinite sum or reference; one without a finite logit has none
    const bool ok = Mrow > kNoRef && Mrow < INFINITY && Z > 0.0 && Z < INFINITY && total > 0.0 && total < static_cast<double>(INFINITY);
    if (release_pairs >= 0) named_bar_arrive(release_pairs, kSAllThreads);   // (the pairs are in registers: their buffer may be written again)
    int found = -1;
    if (ok) {
        const double t = static_cast<double>(u) * total;
        double exc = shfl_up_d(inc, 1);
        if (lane == 0) exc = 0.0;
        const double p0 = exc, p1 = exc + l1, p2 = exc + l2, p3 = exc + l3, p4 = exc + l4;
        // first non-empty sub-segment whose inclusive prefix exceeds t, else the last non-empty one
        const bool h1 = p1 > t && w[0] > 0.0, h2 = p2 > t && w[1] > 0.0;
        const bool h3 = p3 > t && w[2] > 0.0, h4 = p4 > t && w[3] > 0.0;
        const unsigned hit = __ballot_sync(0xffffffffu, h1 || h2 || h3 || h4);
        const unsigned nz = __ballot_sync(0xffffffffu, l4 > 0.0);
        int e = 3; double bef = p3; int src;
        if (hit) {
            src = __ffs(hit) - 1;
            if (h1) { e = 0; bef = p0; } else if (h2) { e = 1; bef = p1; } else if (h3) { e = 2; bef = p2; }
        } else {
            src = 31 - __clz(nz);
            e = 0; bef = p0;
            if (w[3] > 0.0) { e = 3; bef = p3; } else if (w[2] > 0.0) { e = 2; bef = p2; }
            else if (w[1] > 0.0) { e = 1; bef = p1; }
        }
        const int sel = __shfl_sync(0xffffffffu, 4 * lane + e, src);
        const double before = shfl_d(bef, src);
        int a0, a1;
        s_range(units, sel / kSSub, sel % kSSub, a0, a1);
        found = f_rescan<DT>(row, nullptr, a0, a1, lane, kf, 1.f, -Mrow, 0.f, t - before);
    }
    norm[0] = Mrow;
    norm[1] = Z;
    return found;
}
// the row's log-normaliser from what s_draw_row left
__device__ __forceinline__ float s_lse(int found, const double* norm) {
    return found >= 0 ? static_cast<float>((norm[0] + log2(norm[1])) * 0.693147180559945309417232) : __int_as_float(0x7fc00000);
}

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
    if (rc != BV_OK) return rc;               // (before anything is enqueued)
    cudaError_t e;
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
        if ((rc = verify(n, false)) != BV_OK) return rc;
        loop.out_len = out_len;
        loop.tau = out_tau + n * b;
        launches += 2;
    }
    bv::extend_kernel<<<(B + 7) / 8, 256, 0, st>>>(loop, B, gamma);
    if ((e = cudaGetLastError()) != cudaSuccess) return bv::note_cuda_error(e);
    bv::note_launches(launches + 1);
    return BV_OK;
}
