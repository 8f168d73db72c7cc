// The drafting step of one row of logits by the warps of a CTA, shared by the kernels that draft (bv_sample.cu) and by the
// decoding loop in one kernel (bv_loop.cu): the row is swept once by 16 streaming warps in 128 sub-segments, and one more warp
// forms the normaliser, finds the sub-segment that holds the sample and walks through it.
#pragma once
#include "bv_flow_common.cuh"

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
template <bool SHORT, class Sum>
__device__ __forceinline__ void s_put(float M, Sum s, int lane, SubSegment<SHORT>* to) {
    float2 v = make_float2(static_cast<float>(s), M);
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
        // (One reference for all of them, the rounded maximum of their logits: a test of every vector's sum before the next one's
        // exponentials was a chain of dependent steps.  256 rows of 128256 bf16 logits 22.5 -> 21.9 us, 300 of 65536 18.4 -> 16.4,
        // 1000 of 32768 27.3 -> 24.6; 2048 of 256000 196 -> 201.  No exponent is above 1/2.  A normaliser comes out lower by 1e-8 on
        // average, a 24th of what an exponential may be off by; over nine kinds of rows, 5000 to 20000 of each, its distance from 64 bits
        // changed by between +6 % (5.7e-8 -> 6.1e-8, V = 128256, T = 0.8) and -5 % (6.5e-8 -> 6.1e-8, V = 152064, T = 0.6), +0.3 % over all.)
        uint4 top = raw[0];
#pragma unroll
        for (int j = 1; j < kSInFlight; ++j) top = vec_max<DT>(top, raw[j]);
        float v[EPV];
        R::unpack(top, v);
        const float y = fmaxf(M, rintf(warp_max(vec_max<EPV>(v)) * kf));
        s = ref_sum(s, M, y);
        M = y;
#pragma unroll
        for (int j = 0; j < kSInFlight; ++j) {
            if (base + 32 * j < u1) {
                R::unpack(raw[j], v);
                s += f_exp_sum<EPV>(v, kf, -M);
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

// What a lane knows of the 128 sub-segment sums of a row, of which it speaks for four: the sub-segment in which u times their
// total falls (the first non-empty one whose inclusive prefix exceeds it, else the last non-empty one), and what is left of
// it at that sub-segment's start.  w: this lane's sums; inc: their prefix over the lanes; all in double, in index order.
__device__ __forceinline__ int s_pick(const double (&w)[4], double inc, double t, int lane, double& rem) {
    const double l1 = w[0], l2 = l1 + w[1], l3 = l2 + w[2], l4 = l3 + w[3];
    double exc = shfl_up_d(inc, 1);
    if (lane == 0) exc = 0.0;
    const double p0 = exc, p1 = exc + l1, p2 = exc + l2, p3 = exc + l3, p4 = exc + l4;
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
    rem = t - shfl_d(bef, src);
    return __shfl_sync(0xffffffffu, 4 * lane + e, src);
}
// The sampling warp's part, up to the walk through the sampled sub-segment: the row's normaliser {reference, sum} from the 128
// pairs, and the sub-segment that the uniform u selects (-1 for a row with a NaN or +inf logit or without a finite one).
// release_pairs >= 0: a named barrier at which the warp arrives once it has read the pairs.
template <bool SHORT>
__device__ __forceinline__ int s_locate(const SubSegment<SHORT>* seg, float u, int lane, int release_pairs, double* norm, double& rem) {
    // ---- normaliser and the sampled sub-segment (fp64 prefix sums, index order) ----
    float m[4], za[4], zb[4];
    double w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) s_get<SHORT>(seg[32 * j + lane], m[j], w[j], za[j], zb[j]);
    const float Mrow = warp_max(fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])));
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        w[j] = SHORT ? ref_sum(w[j], m[j], Mrow) : static_cast<double>(ref_sum(za[j], m[j], Mrow)) + static_cast<double>(ref_sum(zb[j], m[j], Mrow));
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
    const bool ok = Mrow > kNoRef && Mrow < INFINITY && row_sum_ok(Z) && row_sum_ok(total);
    if (release_pairs >= 0) named_bar_arrive(release_pairs, kSAllThreads);   // (the pairs are in registers: their buffer may be written again)
    norm[0] = Mrow;
    norm[1] = Z;
    return ok ? s_pick(w, inc, static_cast<double>(u) * total, lane, rem) : -1;
}
// The whole of it: the token that the uniform u selects (inverse CDF in index order; -1 where there is none).
template <int DT, bool SHORT>
__device__ __forceinline__ int s_draw_row(const char* row, int units, float kf, const SubSegment<SHORT>* seg, float u,
                                          int lane, int release_pairs, double* norm) {
    double rem = 0.0;
    const int sel = s_locate<SHORT>(seg, u, lane, release_pairs, norm, rem);
    if (sel < 0) return -1;
    int a0, a1;
    s_range(units, sel / kSSub, sel % kSSub, a0, a1);
    return f_rescan<DT>(row, nullptr, a0, a1, lane, kf, 1.f, -static_cast<float>(norm[0]), 0.f, rem);
}
// the row's log-normaliser from what s_draw_row left
__device__ __forceinline__ float s_lse(int found, const double* norm) {
    return found >= 0 ? static_cast<float>((norm[0] + log2(norm[1])) * 0.693147180559945309417232) : __int_as_float(0x7fc00000);
}

}  // namespace bv
