// The decoding loop of Algorithm 3 for two last-token table models in one kernel: sequences are independent of one another
// in every step of it (Algorithms 1 and 2 look at one block), so a CTA takes a sequence through all iterations and nothing is
// ever exchanged between CTAs, nor left in memory between steps but the rows themselves.
//
// A drafting step is the sweep of the draft row of the last token by 16 streaming warps and the draw by one more, by the sampler's
// cut of a row and its choice of a sub-segment.  (Its sums in rows of up to 2048 vectors too, bit for bit; in longer ones the reference is
// raised every four runs here and every eight in bv_draft_chain, so a uniform within rounding of a cell's edge may fall to the neighbour.)
// Without supplied normalisers the verification still takes the one that the drafting step has formed, before it is rounded to
// 32 bits: sixteen lanes of it are joined in fp32 from 2048 vectors on, as there.  Both models' rows of a step are
// copied into shared memory at once; while the sampling warp draws, the streaming warps sweep the target row, so that when
// the block is drafted all normalisers of its verification are known.  What is left of the verification is the recursion
// of Eq. "def_as" or the tests of Algorithm 1 and, position after position from the top, the residual sums of the candidates
// (Eq. "pacc_block"), whose rows come from L2 once more.
//
// Bound: latency, gamma dependent rows and one or two dependent sweeps an iteration; bytes B (2 gamma + 1) rows an iteration.
// 128 sequences of gamma = 5 over V = 16384 in bf16, 8 iterations: 283 us, 35 an iteration (two launches an iteration, the
// chain and a verification by all SMs together with its waits for the whole batch: 606 us; the bytes take 56).
#include <climits>
#include <type_traits>

#include "bv_sample_row.cuh"

namespace bv {

struct LoopShared {
    double MP[kMaxGamma], ZP[kMaxGamma], MQ[kMaxGamma], ZQ[kMaxGamma];   // normalisers of the block's rows
    float zp[kMaxGamma], zq[kMaxGamma];   // logits of the drafted tokens
    float csc[kMaxGamma];                 // p_i Z_Q / Z_P
    double p[kMaxGamma];                  // p_i
    double wM[kSWarps], wZ[kSWarps];      // the streaming warps' shares of a target row
    double res[kSSegs];                   // residual sums of a position's sub-segments
    float u[kMaxGamma + 2];
    int tok[kMaxGamma];
    int next;                             // the token drawn last
    unsigned lo, hi;                      // candidates
    int last, over;                       // position gamma is the selected one; the iteration has ended
};

// A warp's part of a row into the row's image in shared memory; every lane reads the cells that it has asked for itself.
__device__ __forceinline__ void l_fetch(uint32_t image, const char* row, int units, int warp, int lane) {
    int u0, u1, runs;
    s_part(units, warp, u0, u1, runs);
    for (int i = u0 + lane; i < u1; i += 32) cp_async16_s(image + static_cast<uint32_t>(i) * 16u, row + static_cast<size_t>(i) * 16);
    cp_async_commit();
}
__device__ __forceinline__ uint4 l_cell(uint32_t image, int i, int u1, uint32_t pad) {
    return i < u1 ? lds128(image + static_cast<uint32_t>(i) * 16u) : make_uint4(pad, pad, pad, pad);
}
constexpr int kLoopRuns = 4;                      // runs of 32 vectors that a warp goes through together
// A step waits for each of these sweeps, and a warp has few runs of its row: what costs is the chain of dependent instructions,
// not their number.  So kLoopRuns runs share one reference, the rounded maximum of all their logits, found before the first
// exponential (a run at a time, each testing whether its sum shows a logit above the reference: 1.65 us for a row of 2048
// vectors; like this 1.2), and their sums cross the lanes side by side.

// kLoopRuns runs of a row from vector `base` on: the reference raised to their maximum, the sum so far against it, and each
// run's sum of this lane's terms
template <int DT, class Sum>
__device__ __forceinline__ void l_group(uint32_t image, int base, int u1, int lane, float kf, float& M, Sum& s, float (&vs)[kLoopRuns]) {
    using R = Raw<DT>;
    constexpr int EPV = R::EPV;
    uint4 raw[kLoopRuns];
#pragma unroll
    for (int j = 0; j < kLoopRuns; ++j) raw[j] = l_cell(image, base + 32 * j + lane, u1, R::kNegInf);
    uint4 top = raw[0];
#pragma unroll
    for (int j = 1; j < kLoopRuns; ++j) top = vec_max<DT>(top, raw[j]);
    float v[EPV];
    R::unpack(top, v);
    const float y = fmaxf(M, rintf(warp_max(vec_max<EPV>(v)) * kf));
    s = ref_sum(s, M, y);
    M = y;
#pragma unroll
    for (int j = 0; j < kLoopRuns; ++j) {
        R::unpack(raw[j], v);
        vs[j] = f_exp_sum<EPV>(v, kf, -M);
    }
}

// s_sweep_row on the row's image.  (Sub-segments of the last target row, from which a token of the output is drawn, hold doubles
// (SHORT) whatever the row's length: a lane's vectors are added in double as well, where there are several to a sub-segment, from 4096
// vectors a row on.  In fp32 the sum of a flat row of 6656 vectors was off by 4.5e-10 on average, like this by 3.0e-10, as in the verification kernels.)
template <int DT, bool SHORT>
__device__ __forceinline__ void l_sweep_draft(uint32_t image, int units, float kf, int warp, int lane, SubSegment<SHORT>* seg) {
    using Sum = std::conditional_t<SHORT, double, float>;
    float M = kNoRef;
    Sum s = 0;
    int u0, u1, runs;
    s_part(units, warp, u0, u1, runs);
    int sub = 0, left = runs;
    for (int base = u0; base < u1; base += 32 * kLoopRuns) {
        float vs[kLoopRuns];
        l_group<DT>(image, base, u1, lane, kf, M, s, vs);
        const int n = min((u1 - base + 31) / 32, kLoopRuns);
        if (runs == 1) {                          // (a sub-segment a run; a group of fewer has empty ones behind it)
            if (SHORT) {
                double z[kLoopRuns];
#pragma unroll
                for (int j = 0; j < kLoopRuns; ++j) z[j] = static_cast<double>(vs[j]);
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
                    for (int j = 0; j < kLoopRuns; ++j) z[j] += shfl_xor_d(z[j], off);
                }
#pragma unroll
                for (int j = 0; j < kLoopRuns; ++j)
                    if (j < n && (lane & 15) == 0)
                        reinterpret_cast<float2*>(seg + s_place(warp, sub + j))[lane >> 4] =
                            lane == 0 ? make_float2(__int_as_float(__double2loint(z[j])), __int_as_float(__double2hiint(z[j]))) : make_float2(M, 0.f);
            } else {
#pragma unroll
                for (int off = 8; off > 0; off >>= 1) {
#pragma unroll
                    for (int j = 0; j < kLoopRuns; ++j) vs[j] += __shfl_xor_sync(0xffffffffu, vs[j], off);
                }
#pragma unroll
                for (int j = 0; j < kLoopRuns; ++j)
                    if (j < n && (lane & 15) == 0) reinterpret_cast<float2*>(seg + s_place(warp, sub + j))[lane >> 4] = make_float2(vs[j], M);
            }
            sub += n;
        } else {
#pragma unroll
            for (int j = 0; j < kLoopRuns; ++j) {
                if (j >= n) break;
                s += static_cast<Sum>(vs[j]);
                if (--left == 0) {
                    s_put<SHORT>(M, s, lane, seg + s_place(warp, sub));
                    ++sub;
                    left = runs;
                    s = 0;
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
// a warp's share {reference, sum} of a target row: fp32 over a lane's vectors (13 at most), joined in double
template <int DT>
__device__ __forceinline__ void l_sweep_target(uint32_t image, int units, float kf, int warp, int lane, LoopShared& sh) {
    float M = kNoRef, s = 0.f;
    int u0, u1, runs;
    s_part(units, warp, u0, u1, runs);
    for (int base = u0; base < u1; base += 32 * kLoopRuns) {
        float vs[kLoopRuns];
        l_group<DT>(image, base, u1, lane, kf, M, s, vs);
        s += (vs[0] + vs[1]) + (vs[2] + vs[3]);
    }
    const double z = warp_sum_d(static_cast<double>(s));
    if (lane == 0) { sh.wM[warp] = static_cast<double>(M); sh.wZ[warp] = z; }
}
// residual sums of a position's sub-segments
template <int DT>
__device__ __forceinline__ void l_sweep_pair(uint32_t imageP, uint32_t imageQ, int units, float kf, float cp, float nMP, float nMQ,
                                             int warp, int lane, double* res) {
    using R = Raw<DT>;
    constexpr int EPV = R::EPV;
    int u0, u1, runs;
    s_part(units, warp, u0, u1, runs);
    double acc = 0.0;
    int sub = 0, left = runs;
    for (int base = u0; base < u1; base += 32 * kLoopRuns) {
        double z[kLoopRuns];
#pragma unroll
        for (int j = 0; j < kLoopRuns; ++j) {
            float vp[EPV], vq[EPV], t[EPV];
            R::unpack(l_cell(imageP, base + 32 * j + lane, u1, R::kNegInf), vp);
            R::unpack(l_cell(imageQ, base + 32 * j + lane, u1, R::kNegInf), vq);
            z[j] = static_cast<double>(f_pair_sum<EPV, true>(vp, vq, kf, cp, nMP, nMQ, t));
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
            for (int j = 0; j < kLoopRuns; ++j) z[j] += shfl_xor_d(z[j], off);
        }
#pragma unroll
        for (int j = 0; j < kLoopRuns; ++j) {
            if (base + 32 * j >= u1) break;
            acc += z[j];
            if (--left == 0 || base + 32 * (j + 1) >= u1) {
                if (lane == 0) res[warp * kSSub + sub] = acc;
                ++sub;
                left = runs;
                acc = 0.0;
            }
        }
    }
    if (lane >= sub && lane < kSSub) res[warp * kSSub + lane] = 0.0;
}
// f_rescan on the rows' images (one warp): the first element of sub-segment `sel` at which the running mass exceeds tw
template <int DT, bool HAVEQ>
__device__ __forceinline__ int l_rescan(uint32_t imageP, uint32_t imageQ, int units, int sel, int lane, float kf, float cp, float nMP,
                                        float nMQ, double tw) {
    using R = Raw<DT>;
    constexpr int EPV = R::EPV;
    int w0, w1;
    s_range(units, sel / kSSub, sel % kSSub, w0, w1);
    double run = 0.0;
    int found = -1, last_pos = -1;
    for (int base = w0; base < w1 && found < 0; base += 32) {
        const int i = base + lane;
        float vp[EPV], vq[EPV], t[EPV];
        R::unpack(l_cell(imageP, i, w1, R::kNegInf), vp);
        if (HAVEQ) R::unpack(l_cell(imageQ, i, w1, R::kNegInf), vq);
        f_pair_sum<EPV, HAVEQ>(vp, vq, kf, cp, nMP, nMQ, t);
        // (a lane's own prefix sums beside the sums over the lanes, so that the lane that is found has only to compare)
        double own[EPV];
#pragma unroll
        for (int e = 0; e < EPV; ++e) {
            own[e] = (e > 0 ? own[e > 0 ? e - 1 : 0] : 0.0) + static_cast<double>(t[e]);
            if (t[e] > 0.f) last_pos = i * EPV + e;
        }
        const double ls = own[EPV - 1];
        double inc = ls;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const double o = shfl_up_d(inc, off);
            if (lane >= off) inc += o;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, run + inc > tw && ls > 0.0);
        if (bal) {
            const double before = run + inc - ls;
            int f = -1, lp = -1;
#pragma unroll
            for (int e = EPV - 1; e >= 0; --e) {
                if (t[e] > 0.f && lp < 0) lp = i * EPV + e;
                if (t[e] > 0.f && before + own[e] > tw) f = i * EPV + e;
            }
            if (f < 0) f = lp;
            found = __shfl_sync(0xffffffffu, f, __ffs(bal) - 1);
        }
        run += shfl_d(inc, 31);
    }
    if (found < 0) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) last_pos = max(last_pos, __shfl_xor_sync(0xffffffffu, last_pos, off));
        found = last_pos;
    }
    return found;
}
// the token at which a row's own law reaches the uniform (one warp): the draft row of a step, the last target row
template <int DT, bool SHORT>
__device__ __forceinline__ int l_draw(uint32_t image, int units, float kf, const SubSegment<SHORT>* seg, float u, int lane, double* norm) {
    double rem = 0.0;
    const int sel = s_locate<SHORT>(seg, u, lane, -1, norm, rem);
    return sel < 0 ? -1 : l_rescan<DT, false>(image, 0u, units, sel, lane, kf, 1.f, -static_cast<float>(norm[0]), 0.f, rem);
}

// The scalar part of a block's verification (the sampling warp; lanes c and c + 32 speak for rows / positions c and c + 32):
// the recursion or the tests, which positions can be the selected one (reading as in f_fold_block), faults.
__device__ __forceinline__ int l_decide(const LoopArgs& a, LoopShared& sh, int lane) {
    const int g = a.gamma;
    double rat[2] = {1.0, 1.0}, zr[2] = {1.0, 1.0};
    bool badrow[2] = {false, false};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c >= g) continue;
        const double MP = sh.MP[c], ZP = sh.ZP[c], MQ = sh.MQ[c], ZQ = sh.ZQ[c], zp = sh.zp[c], zq = sh.zq[c];
        const double none = static_cast<double>(kNoRef), inf = static_cast<double>(INFINITY);
        badrow[h] = !(MP > none && MP < inf) || !row_sum_ok(ZP) || !(MQ > none && MQ < inf) || !row_sum_ok(ZQ) || sh.tok[c] < 0 || zq == -inf;
        zr[h] = ZQ / ZP;
        rat[h] = badrow[h] ? 0.0 : exp2((zp - zq) * a.kd - (MP - MQ)) * zr[h];
    }
    const unsigned bad_lo = __ballot_sync(0xffffffffu, badrow[0]), bad_hi = __ballot_sync(0xffffffffu, badrow[1]);
    double mine[2] = {1.0, 1.0};
    unsigned lo = 0, hi = 0;
    int last = 0, bad = 0;
    if (a.token) {
        bool pass[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = lane + 32 * h;
            const double hw = fmin(rat[h], 1.0);
            pass[h] = c >= g || (hw > 0.0 && static_cast<double>(sh.u[c < g ? c : 0]) <= hw);
        }
        const unsigned f_lo = __ballot_sync(0xffffffffu, !pass[0]), f_hi = __ballot_sync(0xffffffffu, !pass[1]);
        const int tau = f_lo ? __ffs(f_lo) - 1 : (f_hi ? 32 + __ffs(f_hi) - 1 : g);
        const int last_pair = tau < g ? tau : g - 1;         // (a fault counts if its row is among rows 0 .. min(tau, gamma - 1))
        const unsigned long long badrows = static_cast<unsigned long long>(bad_lo) | (static_cast<unsigned long long>(bad_hi) << 32);
        bad = (badrows & (last_pair >= 63 ? ~0ull : ((2ull << last_pair) - 1ull))) != 0ull;
        if (tau == g) last = 1;
        else if (tau < 32) lo = 1u << tau;
        else hi = 1u << (tau - 32);
    } else {
        double pc = 1.0;
        for (int c = 0; c < g; ++c) {
            if (c == lane) mine[0] = pc;
            if (c == lane + 32) mine[1] = pc;
            pc = fmin(pc * shfl_d(c < 32 ? rat[0] : rat[1], c & 31), 1.0);
        }
        // h_c <= p_c: a position whose uniform lies above p_c cannot be the selected one
        bool need[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = lane + 32 * h;
            need[h] = c < g && (c == 0 || static_cast<double>(sh.u[c < g ? c - 1 : 0]) <= mine[h] * (1.0 + 1e-6));
        }
        lo = __ballot_sync(0xffffffffu, need[0]);
        hi = __ballot_sync(0xffffffffu, need[1]);
        last = pc > 0.0 && static_cast<double>(sh.u[g - 1]) <= pc;           // position gamma passes: no other is wanted
        bad = (bad_lo | bad_hi) != 0u;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c < g) {
            sh.p[c] = mine[h];
            sh.csc[c] = static_cast<float>(mine[h] * zr[h]);
        }
    }
    if (lane == 0) { sh.lo = lo; sh.hi = hi; sh.last = last; sh.over = bad; }
    return bad;
}

template <int DT, bool SHORT>
__global__ void __launch_bounds__(kSAllThreads, 2) decode_loop_kernel(const __grid_constant__ LoopArgs a) {
    using R = Raw<DT>;
    constexpr int EPV = R::EPV;
    constexpr size_t ESZ = (DT == kF32) ? 4 : 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = a.gamma, B = a.B, V = a.V, units = V / EPV;
    const size_t row_bytes = static_cast<size_t>(V) * ESZ;
    const float kf = a.kf;
    __shared__ SubSegment<SHORT> seg[kSSegs];     // the draft row's
    __shared__ SubSegment<true> segL[kSSegs];     // the last target row's: a token of the output is drawn from it
    __shared__ LoopShared sh;
    extern __shared__ __align__(16) unsigned char dyn[];
    const uint32_t imageQ = smem_u32(dyn), imageP = imageQ + static_cast<uint32_t>(row_bytes);
    const char* const tgt = static_cast<const char*>(a.tgt);
    const char* const drf = static_cast<const char*>(a.drf);
    const int b = blockIdx.x;
    const bool sampling = warp == kSWarps;
    auto logit = [&](const char* row, int x) { return static_cast<float>(load_logit<DT>(row, x)); };

    int last = a.first[b];
    long long pos = 0;
    for (int n = 0; n < a.iterations; ++n) {
        const int start = last;
        const size_t nb = static_cast<size_t>(n) * B + b;
        // ---------------- the block is drafted ----------------
        for (int i = 0; i < g; ++i) {
            const bool ok = last >= 0 && last < V;
            const size_t at = static_cast<size_t>(ok ? last : 0) * row_bytes;
            float u = 0.f;
            if (!sampling) {
                if (ok) {
                    l_fetch(imageQ, drf + at, units, warp, lane);
                    l_fetch(imageP, tgt + at, units, warp, lane);
                    cp_async_wait<1>();
                    l_sweep_draft<DT, SHORT>(imageQ, units, kf, warp, lane, seg);
                }
            } else {
                u = a.u_draft[(static_cast<size_t>(n) * g + i) * B + b];
                if (i == 0) for (int c = lane; c < g + 2; c += 32) sh.u[c] = a.u_verify[nb * (g + 2) + c];
            }
            __syncthreads();
            int found = -1;
            double norm[2] = {0.0, 0.0};
            if (sampling) {
                if (ok) found = l_draw<DT, SHORT>(imageQ, units, kf, seg, u, lane, norm);
                if (lane == 0) sh.next = found;
            } else if (ok) {
                cp_async_wait<0>();
                l_sweep_target<DT>(imageP, units, kf, warp, lane, sh);
            }
            __syncthreads();
            last = sh.next;               // (written again after the next step's first barrier)
            if (sampling) {
                // behind the streaming warps' next loads: what the verification wants to know of this row
                const float m = lane < kSWarps && ok ? static_cast<float>(sh.wM[lane]) : kNoRef, mr = warp_max(m);
                const double z = warp_sum_d(lane < kSWarps && ok ? ref_sum(sh.wZ[lane], m, mr) : 0.0);
                float zl = 0.f;           // the drafted token's logits
                if (found >= 0 && lane < 2) zl = logit((lane == 0 ? tgt : drf) + at, found);
                const float zq = __shfl_sync(0xffffffffu, zl, 1);
                if (lane == 0) {
                    double MQ = norm[0], ZQ = norm[1];
                    if (found < 0) { MQ = kNoRef; ZQ = 0.0; }
                    else if (a.lse) {
                        // as supplied normalisers are taken: rounded to 32 bits, an integer reference and a sum in [2^-1/2, 2^1/2]
                        const double L2 = static_cast<double>(s_lse(found, norm)) * 1.4426950408889634073599246810019;
                        MQ = rint(L2);
                        ZQ = exp2(L2 - MQ);
                    }
                    sh.MP[i] = mr; sh.ZP[i] = z; sh.MQ[i] = MQ; sh.ZQ[i] = ZQ;
                    sh.zp[i] = zl; sh.zq[i] = zq; sh.tok[i] = found;
                    a.drafted[nb * g + i] = found;
                }
            }
        }
        // ---------------- and verified: the last target row while the scalar part is done ----------------
        const bool have_last = last >= 0 && last < V;
        int bad = 0;
        if (!sampling) {
            if (have_last) {
                l_fetch(imageP, tgt + static_cast<size_t>(last) * row_bytes, units, warp, lane);
                cp_async_wait<0>();
                l_sweep_draft<DT, true>(imageP, units, kf, warp, lane, segL);
            }
        } else {
            __syncwarp();
            bad = l_decide(a, sh, lane);
        }
        __syncthreads();
        int tau = -1, found = -1;
        if (sampling && !bad && have_last) {
            // (a fault in the last target row is the sequence's if it is the row to sample from, or if it counts in any case)
            double norm[2], rem = 0.0;
            const int sel = s_locate<true>(segL, sh.u[g + 1], lane, -1, norm, rem);
            if (sh.last) { tau = g; if (sel >= 0) found = l_rescan<DT, false>(imageP, 0u, units, sel, lane, kf, 1.f, -static_cast<float>(norm[0]), 0.f, rem); }
            else if (sel < 0 && a.last_counts) bad = 1;
        }
        unsigned lo = sh.lo, hi = sh.hi;
        bool over = sh.last != 0 || sh.over != 0;
        while (!over && (lo | hi) != 0u) {
            int c;                        // the highest candidate
            if (hi) { c = 63 - __clz(hi); hi &= ~(1u << (c - 32)); } else { c = 31 - __clz(lo); lo &= ~(1u << c); }
            if (!sampling) {
                const size_t at = static_cast<size_t>(c == 0 ? start : sh.tok[c - 1]) * row_bytes;
                l_fetch(imageP, tgt + at, units, warp, lane);
                l_fetch(imageQ, drf + at, units, warp, lane);
                cp_async_wait<0>();
                l_sweep_pair<DT>(imageP, imageQ, units, kf, sh.csc[c], -static_cast<float>(sh.MP[c]), -static_cast<float>(sh.MQ[c]), warp, lane, sh.res);
            }
            __syncthreads();
            if (sampling) {
                double w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = sh.res[4 * lane + j];
                double inc = ((w[0] + w[1]) + w[2]) + w[3];
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const double o = shfl_up_d(inc, off);
                    if (lane >= off) inc += o;
                }
                const double total = shfl_d(inc, 31);
                const double hw = a.token || c == 0 ? 1.0 : f_weight(sh.p[c], total / sh.ZQ[c]);
                if (bad) tau = 0;
                else if (a.token || c == 0 || (hw > 0.0 && static_cast<double>(sh.u[c - 1]) <= hw)) {
                    tau = c;
                    if (total > 0.0 && total < static_cast<double>(INFINITY)) {
                        double rem;
                        const int sel = s_pick(w, inc, static_cast<double>(sh.u[g]) * total, lane, rem);
                        found = l_rescan<DT, true>(imageP, imageQ, units, sel, lane, kf, sh.csc[c], -static_cast<float>(sh.MP[c]), -static_cast<float>(sh.MQ[c]), rem);
                    }
                }
                if (lane == 0) sh.over = tau >= 0;
            }
            __syncthreads();
            over = sh.over != 0;
        }
        // ---------------- the sequence is extended ----------------
        if (sampling) {
            if (found < 0) bad = 1;       // (a fault of a row, or an empty residual where the algorithm must sample)
            const int m = bad ? 1 : tau + 1;
            int32_t* out = a.seq + static_cast<size_t>(b) * a.width + pos;
            for (int i = lane; i < m; i += 32) out[i] = bad ? -1 : (i < tau ? sh.tok[i] : found);
            if (lane == 0) {
                a.tau[nb] = bad ? -2 : tau;
                if (bad) atomicExch(a.fault, 1);
                sh.next = bad ? -1 : found;
            }
            pos += m;
        }
        __syncthreads();
        last = sh.next;
    }
    if (sampling) {
        for (long long i = pos + lane; i < a.width; i += 32) a.seq[static_cast<size_t>(b) * a.width + i] = -1;
        if (lane == 0) a.lengths[b] = pos;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
constexpr size_t kLoopSmem = 212992;              // shared memory for the two rows of a step

bool loop_fits(int V, int dtype) { return 2 * static_cast<size_t>(V) * (dtype == kF32 ? 4 : 2) <= kLoopSmem; }

// Where one kernel is the faster loop.  A CTA here sweeps its sequence's rows alone and its candidates one after the other; the two
// launches of an iteration share the batch's candidates over all SMs, but wait for the whole batch twice.  So it is a matter of the
// sequences to an SM (at work at once: 2 with rows of up to 53200 bytes, else 1), of the steps that a sweep takes (kLoopRuns runs of
// 16 warps: 2048 vectors each) and of gamma, with which the candidates grow.  Per length of a row, and for up to 8 sequences, 24, one to an
// SM, 2, 3, 4 and more: the largest gamma at which this kernel was measured faster (Algorithm 2).  Measured over 8400 calls of 40
// lengths from 1024 to 53248, drafts of noise 0.1 to 3, against the faster of the two launches as they are and as they were when this
// kernel came; time over theirs, bf16, noise 0.2 / 0.4 / 0.7:
//   V = 16384 gamma = 8: B = 1 0.74 / 0.70 / 0.81, 148 0.57 / 0.55 / 0.53, 296 0.70 / 0.66 / 0.66, 768 0.77 / 0.78 / 0.80
//   V = 2048 gamma = 8: B = 148 0.67, 297 0.81 / 0.89 / 0.91, 450 1.02 / 1.05 / 1.06, 768 1.15;  gamma = 3: 768 0.89 / 0.94 / 0.96
//   V = 24576 gamma = 8: B = 4 1.03 / 1.12 / 1.00, 148 0.82 / 0.74 / 0.69, 768 0.98 / 1.01 / 1.02;  gamma = 16: B = 4 1.12 / 1.24 / 1.15, 148 0.97 / 0.89 / 0.87
//   V = 32768 (one CTA to an SM) gamma = 3: B = 149 0.67, 297 0.74, 768 1.00 / 1.02 / 1.06;  gamma = 12: B = 64 0.89 / 0.94 / 0.81, 149 1.09 / 1.10 / 1.13
//   V = 51200 gamma = 5, noise 1: B = 1 1.22, 32 0.95, 128 0.86, 150 1.18, 768 1.39;  gamma = 1, noise 0.2 / 0.7: B = 1 0.58 / 0.59, 444 0.80 / 0.88, 768 1.04 / 1.11
// Within the lines 2 of 4400 calls were 3 % or more slower than the loop that this kernel replaced (3 and 6 %).  Algorithm 1, which has
// one candidate, gains up to half as much gamma again (V = 17000: gamma = 6 / 10, B = 4 0.83 / 1.01, B = 149 0.84 / 1.01), and up to
// twice where every sequence has an SM (V = 36864, B = 148: gamma = 16 0.84).
// Up to 8 sequences of rows of up to 1024 stay one launch at any gamma, as the calls that launches count most for; on the device that
// is no gain from gamma = 24 on in 16 bits: V = 1024, B = 3, 3 iterations, noise 0.2 / 0.7 / 1.5: gamma = 16 0.98 / 0.97 / 0.94, 24 1.31 / 1.08 / 0.98,
// 64 1.25 / 1.13 / 1.12; in 32 bits 16 0.90 / 0.83 / 0.80, 24 1.04 / 0.90 / 0.86, 64 1.13 / 0.99 / 0.98.
bool loop_pays(int V, int dtype, int B, int gamma, bool token, int sms) {
    struct Line { int V; unsigned char gamma[7]; };
    static constexpr Line kBf16[] = {{1024, {64, 16, 16, 8, 8, 4, 3}},      {3072, {12, 16, 16, 8, 8, 4, 3}},  {6144, {12, 32, 32, 12, 8, 8, 5}},
                                     {10240, {16, 32, 32, 16, 16, 16, 12}}, {16384, {16, 32, 32, 32, 32, 32, 32}},
                                     {20000, {5, 6, 16, 8, 6, 4, 3}},       {26600, {5, 6, 16, 8, 8, 6, 5}},   {32768, {5, 16, 32, 5, 4, 2, 1}},
                                     {34816, {2, 3, 6, 2, 2, 1, 1}},        {49152, {2, 3, 8, 3, 2, 1, 1}},    {53248, {2, 3, 5, 2, 1, 1, 0}},
                                     {INT_MAX, {}}};
    static constexpr Line kF32s[] = {{1024, {64, 32, 32, 24, 16, 12, 8}},   {1536, {16, 32, 32, 24, 16, 12, 8}},   {3072, {32, 32, 32, 32, 16, 16, 12}}, {6144, {32, 32, 32, 32, 16, 16, 16}},
                                     {8192, {64, 64, 64, 64, 64, 64, 64}},  {13300, {8, 16, 32, 32, 32, 32, 32}}, {16384, {8, 16, 24, 10, 8, 6, 3}},
                                     {24576, {5, 6, 16, 5, 5, 3, 2}},       {26624, {2, 2, 8, 3, 3, 2, 1}},       {INT_MAX, {}}};
    const int load = B <= 8 ? 0 : B <= 24 ? 1 : B > 4 * sms ? 6 : 2 + (B - 1) / sms;
    const Line* line = dtype == kF32 ? kF32s : kBf16;
    while (V > line->V) ++line;
    const int most = line->gamma[load];
    return gamma <= (token ? most * (load == 2 ? 4 : 3) / 2 : most);
}

cudaError_t launch_loop(const LoopArgs& args, int dtype, cudaStream_t stream) {
    const size_t row_bytes = static_cast<size_t>(args.V) * (dtype == kF32 ? 4 : 2);
    const bool brief = s_short(row_bytes);
    const auto kernel = dtype == kF32 ? (brief ? decode_loop_kernel<kF32, true> : decode_loop_kernel<kF32, false>)
                                      : (brief ? decode_loop_kernel<kBF16, true> : decode_loop_kernel<kBF16, false>);
    const size_t smem = 2 * row_bytes;
    const cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kLoopSmem));
    if (e != cudaSuccess) return e;
    kernel<<<args.B, kSAllThreads, smem, stream>>>(args);
    return cudaGetLastError();
}

}  // namespace bv
