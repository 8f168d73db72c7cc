// Verification in phases (Algorithm 2, also with supplied draft normalisers, Algorithms 4 and 1, logits or
// probabilities) for batches between the latency regime of the small-batch kernel and the sizes at which the
// flow kernel's overlap of the two sweeps pays, and for rows at any alignment.
//
// One persistent CTA per SM (a cooperative launch).  Every streaming warp is on its own:
//   1. the first sweep of all rows 0 .. gamma-1 is one list of units (64 vectors of a row), of which each warp
//      takes an equal contiguous part; it leaves {reference, sum 2^{z k - M}} of its piece of every row.
//      The warp whose part completes a sequence folds it: normalisers, the recursion of Eq. "def_as" or
//      the tests of Algorithm 1, and which positions can be the selected one.
//   2. when every sequence is folded, all CTAs read the same table of candidate positions and cut the list of
//      their second sweeps the same way; the warp whose part completes a sequence forms S_i and h_i
//      (Eq. "pacc_block") from the top down and, if a position passes, draws the token and ends the
//      sequence.  Sequences none of whose listed candidates passed go into another round.
// There are no queues and no hand-overs inside a CTA: an item costs nothing but its bytes.  The price is that
// the GPU idles while the last sequences are folded, which is why the largest batches stay with the flow kernel.
#include "bv_flow_common.cuh"

namespace bv {

constexpr int kPhWarps = 23;                   // streaming warps; one more fetches scalars and walks ahead through the code of
constexpr int kPhThreads = 32 * (kPhWarps + 1);   // the folds and the ends of sequences, which the others then find in the caches
constexpr int kPhSlots = 5;                    // ring steps a warp's loads run ahead of its arithmetic
constexpr uint32_t kPhSlotBytes = 512 + 512 + 16;   // two cells a lane, and the vector after the second 32 (unaligned pairs)
constexpr int kPhQueue = 8;                    // runs opened by the issue side and not yet consumed (at most kPhSlots + 2)
constexpr int kPhUnit = 64;                    // vectors of a row in one unit of work: one ring step of a row, two of a row pair
static_assert(kPhaseMaxB <= kPhThreads, "a thread looks at one sequence");

// One run, consecutive units of one row (pair) in a warp's part, as the issue side hands it to the consuming side.
struct alignas(16) PhRun {
    float4 pos;        // second sweep of a pair: p_c Z_Q / Z_P and minus the references
    int b, c;          // sequence; first sweep: row of the sequence's list, second: position (gamma: the last target row)
    int k, n;          // its units
    int v0, v1;        // its vectors
    int hP, shift;     // unaligned rows: elements of the first vector that belong to the row before; shift of the draft row
};
struct PhShared {
    PhRun q[kPhWarps][kPhQueue];
    int scan[kPhWarps + 1];
    int fail;
    unsigned word;
};

__device__ __forceinline__ int warp_sum_i(int x) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
}
__device__ __forceinline__ bool ph_wait(unsigned* word, unsigned mask, unsigned target, int* status, unsigned limit) {
    for (unsigned spins = 0; (ld_volatile(word) & mask) < target; ++spins) {
        if (spins > limit) { if (status) atomicExch(status, 1); return false; }
        __nanosleep(20);
    }
    return true;
}
// One lane reports n units of a counter's total as in: whatever the warp has written before is visible to the warp whose
// report completes the total, and to that one only it returns true.
__device__ __forceinline__ bool ph_arrive(unsigned* counter, unsigned n, unsigned total) {
    __threadfence();
    const bool last = atomicAdd(counter, n) + n == total;
    if (last) __threadfence();
    return last;
}

// The highest of the positions in the masks (position gamma, if `last`, before all of them); it is taken out.
__device__ __forceinline__ int ph_pop(unsigned& lo, unsigned& hi, int& last, int g) {
    if (last) { last = 0; return g; }
    if (hi) { const int i = 31 - __clz(hi); hi &= ~(1u << i); return 32 + i; }
    const int i = 31 - __clz(lo);
    lo &= ~(1u << i);
    return i;
}

// The uniforms that lanes c and c + 32 test their row or position with, and position gamma's.
__device__ __forceinline__ void ph_uniforms(const Params& prm, int b, int lane, float (&eta)[2], float& eta_g) {
    const int g = prm.gamma;
    const float* u = prm.uni + static_cast<size_t>(b) * (g + 2);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h, i = prm.algo == kTokenVerify ? c : c - 1;
        eta[h] = c < g && i >= 0 ? u[i] : 0.f;
    }
    eta_g = u[g - 1];
}

// One sequence folded by one warp.  Lanes c and c + 32 speak for rows / positions c and c + 32: reference and
// sum of the target and the draft row, whether the row holds a fault, and the ratio of its drafted token.
// (dry: walk the code, write nothing)
static __device__ __forceinline__ void ph_decide(const Params& prm, const PhaseScratch& ps, int b, int lane, const float (&MP)[2], const double (&ZP)[2],
                                                 const float (&MQ)[2], const double (&ZQ)[2], const double (&rat)[2], const bool (&badrow)[2],
                                                 const float (&eta)[2], float eta_g, bool dry) {
    const int g = prm.gamma;
    const bool all = f_all_positions(prm) && !dry;
    const size_t row0 = static_cast<size_t>(b) * (g + 1);
    const unsigned long long badrows = static_cast<unsigned long long>(__ballot_sync(0xffffffffu, badrow[0])) |
                                       (static_cast<unsigned long long>(__ballot_sync(0xffffffffu, badrow[1])) << 32);
    const double ln2 = 0.693147180559945309417232;
    const float nanf_ = __int_as_float(0x7fc00000);
    unsigned long long A = 0, rest = 0;
    int last = 0, bad = 0;
    double mine[2] = {1.0, 1.0}, p_g = 1.0;
    if (prm.algo == kTokenVerify) {
        // test c + 1 on row c; tau = the tests passed before the first failure
        bool pass[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = lane + 32 * h;
            const double hw = fmin(rat[h], 1.0);
            pass[h] = c >= g || (hw > 0.0 && static_cast<double>(eta[h]) <= hw);
        }
        const unsigned f_lo = __ballot_sync(0xffffffffu, !pass[0]), f_hi = __ballot_sync(0xffffffffu, !pass[1]);
        const int tau = f_lo ? __ffs(f_lo) - 1 : (f_hi ? 32 + __ffs(f_hi) - 1 : g);
        const int last_pair = tau < g ? tau : g - 1;         // (a fault counts if its row is among rows 0 .. min(tau, gamma - 1))
        bad = (badrows & (last_pair >= 63 ? ~0ull : ((2ull << last_pair) - 1ull))) != 0ull;
        if (tau == g) last = 1; else A = 1ull << tau;
        if (all) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = lane + 32 * h;
                if (c < g) {
                    if (prm.out_h) prm.out_h[row0 + c + 1] = c <= tau ? static_cast<float>(fmin(rat[h], 1.0)) : nanf_;
                    if (prm.out_S && c != tau) prm.out_S[static_cast<size_t>(b) * g + c] = nanf_;
                    if (prm.out_lse_t) prm.out_lse_t[row0 + c] = c <= tau ? static_cast<float>((static_cast<double>(MP[h]) + log2(ZP[h])) * ln2) : nanf_;
                    if (prm.out_lse_d) prm.out_lse_d[static_cast<size_t>(b) * g + c] = c <= last_pair ? static_cast<float>((static_cast<double>(MQ[h]) + log2(ZQ[h])) * ln2) : nanf_;
                    if (prm.out_p) prm.out_p[row0 + c] = nanf_;
                }
            }
            if (lane == 0 && prm.out_p) prm.out_p[row0 + g] = nanf_;
            if (lane == 0 && prm.out_h) prm.out_h[row0] = 1.f;
            if (lane == 0 && prm.out_lse_t && !last) prm.out_lse_t[row0 + g] = nanf_;
        }
    } else {
        double pc = 1.0;
        for (int c = 0; c < g; ++c) {
            if (c == lane) mine[0] = pc;
            if (c == lane + 32) mine[1] = pc;
            const double next = pc * shfl_d(c < 32 ? rat[0] : rat[1], c & 31);
            pc = prm.greedy ? next : fmin(next, 1.0);
        }
        p_g = pc;
        bad = badrows != 0ull;
        // h_c <= p_c: a position whose uniform lies above p_c cannot be the selected one (f_fold_block)
        bool need[2] = {false, false}, one[2] = {false, false};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = lane + 32 * h;
            if (c < g) {
                need[h] = all || c == 0 || static_cast<double>(eta[h]) <= mine[h] * (1.0 + 1e-6);
                one[h] = need[h] && mine[h] >= 1.0;
                if (all && prm.out_p) prm.out_p[row0 + c] = static_cast<float>(mine[h]);
                if (all && prm.out_lse_t) prm.out_lse_t[row0 + c] = static_cast<float>((static_cast<double>(MP[h]) + log2(ZP[h])) * ln2);
                if (all && prm.out_lse_d) prm.out_lse_d[static_cast<size_t>(b) * g + c] = static_cast<float>((static_cast<double>(MQ[h]) + log2(ZQ[h])) * ln2);
            }
        }
        if (lane == 0 && all && prm.out_p) prm.out_p[row0 + g] = static_cast<float>(p_g);
        last = all || static_cast<double>(eta_g) <= p_g * (1.0 + 1e-6);
        A = static_cast<unsigned long long>(__ballot_sync(0xffffffffu, need[0])) | (static_cast<unsigned long long>(__ballot_sync(0xffffffffu, need[1])) << 32);
        const unsigned long long ones = static_cast<unsigned long long>(__ballot_sync(0xffffffffu, one[0])) |
                                        (static_cast<unsigned long long>(__ballot_sync(0xffffffffu, one[1])) << 32);
        if (!all) {
            if (p_g > 0.0 && static_cast<double>(eta_g) <= p_g) A = 0;       // position gamma passes: nothing else is wanted
            else if (ones) {
                // A position with p_c = 1 passes whatever its uniform (h_c = S_c / (S_c + 1 - p_c) >= 1) unless S_c = 0:
                // the candidates below the highest such one are kept for that case only
                const int top = 63 - __clzll(static_cast<long long>(ones));
                rest = A & ((1ull << top) - 1ull);
                A &= ~((1ull << top) - 1ull);
            }
        }
    }
    if (dry) return;
    if (lane == 0) ps.pos[row0 + g].p = p_g;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && g <= 32) break;
        const int c = lane + 32 * h;
        if (c < g) {
            PhPos q;
            q.cp = static_cast<float>(mine[h] * (ZQ[h] / ZP[h]));
            q.nMP = -MP[h]; q.nMQ = -MQ[h]; q.pad = 0.f;
            q.p = mine[h]; q.ZQ = ZQ[h];
            ps.pos[row0 + c] = q;
        }
    }
    if (bad && !all) {                    // a data fault: the sequence ends here
        A = rest = 0; last = 0;
        for (int i = lane; i <= g; i += 32) prm.out_tokens[row0 + i] = -1;
        if (lane == 0) prm.out_len[b] = -1;
    }
    if (lane == 0) {
        ps.sel[b] = make_uint4(static_cast<unsigned>(A), static_cast<unsigned>(A >> 32), static_cast<unsigned>(last), static_cast<unsigned>(bad));
        ps.rest[b] = make_uint2(static_cast<unsigned>(rest), static_cast<unsigned>(rest >> 32));
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) atomicAdd(&ps.ctr[kPhFolded], 1u);
}

// References and sums of a sequence's first-sweep rows from their pieces: target and draft row c to lane c & 31, half c >> 5.
static __device__ __forceinline__ void ph_reduce_rows(const PhaseScratch& ps, int g, int b, int lane, float (&MP)[2], double (&ZP)[2],
                                                      float (&MQ)[2], double (&ZQ)[2]) {
    const int slots = ps.slots, rows = ps.rows;
    if (slots <= 32) {
        // a lane per row: no step waits for another lane, and eight pieces are asked for at a time
        for (int r0 = 0; r0 < rows; r0 += 32) {
            const int r = r0 + lane;
            const unsigned x = static_cast<unsigned>((b * rows + r) * ps.units);
            const int np = r < rows ? static_cast<int>((x + ps.units - 1) / ps.per1 - x / ps.per1) + 1 : 0;
            const double2* part = ps.part + (static_cast<size_t>(b) * rows + r) * slots;
            float m = kNoRef;
            double s = 0.0;
            for (int p0 = 0; p0 < slots; p0 += 8) {
                double2 v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = p0 + j < np ? __ldcg(&part[p0 + j]) : make_double2(kNoRef, 0.0);
                float mm = m;
#pragma unroll
                for (int j = 0; j < 8; ++j) mm = fmaxf(mm, static_cast<float>(v[j].x));
                s *= static_cast<double>(ref_scale(m, mm));
#pragma unroll
                for (int j = 0; j < 8; ++j) s += v[j].y * static_cast<double>(ref_scale(static_cast<float>(v[j].x), mm));
                m = mm;
            }
#pragma unroll
            for (int h = 0; h < 4; ++h) {                     // target rows c and c + 32, draft rows c and c + 32
                if ((h & 1) && g <= 32) continue;
                if (h >= 2 && rows == g) continue;
                const int c = lane + 32 * (h & 1), src = c + (h < 2 ? 0 : g) - r0;
                const bool here = c < g && src >= 0 && src < 32;
                const float mq = __shfl_sync(0xffffffffu, m, here ? src : 0);
                const double zq = shfl_d(s, here ? src : 0);
                if (here) {
                    if (h < 2) { MP[h & 1] = mq; ZP[h & 1] = zq; }
                    else { MQ[h & 1] = mq; ZQ[h & 1] = zq; }
                }
            }
        }
        return;
    }
    // (few long rows, in more pieces than that: all lanes on one row, four rows asked for at a time)
    for (int r0 = 0; r0 < rows; r0 += 4) {
        double2 v[4];
        int np[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = r0 + q;
            const unsigned x = static_cast<unsigned>((b * rows + r) * ps.units);
            np[q] = r < rows ? static_cast<int>((x + ps.units - 1) / ps.per1 - x / ps.per1) + 1 : 0;
            v[q] = lane < np[q] ? __ldcg(&ps.part[(static_cast<size_t>(b) * rows + r) * slots + lane]) : make_double2(kNoRef, 0.0);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = r0 + q;
            if (r >= rows) break;
            float m = static_cast<float>(v[q].x);
            double s = v[q].y;
            for (int p = lane + 32; p < np[q]; p += 32) {
                const double2 w = __ldcg(&ps.part[(static_cast<size_t>(b) * rows + r) * slots + p]);
                const float wm = static_cast<float>(w.x), mm = fmaxf(m, wm);
                s = s * static_cast<double>(ref_scale(m, mm)) + w.y * static_cast<double>(ref_scale(wm, mm));
                m = mm;
            }
            const float mr = warp_max(m);
            s = warp_sum_d(s * static_cast<double>(ref_scale(m, mr)));
            const int c = r < g ? r : r - g;                  // target row c or draft row c
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (c != lane + 32 * h) continue;
                if (r < g) { MP[h] = mr; ZP[h] = s; }
                else { MQ[h] = mr; ZQ[h] = s; }
            }
        }
    }
}

// the logits of a sequence's drafted tokens in both rows (a token outside the vocabulary: as one the draft cannot have drawn)
template <int DT>
__device__ __forceinline__ void ph_fetch_drafted(const Params& prm, const PhaseScratch& ps, int b, int lane) {
    const int g = prm.gamma;
    constexpr size_t ESZ = (DT == kF32) ? 4 : 2;
    const size_t row_bytes = static_cast<size_t>(prm.V) * ESZ;
    for (int c = lane; c < g; c += 32) {
        const int x = prm.tok[static_cast<size_t>(b) * g + c];
        float2 z = make_float2(0.f, -INFINITY);
        if (x >= 0 && x < prm.V) {
            z.x = static_cast<float>(load_logit<DT>(static_cast<const char*>(prm.tgt) + target_row(prm, b, c) * row_bytes, x));
            z.y = static_cast<float>(load_logit<DT>(static_cast<const char*>(prm.drf) + draft_row(prm, b, c) * row_bytes, x));
        }
        __stcg(&ps.drafted[static_cast<size_t>(b) * g + c], z);
    }
}

static __device__ __noinline__ void ph_fold(const Params& prm, const PhaseScratch& ps, int b, int lane, bool dry) {
    const int g = prm.gamma;
    double zp[2] = {0.0, 0.0}, zq[2] = {0.0, 0.0};
    float eta[2], eta_g, lse[2] = {0.f, 0.f};
    ph_uniforms(prm, b, lane, eta, eta_g);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c < g) {
            const float2 z = __ldcg(&ps.drafted[static_cast<size_t>(b) * g + c]);
            zp[h] = z.x; zq[h] = z.y;
            if (prm.lse_d != nullptr) lse[h] = prm.lse_d[static_cast<size_t>(b) * g + c];
        }
    }
    float MP[2] = {0.f, 0.f}, MQ[2] = {0.f, 0.f};
    double ZP[2] = {1.0, 1.0}, ZQ[2] = {1.0, 1.0};
    ph_reduce_rows(ps, g, b, lane, MP, ZP, MQ, ZQ);
    if (prm.lse_d != nullptr) {
        // the supplied normaliser as an integer reference at or above every scaled logit of the row plus a
        // sum in [2^-1/2, 2^1/2]; a value that is not finite leaves the row without a reference
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const double L2 = static_cast<double>(lse[h]) * 1.4426950408889634073599246810019;
            const bool fin = L2 > -1e300 && L2 < 1e300;
            MQ[h] = fin ? static_cast<float>(rint(L2)) : kNoRef;
            ZQ[h] = fin ? exp2(L2 - rint(L2)) : 0.0;
        }
    }
    double rat[2] = {1.0, 1.0};
    bool badrow[2] = {false, false};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && g <= 32) break;
        if (lane + 32 * h < g) {
            // the row's maximum is finite iff its reference is; Z is NaN / inf iff the row holds a NaN / overflowed
            badrow[h] = !(MP[h] > kNoRef && MP[h] < INFINITY) || !row_sum_ok(ZP[h]) ||
                        !(MQ[h] > kNoRef && MQ[h] < INFINITY) || !row_sum_ok(ZQ[h]) || zq[h] == -INFINITY;
            rat[h] = badrow[h] ? 0.0 : exp2((zp[h] - zq[h]) * prm.kd - (static_cast<double>(MP[h]) - static_cast<double>(MQ[h]))) * (ZQ[h] / ZP[h]);
        }
    }
    ph_decide(prm, ps, b, lane, MP, ZP, MQ, ZQ, rat, badrow, eta, eta_g, dry);
}
// given probabilities: the ratios are read off the rows
template <int DT>
static __device__ __noinline__ void ph_fold_probs(const Params& prm, const PhaseScratch& ps, int b, int lane) {
    const int g = prm.gamma;
    constexpr size_t ESZ = (DT == kF32) ? 4 : 2;
    const size_t row_bytes = static_cast<size_t>(prm.V) * ESZ;
    const float M[2] = {0.f, 0.f};
    const double Z[2] = {1.0, 1.0};
    float eta[2], eta_g;
    ph_uniforms(prm, b, lane, eta, eta_g);
    double rat[2] = {1.0, 1.0};
    bool badrow[2] = {false, false};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c < g) {
            const int x = prm.tok[static_cast<size_t>(b) * g + c];
            bool ok = x >= 0 && x < prm.V;
            double P = 0.0, Q = 1.0;
            if (ok) {
                P = load_logit<DT>(static_cast<const char*>(prm.tgt) + (static_cast<size_t>(b) * (g + 1) + c) * row_bytes, x);
                Q = load_logit<DT>(static_cast<const char*>(prm.drf) + (static_cast<size_t>(b) * g + c) * row_bytes, x);
                ok = Q > 0.0 && Q < static_cast<double>(INFINITY) && P >= 0.0 && P < static_cast<double>(INFINITY);
            }
            badrow[h] = !ok;
            rat[h] = ok ? P / Q : 0.0;
        }
    }
    ph_decide(prm, ps, b, lane, M, Z, M, Z, rat, badrow, eta, eta_g, false);
}

// Unit totals of a position as a warp looks at them: lane l speaks for `per` consecutive ones.
template <class At> __device__ __forceinline__ double ph_lane_sum(At at, int per, int lane) {
    double s = 0.0;
    for (int j0 = 0; j0 < per; j0 += 8) {
        double w[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] = j0 + j < per ? at(lane * per + j0 + j) : 0.0;
#pragma unroll
        for (int j = 0; j < 8; ++j) s += w[j];
    }
    return s;
}
__device__ __forceinline__ double ph_prefix(double x, int lane) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double o = shfl_up_d(x, off);
        if (lane >= off) x += o;
    }
    return x;
}
// The unit in which u times the sum falls: the first non-empty one whose inclusive prefix exceeds it, else the last
// non-empty one (-1: none); `rem`: what is left of it at the unit's start.  fp64 in index order, as every sum that decides a token.
template <class At>
__device__ __forceinline__ int ph_locate(At at, int per, int lane, double mine, double u, double& rem) {
    double inc = ph_prefix(mine, lane);
    const double t = u * shfl_d(inc, 31);
    auto pick = [&](double x, double upto, bool& hit) -> int {
        const unsigned h = __ballot_sync(0xffffffffu, x > 0.0 && upto > t), nz = __ballot_sync(0xffffffffu, x > 0.0);
        hit = h != 0u;
        return h ? __ffs(h) - 1 : 31 - __clz(nz);
    };
    bool hit;
    rem = 0.0;
    const int src = pick(mine, inc, hit);
    if (src < 0) return -1;
    double base = src > 0 ? shfl_d(inc, src - 1) : 0.0;
    int sel = -1;
    for (int j0 = 0; j0 < per; j0 += 32) {                    // the units of that lane, 32 at a time
        const double w = j0 + lane < per ? at(src * per + j0 + lane) : 0.0;
        inc = ph_prefix(w, lane);
        const int e = pick(w, base + inc, hit);
        if (e >= 0) { sel = src * per + j0 + e; rem = t - (base + (e > 0 ? shfl_d(inc, e - 1) : 0.0)); }
        if (hit) break;
        base += shfl_d(inc, 31);
    }
    return sel;
}

// All listed second sweeps of sequence b are in (one warp): S_i, h_i from the top down, and if a position passes, its
// token and the end of the sequence; else what is left of its candidates goes into the next round.
// (dry: walk the code on whatever the scratch holds, write nothing)
template <int DT, bool PROBS, bool AL>
static __device__ __noinline__ void ph_finalize(const Params& prm, const PhaseScratch& ps, int b, uint4 sel, int round, int lane, bool dry) {
    const int g = prm.gamma, units = ps.units, per = (units + 31) / 32;
    const bool all = f_all_positions(prm) && !dry, tv = prm.algo == kTokenVerify;
    constexpr size_t ESZ = (DT == kF32) ? 4 : 2;
    constexpr int EPV = Raw<DT>::EPV;
    const size_t row_bytes = static_cast<size_t>(prm.V) * ESZ;
    const size_t row0 = static_cast<size_t>(b) * (g + 1);
    const float* u = prm.uni + static_cast<size_t>(b) * (g + 2);
    const double p_g = __ldcg(&ps.pos[row0 + g].p);
    const float u_res = u[g], u_last = u[g + 1], eta_g = u[g - 1];
    const int X0 = lane < g ? prm.tok[static_cast<size_t>(b) * g + lane] : -1, X1 = lane + 32 < g ? prm.tok[static_cast<size_t>(b) * g + lane + 32] : -1;
    unsigned lo = sel.x, hi = sel.y;
    int last = static_cast<int>(sel.z);
    bool bad = sel.w != 0u;
    int tau = -1, found = -1;
    const double ln2 = 0.693147180559945309417232;
    for (int n = __popc(lo) + __popc(hi) + last; n > 0; --n) {
        const int c = ph_pop(lo, hi, last, g);
        const size_t ri = row0 + c;
        const double* seg = ps.seg + ri * units;
        const float* seg_M = ps.seg_M + static_cast<size_t>(b) * units;
        PhPos q;
        q.cp = 1.f; q.nMP = 0.f; q.nMQ = 0.f; q.p = p_g; q.ZQ = 1.0;
        float eta_c = eta_g, Mr = 0.f;
        bool ok = true;
        if (c < g) {
            const float4 a = __ldcg(reinterpret_cast<const float4*>(&ps.pos[ri]));
            const double2 e = __ldcg(reinterpret_cast<const double2*>(&ps.pos[ri].p));
            q.cp = a.x; q.nMP = a.y; q.nMQ = a.z; q.p = e.x; q.ZQ = e.y;
            eta_c = c >= 1 ? u[c - 1] : 0.f;
        } else if (!PROBS) {
            // the last target row was swept once, against the references its units found
            Mr = kNoRef;
            for (int i = lane; i < units; i += 32) Mr = fmaxf(Mr, __ldcg(&seg_M[i]));
            Mr = warp_max(Mr);
            q.nMP = -Mr;
            ok = Mr > kNoRef && Mr < INFINITY;
        }
        auto at = [&](int i) -> double {
            if (i >= units) return 0.0;
            const double w = __ldcg(&seg[i]);
            return c == g && !PROBS ? w * static_cast<double>(ref_scale(__ldcg(&seg_M[i]), Mr)) : w;
        };
        const double mine = ph_lane_sum(at, per, lane), total = warp_sum_d(mine);
        bool pass;
        if (c == g) {
            if (!ok || !(PROBS ? total < static_cast<double>(INFINITY) : row_sum_ok(total))) bad = true;      // (a fault in a last target row that is read is the sequence's)
            pass = tv || (p_g > 0.0 && static_cast<double>(eta_g) <= p_g);
            if (all && prm.out_h && !tv && lane == 0) prm.out_h[ri] = static_cast<float>(p_g);
            if (all && prm.out_lse_t && lane == 0) prm.out_lse_t[ri] = static_cast<float>((static_cast<double>(Mr) + log2(total)) * ln2);
        } else {
            const double S = total / q.ZQ, hw = c == 0 ? 1.0 : f_weight(q.p, S);
            pass = tv || c == 0 || (hw > 0.0 && static_cast<double>(eta_c) <= hw);
            if (all && lane == 0) {
                if (prm.out_S) prm.out_S[static_cast<size_t>(b) * g + c] = static_cast<float>(S);
                if (prm.out_h && !tv) prm.out_h[ri] = static_cast<float>(hw);
            }
        }
        if (!pass || tau >= 0) continue;
        tau = c;
        double rem = 0.0;
        int unit = -1;
        if ((ok && total > 0.0 && total < static_cast<double>(INFINITY)) || dry) unit = ph_locate(at, per, lane, mine, static_cast<double>(c < g ? u_res : u_last), rem);
        if (dry) unit = 0;
        if (unit >= 0) {
            const char* rowP = static_cast<const char*>(prm.tgt) + target_row(prm, b, c) * row_bytes;
            const char* rowQ = c < g ? static_cast<const char*>(prm.drf) + draft_row(prm, b, c) * row_bytes : nullptr;
            const int w0 = unit * kPhUnit;
            if (AL) {
                found = f_rescan<DT, PROBS, 2>(rowP, rowQ, w0, min(w0 + kPhUnit, prm.V / EPV), lane, prm.kf, q.cp, q.nMP, q.nMQ, rem);
            } else {
                // (the units are cut on the 16-byte vectors that the target row's bytes lie in)
                found = f_rescan_any<DT, PROBS, 2>(rowP, rowQ, prm.V, w0, w0 + kPhUnit, lane, prm.kf, q.cp, q.nMP, q.nMQ, rem);
            }
        }
        if (!all) break;
    }
    if (dry) return;
    uint4 next = make_uint4(0u, 0u, 0u, 0u);
    unsigned add = 1u;
    if (tau < 0 && !bad) {
        // no candidate passed: now the ones below a position with p = 1, whose residual turned out to be empty (position
        // 0 is among them, so there is no third time)
        const uint2 r = __ldcg(&ps.rest[b]);
        next = make_uint4(r.x, r.y, 0u, 0u);
        add = 0x10001u;
    } else {
        bad = bad || found < 0;           // (an empty residual where the algorithm must sample: a domain error)
        int32_t* ot = prm.out_tokens + row0;
        for (int i = lane; i <= g; i += 32) ot[i] = bad ? -1 : (i < tau ? (i < 32 ? X0 : X1) : (i == tau ? found : -1));
        if (lane == 0) prm.out_len[b] = bad ? -1 : tau + 1;
    }
    if (lane == 0) {
        ps.sel[static_cast<size_t>(round + 1) * prm.B + b] = next;
        ps.cnt2[b] = 0u;
        __threadfence();
        atomicAdd(&ps.done[round], add);
    }
    __syncwarp();
}

// A warp's vector at `p` into its ring cell, if it belongs to the row (rows at any alignment: a vector that reaches
// outside the tensor [lo, hi) is put together from the elements inside).
template <int DT>
__device__ __forceinline__ void ph_fetch_edge(uint32_t cell, const char* p, bool in, const char* lo, const char* hi, uint32_t pad, uint64_t pol) {
    if (in && p >= lo && p + 16 <= hi) {
        cp_async16_hint(cell, p, pol);
    } else {
        uint4 v = make_uint4(pad, pad, pad, pad);
        if (in) {
            constexpr int ESZ = (DT == kF32) ? 4 : 2;
            int first, n;
            elements_inside<16 / ESZ>(p, lo, hi, first, n);
            v = row_elements<DT>(p + first * ESZ, -first, n - first, pad);
        }
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(cell), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
    }
}
// AL: rows of whole 16-byte vectors on 16-byte aligned bases.  Otherwise a row is read as the aligned vectors that its
// bytes lie in, and what of the first and the last of them belongs to its neighbours weighs nothing; in a second sweep
// the draft row's elements are shifted onto the target row's grid between two neighbouring cells of the ring.
template <int DT, bool PROBS, bool AL>
__global__ void __launch_bounds__(kPhThreads, 1) verify_phase_kernel(const __grid_constant__ Params prm, const __grid_constant__ PhaseScratch ps) {
    using R = Raw<DT>;
    constexpr int EPV = R::EPV;
    constexpr int ESZ = (DT == kF32) ? 4 : 2;
    constexpr uint32_t kPad = PROBS ? 0u : R::kNegInf;
    const float kPadF = PROBS ? 0.f : -INFINITY;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = prm.gamma, B = prm.B, V = prm.V, units = ps.units;
    const size_t row_bytes = static_cast<size_t>(V) * ESZ;
    const float kf = prm.kf;
    const unsigned limit = prm.wait_limit ? prm.wait_limit : (1u << 22);
    __shared__ PhShared sh;
    extern __shared__ __align__(16) unsigned char dyn[];
    // this round's list: first item and candidate masks of every sequence
    int* s_base = reinterpret_cast<int*>(dyn + kPhWarps * kPhSlots * kPhSlotBytes);
    unsigned* s_lo = reinterpret_cast<unsigned*>(s_base + B + 1);
    unsigned* s_hi = s_lo + B;
    unsigned char* s_last = reinterpret_cast<unsigned char*>(s_hi + B);

    const bool helper = warp == kPhWarps;
    const uint32_t ring = smem_u32(dyn) + static_cast<uint32_t>(helper ? 0 : warp) * (kPhSlots * kPhSlotBytes) + static_cast<uint32_t>(lane) * 16u;
    const uint32_t ring_end = ring + kPhSlots * kPhSlotBytes;
    const uint64_t pol = l2_policy_evict_first();
    const int kw = warp * static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x);      // this warp's part of a list
    const int W = static_cast<int>(gridDim.x) * kPhWarps;
    const char* tgt = static_cast<const char*>(prm.tgt);
    const char* drf = static_cast<const char*>(prm.drf);
    const char* tgt_end = tgt + static_cast<size_t>(B) * (g + 1) * row_bytes;
    const char* drf_end = drf + static_cast<size_t>(B) * g * row_bytes;
    PhRun* const runs = sh.q[helper ? 0 : warp];

    // issue side of this warp
    const char* iA = nullptr;
    const char* iB = nullptr;
    int i_rem = 0;                        // vectors of the open run not yet asked for
    bool i_single = true;
    const char* iAlo = nullptr; const char* iAhi = nullptr;   // unaligned: bounds of the tensor that cell A is read from
    int iq = 0, i_nvq = 0;                // unaligned pairs: this lane's vector of the draft row, and how many there are
    auto issue_step = [&](uint32_t cell) {
        if (AL) {
            const int adv = i_single ? 64 : 32;
            if (i_rem >= adv) {
                cp_async16_hint(cell, iA, pol);
                cp_async16_hint(cell + 512, iB, pol);
            } else if (i_rem > 0) {
                ring_fetch_hint(cell, iA, lane < i_rem, kPad, pol);
                ring_fetch_hint(cell + 512, iB, lane + (adv - 32) < i_rem, kPad, pol);
            }
            i_rem -= adv;
            iA += adv * 16;
            iB += adv * 16;
        } else if (i_rem > 0) {
            ph_fetch_edge<DT>(cell, iA, lane < i_rem, iAlo, iAhi, kPad, pol);
            if (i_single) {
                ph_fetch_edge<DT>(cell + 512, iA + 512, lane + 32 < i_rem, iAlo, iAhi, kPad, pol);
                iA += 1024;
                i_rem -= 64;
            } else {
                // the draft row's vectors under these 32 of the target row, and one more
                ph_fetch_edge<DT>(cell + 512, iB, iq >= 0 && iq < i_nvq, drf, drf_end, kPad, pol);
                if (lane == 31) ph_fetch_edge<DT>(cell + 528, iB + 16, iq + 1 >= 0 && iq + 1 < i_nvq, drf, drf_end, kPad, pol);
                iA += 512;
                iB += 512;
                iq += 32;
                i_rem -= 32;
            }
        }
        cp_async_commit();
    };
    // units k .. k+n-1 of the row that starts at `row`
    auto open_row = [&](const char* row, int k, int n, PhRun& q) {
        const char* base; int h, nv;
        row_grid<DT, AL>(row, V, base, h, nv);
        const int v0 = k * kPhUnit, v1 = min((k + n) * kPhUnit, nv);
        iA = base + static_cast<size_t>(v0 + lane) * 16;
        iB = iA + 512;
        i_rem = v1 - v0;
        if (lane == 0) { q.k = k; q.n = n; q.v0 = v0; q.v1 = v1; q.hP = h; }
        return h;
    };

    // the drafted tokens' logits of sequence b (it is not folded before they are in)
    auto drafted = [&](int b) {
        ph_fetch_drafted<DT>(prm, ps, b, lane);
        __threadfence();
        __syncwarp();
        unsigned last = 0;
        if (lane == 0 && prm.never_signal != 1) last = ph_arrive(&ps.cnt1[b], 1u, static_cast<unsigned>(ps.rows * units) + 1u);
        if (__shfl_sync(0xffffffffu, last, 0)) ph_fold(prm, ps, b, lane, false);
    };

    // ---------------- first sweep ----------------
    if (helper) {
        if (!PROBS && blockIdx.x < B) drafted(blockIdx.x);
        if (!PROBS) ph_fold(prm, ps, blockIdx.x % B, lane, true);
        ph_finalize<DT, PROBS, AL>(prm, ps, blockIdx.x % B, make_uint4(1u, 0u, 0u, 0u), 0, lane, true);
    } else if (PROBS) {
        for (int b = kw; b < B; b += W) ph_fold_probs<DT>(prm, ps, b, lane);
    } else {
        const int rows = ps.rows;
        const int x0 = static_cast<int>(min(static_cast<long long>(kw) * ps.per1, static_cast<long long>(ps.n1))), x1 = min(x0 + ps.per1, ps.n1);
        int n_i = 0;
        int row_i = x0 / units, k_i = x0 % units, left = x1 - x0;
        auto open = [&]() {
            const int n = min(left, units - k_i);
            const int b = row_i / rows, j = row_i % rows;
            const bool is_t = j < g;
            PhRun& q = runs[n_i & (kPhQueue - 1)];
            open_row(is_t ? tgt + target_row(prm, b, j) * row_bytes : drf + draft_row(prm, b, j - g) * row_bytes, k_i, n, q);
            if (lane == 0) { q.b = b; q.c = j; }
            if (!AL) { iAlo = is_t ? tgt : drf; iAhi = is_t ? tgt_end : drf_end; }
            __syncwarp();
            left -= n;
            ++row_i;
            k_i = 0;
            ++n_i;
        };
        auto advance = [&](uint32_t cell) {
            while (i_rem <= 0 && left > 0) open();
            issue_step(cell);
        };
        uint32_t rp = ring;
#pragma unroll 1
        for (int j = 0; j < kPhSlots; ++j) advance(ring + j * kPhSlotBytes);
        // (more sequences than helpers: the warps with the last numbers, which have the least to stream)
        for (int b = static_cast<int>(gridDim.x) + W - 1 - kw; b < B; b += W) drafted(b);
        unsigned arrived = 0;
        int todo = x1 - x0;
        for (int n_c = 0; todo > 0; ++n_c) {
            const PhRun& q = runs[n_c & (kPhQueue - 1)];
            const int b = q.b, j = q.c, k = q.k, n = q.n, h = q.hP, v1 = q.v1;
            int v = q.v0;
            const int nv = AL ? 0 : (h + V + EPV - 1) / EPV;
            float M = kNoRef, s = 0.f;
            double sd = 0.0;
            for (int st = 0; v < v1; v += 64, ++st) {
                cp_async_wait<kPhSlots - 1>();
                float va[EPV], vb[EPV];
                R::unpack(lds128(rp), va);
                R::unpack(lds128(rp + 512), vb);
                if (!AL && (v == 0 || v + 64 >= nv)) { row_mask<EPV>(va, v + lane, h, V, kPadF); row_mask<EPV>(vb, v + 32 + lane, h, V, kPadF); }
                // (the run's reference comes from the first vectors of every lane)
                if (st == 0) M = fmaxf(rintf(warp_max(fmaxf(vec_max<EPV>(va), vec_max<EPV>(vb))) * kf), kNoRef);
                const float was = M;
                f_step_sweep1_single<EPV>(va, vb, kf, M, s);
                if (M != was) sd *= static_cast<double>(ref_scale(was, M));
                if ((st & 15) == 15) { sd += static_cast<double>(ref_keep(s)); s = 0.f; }       // (32-bit sums stay short)
                advance(rp);
                rp += kPhSlotBytes;
                if (rp == ring_end) rp = ring;
            }
            sd = warp_sum_d(sd + static_cast<double>(ref_keep(s)));       // (so it is not infinite where it is scaled)
            const int slot = kw - (b * rows + j) * units / ps.per1;
            if (lane == 0) __stcg(&ps.part[(static_cast<size_t>(b) * rows + j) * ps.slots + slot], make_double2(static_cast<double>(M), sd));
            arrived += static_cast<unsigned>(n);
            todo -= n;
            if (todo <= 0 || (j + 1 == rows && k + n == units)) {      // the end of this warp's part, or of the sequence
                unsigned last = 0;
                if (lane == 0 && prm.never_signal != 1) last = ph_arrive(&ps.cnt1[b], arrived, static_cast<unsigned>(rows * units) + 1u);
                arrived = 0;
                if (__shfl_sync(0xffffffffu, last, 0)) ph_fold(prm, ps, b, lane, false);
            }
        }
        cp_async_wait<0>();
    }

    // ---------------- second sweeps, in rounds ----------------
    if (tid == 0) sh.fail = !ph_wait(&ps.ctr[kPhFolded], ~0u, static_cast<unsigned>(B), prm.status, limit);
    __syncthreads();
    const bool alive = sh.fail == 0;
    bool live = tid < B;                  // this thread's sequence was in the round before
    __threadfence();
    for (int round = 0; alive; ++round) {
        // every CTA makes the same list
        uint4 sel = make_uint4(0u, 0u, 0u, 0u);
        if (live) sel = __ldcg(&ps.sel[static_cast<size_t>(round) * B + tid]);
        const int cnt = __popc(sel.x) + __popc(sel.y) + static_cast<int>(sel.z);
        live = cnt > 0;
        int inc = cnt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += o;
        }
        if (lane == 31) sh.scan[warp] = inc;
        const int parts = __syncthreads_count(cnt > 0);
        if (parts == 0) break;
        const int before = warp_sum_i(lane < warp ? sh.scan[lane] : 0);
        if (tid < B) {
            s_base[tid] = before + inc - cnt;
            s_lo[tid] = sel.x; s_hi[tid] = sel.y; s_last[tid] = static_cast<unsigned char>(sel.z | sel.w << 1);
            if (tid == B - 1) s_base[B] = before + inc;
        }
        __syncthreads();
        const int n2 = s_base[B] * units;
        const int per2 = max((n2 + W - 1) / W, 2);            // (two units at least: a few rows are not cut finer than the loads of one ring)
        const int x0 = helper ? n2 : static_cast<int>(min(static_cast<long long>(kw) * per2, static_cast<long long>(n2))), x1 = min(x0 + per2, n2);
        if (x1 > x0) {
            // the place in the list of this warp's first unit
            const int it = x0 / units;
            int a = 0, z = B - 1;
            while (a < z) { const int m = (a + z + 1) >> 1; if (s_base[m] <= it) a = m; else z = m - 1; }
            unsigned i_lo = s_lo[a], i_hi = s_hi[a];          // this sequence's candidates after the open one
            int i_last = s_last[a] & 1, i_c = 0, i_b = a, k_i = x0 % units, left = x1 - x0, n_i = 0;
            for (int i = s_base[a]; i <= it; ++i) i_c = ph_pop(i_lo, i_hi, i_last, g);
            auto open = [&]() {
                const int n = min(left, units - k_i);
                PhRun& q = runs[n_i & (kPhQueue - 1)];
                const size_t ri = static_cast<size_t>(i_b) * (g + 1) + i_c;
                i_single = i_c == g;
                if (!i_single && lane == 0) cp_async16_s(smem_u32(&q.pos), &ps.pos[ri]);
                const int h = open_row(tgt + target_row(prm, i_b, i_c) * row_bytes, k_i, n, q);
                if (!i_single) {
                    const char* baseQ; int hQ, nvQ;
                    row_grid<DT, AL>(drf + draft_row(prm, i_b, i_c) * row_bytes, V, baseQ, hQ, nvQ);
                    int dq = 0, shift = hQ - h;
                    if (!AL && shift < 0) { shift += EPV; dq = -1; }
                    iq = k_i * kPhUnit + lane + dq;
                    i_nvq = nvQ;
                    iB = baseQ + static_cast<long long>(iq) * 16;
                    if (lane == 0) q.shift = shift;
                }
                if (lane == 0) { q.b = i_b; q.c = i_c; }
                if (!AL) { iAlo = tgt; iAhi = tgt_end; }
                __syncwarp();
                ++n_i;
                left -= n;
                k_i = 0;
                if (left > 0) {           // the next position, of this sequence or of the next one with any
                    if ((i_lo | i_hi) == 0u) {
                        do ++i_b; while (s_base[i_b + 1] == s_base[i_b]);
                        i_lo = s_lo[i_b]; i_hi = s_hi[i_b]; i_last = s_last[i_b] & 1;
                    }
                    i_c = ph_pop(i_lo, i_hi, i_last, g);
                }
            };
            auto advance = [&](uint32_t cell) {
                while (i_rem <= 0 && left > 0) open();
                issue_step(cell);
            };
            uint32_t rp = ring;
            i_rem = 0;
#pragma unroll 1
            for (int j = 0; j < kPhSlots; ++j) advance(ring + j * kPhSlotBytes);
            unsigned arrived = 0;
            int todo = x1 - x0;
            for (int n_c = 0; todo > 0; ++n_c) {
                const PhRun& q = runs[n_c & (kPhQueue - 1)];
                const int b = q.b, c = q.c, k = q.k, n = q.n, h = q.hP, v1 = q.v1;
                int v = q.v0;
                const int nv = AL ? V / EPV : (h + V + EPV - 1) / EPV;
                double* seg = ps.seg + (static_cast<size_t>(b) * (g + 1) + c) * units;
                double acc = 0.0;
                if (c == g) {
                    float* seg_M = ps.seg_M + static_cast<size_t>(b) * units;
                    float M = kNoRef;
                    bool first = true;
                    for (; v < v1; v += 64) {
                        cp_async_wait<kPhSlots - 1>();
                        float va[EPV], vb[EPV];
                        R::unpack(lds128(rp), va);
                        R::unpack(lds128(rp + 512), vb);
                        if (!AL && (v == 0 || v + 64 >= nv)) { row_mask<EPV>(va, v + lane, h, V, kPadF); row_mask<EPV>(vb, v + 32 + lane, h, V, kPadF); }
                        acc = 0.0;
                        if (PROBS) {
                            acc = static_cast<double>(f_sum<EPV>(va)) + static_cast<double>(f_sum<EPV>(vb));
                        } else {
                            if (first) M = fmaxf(rintf(warp_max(fmaxf(vec_max<EPV>(va), vec_max<EPV>(vb))) * kf), kNoRef);
                            first = false;
                            f_step_sweep1_single<EPV>(va, vb, kf, M, acc);
                        }
                        acc = warp_sum_d(acc);
                        if (lane == 0) {
                            __stcg(&seg[v / kPhUnit], PROBS ? acc : ref_keep(acc));
                            if (!PROBS) __stcg(&seg_M[v / kPhUnit], M);
                        }
                        advance(rp);
                        rp += kPhSlotBytes;
                        if (rp == ring_end) rp = ring;
                    }
                    if (!AL && lane == 0 && k + n == units && nv <= (units - 1) * kPhUnit) {      // (a last unit without vectors)
                        __stcg(&seg[units - 1], 0.0);
                        if (!PROBS) __stcg(&seg_M[units - 1], kNoRef);
                    }
                } else {
                    const int shift = AL ? 0 : q.shift;
                    cp_async_wait<kPhSlots - 1>();            // (the position's numbers came with the run's first step)
                    __syncwarp();
                    const float cp = q.pos.x, nMP = q.pos.y, nMQ = q.pos.z;
                    for (; v < v1; v += 32) {
                        cp_async_wait<kPhSlots - 1>();
                        float va[EPV], vb[EPV], t[EPV];
                        if (!AL) __syncwarp();
                        R::unpack(lds128(rp), va);
                        if (AL || shift == 0) {
                            R::unpack(lds128(rp + 512), vb);
                        } else {
                            // the draft row lies `shift` elements off the target row's grid: 16 bytes out of two neighbouring cells
                            const uint32_t at = rp + 512 + static_cast<uint32_t>(shift * ESZ & ~3);
                            uint32_t w[5];
#pragma unroll
                            for (int j = 0; j < 5; ++j) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w[j]) : "r"(at + (j < 4 || ESZ == 2 ? 4 * j : 0)) : "memory");
                            const int bits = (shift * ESZ & 3) * 8;
                            R::unpack(make_uint4(__funnelshift_r(w[0], w[1], bits), __funnelshift_r(w[1], w[2], bits),
                                                 __funnelshift_r(w[2], w[3], bits), __funnelshift_r(w[3], w[4], bits)), vb);
                        }
                        if (!AL) {
                            __syncwarp();                     // (every lane has read its neighbours' cells)
                            if (v == 0 || v + 32 >= nv) { row_mask<EPV>(va, v + lane, h, V, kPadF); row_mask<EPV>(vb, v + lane, h, V, kPadF); }
                        }
                        acc += static_cast<double>(f_pair_sum<EPV, true, PROBS>(va, vb, kf, cp, nMP, nMQ, t));
                        if ((v & 32) || v + 32 >= v1) {       // the end of a unit
                            const double tot = warp_sum_d(acc);
                            if (lane == 0) __stcg(&seg[v / kPhUnit], tot);
                            acc = 0.0;
                        }
                        advance(rp);
                        rp += kPhSlotBytes;
                        if (rp == ring_end) rp = ring;
                    }
                    if (!AL && lane == 0 && k + n == units && nv <= (units - 1) * kPhUnit) __stcg(&seg[units - 1], 0.0);
                }
                arrived += static_cast<unsigned>(n);
                todo -= n;
                // (the next run is open already unless this was the last: the issue side runs ahead)
                if (todo <= 0 || runs[(n_c + 1) & (kPhQueue - 1)].b != b) {
                    unsigned done = 0;
                    if (lane == 0 && !prm.never_signal) done = ph_arrive(&ps.cnt2[b], arrived, static_cast<unsigned>((s_base[b + 1] - s_base[b]) * units));
                    arrived = 0;
                    if (__shfl_sync(0xffffffffu, done, 0)) ph_finalize<DT, PROBS, AL>(prm, ps, b, make_uint4(s_lo[b], s_hi[b], s_last[b] & 1u, s_last[b] >> 1), round, lane, false);
                }
            }
            cp_async_wait<0>();
        }
        if (tid == 0) {
            sh.fail = !ph_wait(&ps.done[round], 0xffffu, static_cast<unsigned>(parts), prm.status, limit);
            sh.word = ld_volatile(&ps.done[round]) >> 16;
        }
        __syncthreads();
        if (sh.fail || sh.word == 0u || round == 1) break;
        __threadfence();
        __syncthreads();
    }

    // the last CTA to leave puts the counters back to zero for the next launch (whatever became of the waits)
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        sh.word = atomicAdd(&ps.ctr[kPhExited], 1u);
    }
    __syncthreads();
    if (sh.word == gridDim.x - 1) {
        for (unsigned i = tid; i < ps.zero_words; i += kPhThreads) ps.ctr[i] = 0u;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static size_t up256p(size_t x) { return (x + 255) / 256 * 256; }

PhasePlan phase_plan(int V, int dtype, bool aligned, int B, int gamma, bool lse, int nctas) {
    PhasePlan pl{};
    const int epv = dtype == kF32 ? 4 : 8;
    // (a row that starts inside a vector lies in one more)
    const long long vecs = aligned ? V / epv : (static_cast<long long>(V) + 2 * epv - 2) / epv;
    pl.units = static_cast<int>((vecs + kPhUnit - 1) / kPhUnit);
    pl.rows = lse ? gamma : 2 * gamma;
    const long long n1 = static_cast<long long>(B) * pl.rows * pl.units, W = static_cast<long long>(nctas) * kPhWarps;
    pl.fits = B <= kPhaseMaxB && V <= (1 << 30) && static_cast<long long>(B) * (2 * gamma + 1) * pl.units < (1LL << 30);
    pl.n1 = static_cast<int>(pl.fits ? n1 : 0);
    // (four units at least: where the rows are few, the pieces a row is folded from stay few too)
    pl.per1 = static_cast<int>((n1 + W - 1) / W < 4 ? 4 : (n1 + W - 1) / W);
    pl.slots = (pl.units - 1) / pl.per1 + 2;
    return pl;
}

// counters: apart, zero between launches (the kernel leaves them so)
size_t phase_scratch(void* base, unsigned* counters, int B, int gamma, const PhasePlan& pl, PhaseScratch* ps) {
    const size_t pos = static_cast<size_t>(B) * (gamma + 1);
    size_t used = 0;
    auto take = [&](size_t bytes) { void* q = static_cast<char*>(base) + used; used += up256p(bytes); return q; };
    ps->ctr = counters;
    ps->done = counters + 64;
    ps->cnt1 = counters + 72;
    ps->cnt2 = ps->cnt1 + kPhaseMaxB;
    ps->zero_words = kPhaseCounterWords;
    ps->part = static_cast<double2*>(take(static_cast<size_t>(B) * pl.rows * pl.slots * sizeof(double2)));
    ps->drafted = static_cast<float2*>(take(static_cast<size_t>(B) * gamma * sizeof(float2)));
    ps->pos = static_cast<PhPos*>(take(pos * sizeof(PhPos)));
    ps->sel = static_cast<uint4*>(take(static_cast<size_t>(B) * 3 * sizeof(uint4)));
    ps->rest = static_cast<uint2*>(take(static_cast<size_t>(B) * sizeof(uint2)));
    ps->seg_M = static_cast<float*>(take(static_cast<size_t>(B) * pl.units * sizeof(float)));
    ps->seg = static_cast<double*>(take(pos * pl.units * sizeof(double)));
    ps->n1 = pl.n1; ps->rows = pl.rows; ps->units = pl.units; ps->per1 = pl.per1; ps->slots = pl.slots;
    return used;
}

using PKernelFn = void (*)(const Params, const PhaseScratch);
static PKernelFn pick_phase(int dtype, bool probs, bool aligned) {
    if (probs) return dtype == kF32 ? verify_phase_kernel<kF32, true, true> : verify_phase_kernel<kBF16, true, true>;
    if (aligned) return dtype == kF32 ? verify_phase_kernel<kF32, false, true> : verify_phase_kernel<kBF16, false, true>;
    return dtype == kF32 ? verify_phase_kernel<kF32, false, false> : verify_phase_kernel<kBF16, false, false>;
}

static size_t phase_smem(int B) {
    return static_cast<size_t>(kPhWarps) * kPhSlots * kPhSlotBytes + static_cast<size_t>(B) * 13 + 16;
}

int phase_max_ctas(int dtype, int sm_count) {
    for (int v = 0; v < 3; ++v) {
        PKernelFn fn = pick_phase(dtype, v == 2, v != 1);
        int n = 0;
        if (cudaFuncSetAttribute(reinterpret_cast<const void*>(fn), cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(phase_smem(kPhaseMaxB))) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, kPhThreads, phase_smem(kPhaseMaxB)) != cudaSuccess || n < 1) {
            cudaGetLastError();
            return 0;
        }
    }
    return sm_count;                      // one CTA per SM: all of them resident at once, as the waits need
}

cudaError_t launch_phase(const Params& prm, const PhaseScratch& ps, int dtype, bool aligned, int nctas, cudaStream_t stream) {
    Params p = prm;
    PhaseScratch s = ps;
    void* args[] = {&p, &s};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(pick_phase(dtype, prm.probs != 0, aligned)), dim3(nctas), dim3(kPhThreads), args,
                                       phase_smem(prm.B), stream);
}

}  // namespace bv
