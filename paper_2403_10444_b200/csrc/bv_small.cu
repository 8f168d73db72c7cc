// Block Verification (Algorithm 2, also with supplied draft normalisers), Greedy Block Verification
// (Algorithm 4) and Token Verification (Algorithm 1) for batches so small that a launch is a matter
// of latency, not of bandwidth (a few sequences: the whole input fits in L2).
//
// The flow kernel hands work from CTA to CTA through queues and counters in global memory, and a
// sequence goes through a dozen such hand-overs of a microsecond or more each.  Here all CTAs of a
// cooperative launch walk through three phases, a grid-wide barrier between the first two:
//   1. every row (all 2 gamma + 1 of every sequence, whether the algorithm will want them or not:
//      the bytes are few) is cut into chunks and every CTA reduces its chunks to {reference, sum};
//   2. every CTA combines all chunks (fp64) and runs the scalar part for every sequence itself -
//      normalisers, ratios of the drafted tokens, the recursion of Eq. "def_as" or the tests of
//      Algorithm 1, and which positions can be the selected one - so that all CTAs know the same
//      list of (position, piece) items without talking to each other; each takes its share and
//      leaves per-segment sums of the residual terms max(p_i P_i - Q_i, 0) (rows now come from L2);
//   3. the CTA whose item is the last of a sequence ends it, a warp per candidate: S_i and h_i (Eq. "pacc_block") and, if the
//      position passes, its token by inverse CDF over the segment sums and a rescan of one segment; then tau and the output.
//      (A second barrier, the sums of all candidates, and only then the chosen one's token were two trips to L2 more.)
// Bound: latency, a trip to L2 or memory for each of some eight dependent steps.  Us a call, in brackets with two barriers and pieces
// fixed on the host, in turn on one box: B = 1, gamma = 8, V = 152064 bf16 18.9 (19.1; no more than two runs differ by, and 18.9 to 20.4 by box),
// B = 8, V = 32000 in 32 bits 19.5 (22.6), B = 24, gamma = 5, V = 50257 45.2 (47.3; 42 to 46 by box).
// Arithmetic, sampling convention and outputs are those of the flow kernel.
#include <cooperative_groups.h>

#include "bv_flow_common.cuh"

namespace bv {

constexpr int kSmThreads = 512;       // streaming threads; one more warp fetches the scalars while they stream
constexpr int kSmWarps = kSmThreads / 32;
constexpr int kSmAllThreads = kSmThreads + 32;
constexpr int kSmMaxRows = 1056;      // rows B (2 gamma + 1) whose normalisers a CTA keeps in shared memory
constexpr int kSmMaxPos = 560;        // positions B (gamma + 1)
constexpr int kSmGroup = 4;           // vectors of a thread that the first phase goes through together where its loads run ahead
constexpr int kSmAhead = 3;           // ... groups of them in flight
constexpr int kSmRingBytes = kSmAhead * kSmGroup * kSmThreads * 16;
constexpr int kSmInFlight = 8;        // 16-byte loads a thread has in flight in the first phase
constexpr int kSmPairsInFlight = 5;   // pairs of them in the second (unaligned rows: one less, the registers)
constexpr int kSmMaxUni = kSmMaxPos + kSmallMaxB;   // uniforms B (gamma + 2)

struct SmallShared {
    float rowM[kSmMaxRows];
    double rowZ[kSmMaxRows];
    double pch[kSmMaxPos];            // p_i of every position (Algorithm 1: unused)
    float csc[kSmMaxPos];             // p_i Z_Q / Z_P: the scale of the target terms against the draft terms
    double ratio[kSmMaxPos];          // P_i(X_{i+1}) / Q_i(X_{i+1})
    unsigned mask_lo[kSmallMaxB], mask_hi[kSmallMaxB];   // candidate positions 0 .. 63 of a sequence
    int last_wanted[kSmallMaxB];      // position gamma is a candidate
    int bad[kSmallMaxB];
    int tv_tau[kSmallMaxB];
    int item0[kSmallMaxB + 1];        // first item of every sequence in the second phase
    float wM[2][kSmWarps];
    float wS[2][kSmWarps];
    double cS[kMaxGamma];             // third phase: S_i of this CTA's sequence, the positions' tokens, which of them pass
    int found[kMaxGamma + 1];
    unsigned char pass[kMaxGamma + 1];
    int np;                           // pieces a position is cut into in the second phase
    unsigned ends;                    // sequences whose last item was this CTA's
    // fetched by the extra warp during the first phase: the logits of the drafted tokens, the uniforms
    float zp[kSmMaxPos], zq[kSmMaxPos];
    unsigned char xok[kSmMaxPos];
    float u[kSmMaxUni];
};

// the grid-wide barrier: arrivals are counted up through the launch; the wait is bounded
// (absent: a test switch; the CTA does not arrive, so that every CTA's wait runs out)
__device__ __forceinline__ bool small_grid_barrier(unsigned* counter, unsigned target, int* status, unsigned limit, bool absent) {
    __syncthreads();
    bool ok = true;
    if (threadIdx.x == 0) {
        __threadfence();
        if (!absent) atomicAdd(counter, 1u);
        unsigned spins = 0;
        while (ld_volatile(counter) < target) {
            if (++spins > limit) { if (status) atomicExch(status, 1); ok = false; break; }
        }
        __threadfence();
    }
    return __syncthreads_and(ok ? 1 : 0) != 0;
}

// vectors [s0, s1) of segment `seg` (piece * kSmWarps + warp) of a row cut into nseg segments
__device__ __forceinline__ void small_seg_range(int units, int nseg, int seg, int& s0, int& s1) {
    s0 = static_cast<int>(static_cast<long long>(units) * seg / nseg);
    s1 = static_cast<int>(static_cast<long long>(units) * (seg + 1) / nseg);
}

// row index -> pointer: rows 0 .. gamma of a sequence are its target rows, gamma+1 .. 2 gamma its draft rows
__device__ __forceinline__ const char* small_row(const Params& prm, size_t row_bytes, int b, int j) {
    const int g = prm.gamma;
    return j <= g ? static_cast<const char*>(prm.tgt) + target_row(prm, b, j) * row_bytes
                  : static_cast<const char*>(prm.drf) + draft_row(prm, b, j - g - 1) * row_bytes;
}

// Vector i of a row if it is one of i0 .. i1-1, which lie in the tensor as a whole.
__device__ __forceinline__ uint4 small_load(const char* base, int i, int i0, int i1, uint32_t pad) {
    if (i < i0 || i >= i1) return make_uint4(pad, pad, pad, pad);
    return ld_stream_v4(base + static_cast<long long>(i) * 16);
}
// The first and the last of the nv vectors that a row of V elements lies in, h elements into the first (rows at any alignment):
// the row's own elements, the others as `pad`.
template <int DT>
__device__ __forceinline__ uint4 small_edge(const char* row, int i, int h, int V, uint32_t pad) {
    return row_elements<DT>(row, i * Raw<DT>::EPV - h, V, pad);
}
// PROBS: the rows hold probabilities, used as stored: there is no first phase (and no first barrier).
// AL: rows of whole 16-byte vectors on 16-byte aligned bases.  Otherwise a row is read as the vectors its bytes lie in
// (row_grid), and the draft row of a pair is put on the target row's grid from two neighbouring vectors.
template <int DT, bool PROBS, bool AL>
__global__ void __launch_bounds__(kSmAllThreads, 1) verify_small_kernel(const __grid_constant__ Params prm, const __grid_constant__ SmallScratch sc) {
    using R = Raw<DT>;
    constexpr int EPV = R::EPV;
    constexpr int kPairs = AL ? kSmPairsInFlight : kSmPairsInFlight - 1;
    constexpr uint32_t kPad = PROBS ? 0u : R::kNegInf;       // what a lane beyond the end of a segment finds: no weight
    constexpr size_t ESZ = (DT == kF32) ? 4 : 2;
    __shared__ SmallShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = prm.gamma, B = prm.B, V = prm.V;
    const size_t row_bytes = static_cast<size_t>(prm.V) * ESZ;
    const float kf = prm.kf;
    const int rpb = 2 * g + 1, nrows = B * rpb;
    const unsigned limit = prm.wait_limit ? prm.wait_limit : (1u << 22);
    const bool tv = prm.algo == kTokenVerify;
    const bool all_positions = f_all_positions(prm);
    bool alive = true;

    // ---------------- phase 1: {reference, sum 2^{z k - M}} of every chunk of every row ----------------
    const int nch = sc.nch;
    if (warp == kSmWarps) {
        // nothing here depends on the first phase: the two dependent round trips (token, then its two
        // logits) and the uniforms are over before the streaming warps are
        for (int i = lane; i < B * g; i += 32) {
            const int b = i / g, c = i % g;
            const int x = prm.tok[i];
            const bool xok = x >= 0 && x < prm.V;
            sh.xok[b * (g + 1) + c] = xok;
            sh.zp[b * (g + 1) + c] = xok ? static_cast<float>(load_logit<DT>(small_row(prm, row_bytes, b, c), x)) : 0.f;
            sh.zq[b * (g + 1) + c] = xok ? static_cast<float>(load_logit<DT>(small_row(prm, row_bytes, b, g + 1 + c), x)) : 0.f;
        }
        for (int i = lane; i < B * (g + 2); i += 32) sh.u[i] = prm.uni[i];
    }
    const int items = PROBS ? 0 : nrows * nch;
    // With loads ahead (small_plan) every thread's vectors go through a ring of its own in shared memory, kSmAhead groups ahead of the
    // arithmetic and on into the next item: a CTA has as many warps as one item can use, and with the loads of eight vectors waited for
    // together and then their exponentials, neither memory nor the exponential pipe is busy for more than half of the time.
    if (sc.ahead) {
        extern __shared__ __align__(16) unsigned char cells[];
        const uint32_t ring = smem_u32(cells) + static_cast<uint32_t>(tid) * 16u;
        struct Part { const char* base; int h, nv, u0, u1, i0, i1; } pt;      // chunk of a row: its vectors, and those between the row's outer two
        auto part_of = [&](int item) {
            const int rid = item / nch;
            row_grid<DT, AL>(small_row(prm, row_bytes, rid / rpb, rid % rpb), V, pt.base, pt.h, pt.nv);
            small_seg_range(pt.nv, nch, item % nch, pt.u0, pt.u1);
            pt.i0 = AL ? pt.u0 : max(pt.u0, 1);
            pt.i1 = AL ? pt.u1 : min(pt.u1, pt.nv - 1);
        };
        auto wanted = [&](int item) { return prm.lse_d == nullptr || item / nch % rpb <= g; };      // (a draft row whose normaliser is supplied: nothing to learn)
        int item_i = static_cast<int>(blockIdx.x), i_at = 0, i_end = 0;       // issue side: item, the next of its vectors, their end
        const char* i_base = nullptr;
        auto open = [&]() {
            for (; item_i < items; item_i += gridDim.x) {
                if (!wanted(item_i)) continue;
                part_of(item_i);
                i_base = pt.base; i_at = pt.i0 + tid; i_end = pt.i1;
                if (pt.i0 < pt.i1) break;
            }
        };
        auto issue = [&](uint32_t cell) {
            if (item_i < items) {
#pragma unroll
                for (int j = 0; j < kSmGroup; ++j)
                    ring_fetch_s(cell + j * kSmThreads * 16, i_base + static_cast<long long>(i_at + j * kSmThreads) * 16, i_at + j * kSmThreads < i_end, R::kNegInf);
                i_at += kSmGroup * kSmThreads;
                if (i_at - tid >= i_end) { item_i += gridDim.x; open(); }
            }
            cp_async_commit();
        };
        if (warp < kSmWarps) {
            open();
#pragma unroll 1
            for (int a = 0; a < kSmAhead; ++a) issue(ring + a * kSmGroup * kSmThreads * 16);
        }
        uint32_t rp = ring;
        int turn = 0;
        for (int item = blockIdx.x; item < items; item += gridDim.x) {
            if (!wanted(item)) continue;
            const int rid = item / nch;
            part_of(item);
            // (a row that is not whole vectors: its outer two are put together from elements, one each by two lanes of a warp)
            uint4 outer = make_uint4(R::kNegInf, R::kNegInf, R::kNegInf, R::kNegInf);
            if (!AL && warp == kSmWarps - 1) {
                const char* row = small_row(prm, row_bytes, rid / rpb, rid % rpb);
                if (lane == 0 && pt.u0 == 0) outer = small_edge<DT>(row, 0, pt.h, V, R::kNegInf);
                if (lane == 1 && pt.u1 == pt.nv && pt.nv > 1) outer = small_edge<DT>(row, pt.nv - 1, pt.h, V, R::kNegInf);
            }
            const int i1 = pt.i1;
            float M = kNoRef, s = 0.f;
            for (int base = pt.i0; warp < kSmWarps && base < i1; base += kSmThreads * kSmGroup) {
                cp_async_wait<kSmAhead - 1>();
                uint4 raw[kSmGroup];
#pragma unroll
                for (int j = 0; j < kSmGroup; ++j) raw[j] = lds128(rp + j * kSmThreads * 16);
                // one reference for all of them, the rounded maximum of their logits (a test of every vector's sum before the next
                // one's exponentials is a chain that a few warps do not hide)
                uint4 top = raw[0];
#pragma unroll
                for (int j = 1; j < kSmGroup; ++j) top = vec_max<DT>(top, raw[j]);
                float v[EPV];
                R::unpack(top, v);
                const float y = fmaxf(M, rintf(warp_max(vec_max<EPV>(v)) * kf));
                s = ref_sum(s, M, y);
                M = y;
#pragma unroll
                for (int j = 0; j < kSmGroup; ++j) {
                    if (base + j * kSmThreads + (warp << 5) < i1) {          // (warp-uniform)
                        R::unpack(raw[j], v);
                        s += f_exp_sum<EPV>(v, kf, -M);
                    }
                }
                issue(rp);
                rp += kSmGroup * kSmThreads * 16;
                if (rp == ring + kSmAhead * kSmGroup * kSmThreads * 16) rp = ring;
            }
            if (!AL && warp == kSmWarps - 1) {
                float v[EPV];
                R::unpack(outer, v);
                f_accumulate<EPV>(v, kf, M, s);
            }
            s = warp_sum(s);
            if (lane == 0 && warp < kSmWarps) { sh.wM[turn][warp] = M; sh.wS[turn][warp] = s; }
            __syncthreads();
            if (warp == 0) {                  // (the next item's shares go to the other half, and the barrier after it is behind this)
                const float m = lane < kSmWarps ? sh.wM[turn][lane] : kNoRef;
                const float Mc = warp_max(m);
                double z = lane < kSmWarps ? static_cast<double>(ref_keep(sh.wS[turn][lane])) * static_cast<double>(ref_scale(m, Mc)) : 0.0;
                z = warp_sum_d(z);
                if (lane == 0) __stcg(&sc.part[static_cast<size_t>(rid) * nch + item % nch], make_double2(static_cast<double>(Mc), z));
            }
            turn ^= 1;
        }
    } else {
        for (int item = blockIdx.x; item < items; item += gridDim.x) {
            const int rid = item / nch, ch = item % nch;
            if (prm.lse_d != nullptr && rid % rpb > g) continue;      // (a draft row whose normaliser is supplied: nothing to learn)
            const char* row = small_row(prm, row_bytes, rid / rpb, rid % rpb);
            const char* base16; int h, nv, u0, u1;
            row_grid<DT, AL>(row, V, base16, h, nv);
            small_seg_range(nv, nch, ch, u0, u1);
            // (a row that is not whole vectors: its outer two are put together from elements, one each by two lanes of a warp that
            // has a vector less to stream than others, and between them nothing tells one vector from another)
            const int i0 = AL ? u0 : max(u0, 1), i1 = AL ? u1 : min(u1, nv - 1);
            uint4 outer = make_uint4(R::kNegInf, R::kNegInf, R::kNegInf, R::kNegInf);
            if (!AL && warp == kSmWarps - 1) {
                if (lane == 0 && u0 == 0) outer = small_edge<DT>(row, 0, h, V, R::kNegInf);
                if (lane == 1 && u1 == nv && nv > 1) outer = small_edge<DT>(row, nv - 1, h, V, R::kNegInf);
            }
            float M = kNoRef, s = 0.f;
            for (int base = i0; warp < kSmWarps && base < i1; base += kSmThreads * kSmInFlight) {
                uint4 raw[kSmInFlight];
#pragma unroll
                for (int j = 0; j < kSmInFlight; ++j) raw[j] = small_load(base16, base + j * kSmThreads + tid, i0, i1, R::kNegInf);
                // One reference for all of them, the rounded maximum of their logits: a test of every vector's sum before the next
                // one's exponentials (f_accumulate) is a chain that sixteen warps do not hide (B = 1: 3.7 us until the last row is in,
                // like this 3.2).
                uint4 top = raw[0];
#pragma unroll
                for (int j = 1; j < kSmInFlight; ++j) top = vec_max<DT>(top, raw[j]);
                {
                    float v[EPV];
                    R::unpack(top, v);
                    const float y = fmaxf(M, rintf(warp_max(vec_max<EPV>(v)) * kf));
                    s = ref_sum(s, M, y);
                    M = y;
                }
#pragma unroll
                for (int j = 0; j < kSmInFlight; ++j) {
                    if (base + j * kSmThreads + (warp << 5) < i1) {          // (warp-uniform)
                        float v[EPV];
                        R::unpack(raw[j], v);
                        s += f_exp_sum<EPV>(v, kf, -M);
                    }
                }
            }
            if (!AL && warp == kSmWarps - 1) {
                float v[EPV];
                R::unpack(outer, v);
                f_accumulate<EPV>(v, kf, M, s);
            }
            s = warp_sum(s);
            if (lane == 0 && warp < kSmWarps) { sh.wM[0][warp] = M; sh.wS[0][warp] = s; }
            __syncthreads();
            if (warp == 0) {
                const float m = lane < kSmWarps ? sh.wM[0][lane] : kNoRef;
                const float Mc = warp_max(m);
                double z = lane < kSmWarps ? static_cast<double>(ref_keep(sh.wS[0][lane])) * static_cast<double>(ref_scale(m, Mc)) : 0.0;
                z = warp_sum_d(z);
                if (lane == 0) sc.part[static_cast<size_t>(rid) * nch + ch] = make_double2(static_cast<double>(Mc), z);
            }
            __syncthreads();
        }
    }
    if (PROBS) __syncthreads();
    else alive = small_grid_barrier(sc.barrier, gridDim.x, prm.status, limit, prm.never_signal && blockIdx.x == 0);

    // ---------------- phase 2a: normalisers of every row, the scalar part of every sequence ----------------
    if (alive) {
        for (int rid = tid; rid < nrows; rid += kSmAllThreads) {
            if (PROBS) { sh.rowM[rid] = 0.f; sh.rowZ[rid] = 1.0; continue; }
            if (prm.lse_d != nullptr && rid % rpb > g) {
                // the supplied normaliser as an integer reference at or above every scaled logit of the row
                // plus a sum in [2^-1/2, 2^1/2]; a value that is not finite leaves the row without a reference
                const double L2 = static_cast<double>(prm.lse_d[static_cast<size_t>(rid / rpb) * g + (rid % rpb - g - 1)]) * 1.4426950408889634073599246810019;
                const bool fin = L2 > -1e300 && L2 < 1e300;
                sh.rowM[rid] = fin ? static_cast<float>(rint(L2)) : kNoRef;
                sh.rowZ[rid] = fin ? exp2(L2 - rint(L2)) : 0.0;
                continue;
            }
            float M = kNoRef;
            double Z = 0.0;
            for (int c0 = 0; c0 < nch; c0 += 8) {             // (eight loads in flight, nothing in local memory)
                double2 p[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) p[j] = c0 + j < nch ? __ldcg(&sc.part[static_cast<size_t>(rid) * nch + c0 + j]) : make_double2(kNoRef, 0.0);
                float mm = M;
#pragma unroll
                for (int j = 0; j < 8; ++j) mm = fmaxf(mm, static_cast<float>(p[j].x));
                Z *= static_cast<double>(ref_scale(M, mm));
#pragma unroll
                for (int j = 0; j < 8; ++j) Z += p[j].y * static_cast<double>(ref_scale(static_cast<float>(p[j].x), mm));
                M = mm;
            }
            sh.rowM[rid] = M;
            sh.rowZ[rid] = Z;
        }
    }
    __syncthreads();
    if (alive) {
        for (int b = warp; warp < kSmWarps && b < B; b += kSmWarps) {
            // lanes c and c + 32 speak for rows / positions c and c + 32
            double rat[2] = {1.0, 1.0};
            bool badrow[2] = {false, false};
            float eta[2] = {0.f, 0.f};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h == 1 && g <= 32) break;
                const int c = lane + 32 * h;
                if (c < g) {
                    const float MP = sh.rowM[b * rpb + c], MQ = sh.rowM[b * rpb + g + 1 + c];
                    const double ZP = sh.rowZ[b * rpb + c], ZQ = sh.rowZ[b * rpb + g + 1 + c];
                    const bool xok = sh.xok[b * (g + 1) + c] != 0;
                    const double zp = sh.zp[b * (g + 1) + c], zq = sh.zq[b * (g + 1) + c];
                    bool bad;
                    if (PROBS) {
                        // the stored numbers themselves: Q must be a positive finite number, P a non-negative finite one
                        bad = !xok || !(zq > 0.0 && zq < static_cast<double>(INFINITY)) || !(zp >= 0.0 && zp < static_cast<double>(INFINITY));
                        rat[h] = bad ? 0.0 : zp / zq;
                    } else {
                        bad = !(MP > kNoRef && MP < INFINITY) || !row_sum_ok(ZP) ||
                              !(MQ > kNoRef && MQ < INFINITY) || !row_sum_ok(ZQ) || !xok || zq == -INFINITY;
                        rat[h] = bad ? 0.0 : exp2((zp - zq) * prm.kd - (static_cast<double>(MP) - static_cast<double>(MQ))) * (ZQ / ZP);
                    }
                    badrow[h] = bad;
                    sh.ratio[b * (g + 1) + c] = rat[h];
                    // the uniform that decides about this lane's row / position
                    eta[h] = tv ? sh.u[b * (g + 2) + c] : (c >= 1 ? sh.u[b * (g + 2) + c - 1] : 0.f);
                }
            }
            const float MPg = sh.rowM[b * rpb + g];
            const double ZPg = sh.rowZ[b * rpb + g];
            const bool bad_last = !PROBS && (!(MPg > kNoRef && MPg < INFINITY) || !row_sum_ok(ZPg));
            const unsigned bad_lo = __ballot_sync(0xffffffffu, badrow[0]), bad_hi = __ballot_sync(0xffffffffu, badrow[1]);
            unsigned m_lo = 0, m_hi = 0;
            int lastw = 0, bad = 0, tau_tv = 0;
            if (tv) {
                // Algorithm 1: test c + 1 on row c; tau = the tests passed before the first failure
                bool pass[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int c = lane + 32 * h;
                    const double hw = fmin(rat[h], 1.0);
                    pass[h] = c >= g || (hw > 0.0 && static_cast<double>(eta[h]) <= hw);
                }
                const unsigned f_lo = __ballot_sync(0xffffffffu, !pass[0]), f_hi = __ballot_sync(0xffffffffu, !pass[1]);
                tau_tv = f_lo ? __ffs(f_lo) - 1 : (f_hi ? 32 + __ffs(f_hi) - 1 : g);
                // (a fault counts if its row is among rows 0 .. min(tau, gamma - 1), or in the last target row when tau = gamma)
                const int last_pair = tau_tv < g ? tau_tv : g - 1;
                const unsigned long long badrows = static_cast<unsigned long long>(bad_lo) | (static_cast<unsigned long long>(bad_hi) << 32);
                bad = (badrows & (last_pair >= 63 ? ~0ull : ((2ull << last_pair) - 1ull))) != 0ull || (tau_tv == g && bad_last);
                if (all_positions) bad = bad;     // (diagnostics never widen what counts as a fault)
                if (tau_tv == g) lastw = 1;
                else if (tau_tv < 32) m_lo = 1u << tau_tv;
                else m_hi = 1u << (tau_tv - 32);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int c = lane + 32 * h;
                    if (c < g) sh.csc[b * (g + 1) + c] = static_cast<float>(sh.rowZ[b * rpb + g + 1 + c] / sh.rowZ[b * rpb + c]);
                }
            } else {
                // (every lane walks the chain, the ratios read together beforehand from where they have just been left)
                __syncwarp();
                double pc = 1.0, mine[2] = {1.0, 1.0};
                for (int c0 = 0; c0 < g; c0 += 8) {
                    double r[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) r[j] = c0 + j < g ? sh.ratio[b * (g + 1) + c0 + j] : 1.0;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int c = c0 + j;
                        if (c >= g) break;
                        if (c == lane) mine[0] = pc;
                        if (c == lane + 32) mine[1] = pc;
                        const double next = pc * r[j];
                        pc = prm.greedy ? next : fmin(next, 1.0);
                    }
                }
                const double p_g = pc;
                bool need[2] = {false, false};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int c = lane + 32 * h;
                    if (c < g) {
                        // h_c <= p_c: a position whose uniform lies above p_c cannot be the selected one
                        need[h] = all_positions || c == 0 || static_cast<double>(eta[h]) <= mine[h] * (1.0 + 1e-6);
                        sh.pch[b * (g + 1) + c] = mine[h];
                        sh.csc[b * (g + 1) + c] = static_cast<float>(mine[h] * (sh.rowZ[b * rpb + g + 1 + c] / sh.rowZ[b * rpb + c]));
                    }
                }
                m_lo = __ballot_sync(0xffffffffu, need[0]);
                m_hi = __ballot_sync(0xffffffffu, need[1]);
                const float eta_g = sh.u[b * (g + 2) + g - 1];
                lastw = all_positions || static_cast<double>(eta_g) <= p_g * (1.0 + 1e-6);
                bad = (bad_lo | bad_hi) != 0u || bad_last;
                if (lane == 0) sh.pch[b * (g + 1) + g] = p_g;
            }
            if (lane == 0) {
                sh.mask_lo[b] = m_lo; sh.mask_hi[b] = m_hi; sh.last_wanted[b] = lastw;
                sh.bad[b] = bad; sh.tv_tau[b] = tau_tv;
                sh.csc[b * (g + 1) + g] = 1.f;
            }
        }
    }
    __syncthreads();
    if (warp == 0) {
        const int n = alive && lane < B ? __popc(sh.mask_lo[lane]) + __popc(sh.mask_hi[lane]) + sh.last_wanted[lane] : 0;
        int acc = n;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, acc, off);
            if (lane >= off) acc += o;
        }
        // Pieces a position: a CTA goes through its items one after the other, each its share of the row and what ends it (as
        // long as streaming some 1200 vectors), so the count is the one with the least rounds x (vectors + 1200).
        const int all = __shfl_sync(0xffffffffu, acc, 31), k = (lane & 7) + 1, units = V / EPV;
        const unsigned rounds = static_cast<unsigned>((all * k + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x));
        const unsigned cost = k == 1 || (k <= sc.np && units / k >= 512) ? min(rounds * static_cast<unsigned>(units / k + 1200), 0x0fffffffu) : 0x0fffffffu;
        const unsigned least = __reduce_min_sync(0xffffffffu, cost);
        const int np = ((__ffs(__ballot_sync(0xffffffffu, cost == least)) - 1) & 7) + 1;
        if (lane < B) sh.item0[lane] = (acc - n) * np;
        if (lane == B - 1) { sh.item0[B] = acc * np; sh.np = np; }
    }
    __syncthreads();

    const int np = sh.np, nseg = np * kSmWarps;

    // ---------------- phase 3: the end of sequence b (all warps of a CTA) ----------------
    auto finish = [&](int b) {
        const unsigned m_lo = sh.mask_lo[b], m_hi = sh.mask_hi[b];
        const float* u = sh.u + b * (g + 2);
        for (int i = warp; i <= g; i += kSmAllThreads / 32) {
            const bool have_q = i < g, cand = have_q ? ((i < 32 ? m_lo >> i : m_hi >> (i - 32)) & 1u) != 0u : sh.last_wanted[b] != 0;
            double S = 0.0;
            int y = -1;
            bool pass = false;
            if (cand) {
                // S_i, and by fp64 sums of the segment totals in index order the segment that holds the sample
                const double* segs = sc.seg + (static_cast<size_t>(b) * (g + 1) + i) * (sc.np * kSmWarps);
                double w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = 4 * lane + j < nseg ? __ldcg(&segs[4 * lane + j]) : 0.0;
                const double d1 = w[0], d2 = d1 + w[1], d3 = d2 + w[2], d4 = d3 + w[3];
                double inc = d4;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const double o = shfl_up_d(inc, off);
                    if (lane >= off) inc += o;
                }
                const double total = shfl_d(inc, 31);
                // h_gamma = p_gamma, h_i = S_i / (S_i + 1 - p_i); position 0 is what remains when no other passes
                if (have_q) S = total / sh.rowZ[b * rpb + g + 1 + i];
                if (tv || i == 0) {
                    pass = true;
                } else {
                    const double p = sh.pch[b * (g + 1) + i], hw = have_q ? f_weight(p, S) : p;
                    pass = hw > 0.0 && static_cast<double>(u[i - 1]) <= hw;
                }
                if (pass && total > 0.0 && total < static_cast<double>(INFINITY)) {
                    const double t = static_cast<double>(u[have_q ? g : g + 1]) * total;
                    double exc = shfl_up_d(inc, 1);
                    if (lane == 0) exc = 0.0;
                    const double p0 = exc, p1 = exc + d1, p2 = exc + d2, p3 = exc + d3, p4 = exc + d4;
                    const bool h1 = p1 > t && w[0] > 0.0, h2 = p2 > t && w[1] > 0.0;
                    const bool h3 = p3 > t && w[2] > 0.0, h4 = p4 > t && w[3] > 0.0;
                    const unsigned hit = __ballot_sync(0xffffffffu, h1 || h2 || h3 || h4);
                    const unsigned nz = __ballot_sync(0xffffffffu, d4 > 0.0);
                    int e = 3, src;
                    double bef = p3;
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
                    const char* rowP = small_row(prm, row_bytes, b, i);
                    const char* rowQ = have_q ? small_row(prm, row_bytes, b, g + 1 + i) : nullptr;
                    const float cp = sh.csc[b * (g + 1) + i], nMP = -sh.rowM[b * rpb + i], nMQ = have_q ? -sh.rowM[b * rpb + g + 1 + i] : 0.f;
                    const char* baseP; int h, nv, s0, s1;
                    row_grid<DT, AL>(rowP, V, baseP, h, nv);
                    small_seg_range(nv, nseg, sel, s0, s1);
                    y = AL ? f_rescan<DT, PROBS, 5>(rowP, rowQ, s0, s1, lane, kf, cp, nMP, nMQ, t - before)
                           : f_rescan_any<DT, PROBS, 3>(rowP, rowQ, V, s0, s1, lane, kf, cp, nMP, nMQ, t - before);
                }
            }
            if (lane == 0) { if (have_q) sh.cS[i] = S; sh.found[i] = y; sh.pass[i] = pass; }
        }
        __syncthreads();
        if (warp == 0) {
            // tau = max{i >= 1 : h_i > 0 and eta_i <= h_i}, else 0
            int tau = tv ? sh.tv_tau[b] : 0;
            if (!tv) {
                const unsigned p_lo = __ballot_sync(0xffffffffu, lane < g && sh.pass[lane < g ? lane : 0] != 0), p_hi = __ballot_sync(0xffffffffu, lane + 32 < g && sh.pass[lane + 32 < g ? lane + 32 : 0] != 0);
                if (sh.pass[g]) tau = g;
                else if (p_hi) tau = 32 + 31 - __clz(p_hi);
                else if (p_lo) tau = 31 - __clz(p_lo);
            }
            const int found = sh.found[tau];
            const bool bad = sh.bad[b] != 0 || found < 0;      // (an empty residual where the algorithm must sample: a domain error)
            int32_t* ot = prm.out_tokens + static_cast<size_t>(b) * (g + 1);
            const int32_t* X = prm.tok + static_cast<size_t>(b) * g;
            for (int i = lane; i <= g; i += 32) ot[i] = bad ? -1 : (i < tau ? X[i] : (i == tau ? found : -1));
            if (lane == 0) prm.out_len[b] = bad ? -1 : tau + 1;
            if (all_positions) {
                const double ln2 = 0.693147180559945309417232;
                const float nanf_ = __int_as_float(0x7fc00000);
                for (int i = lane; i <= g; i += 32) {
                    const size_t o1 = static_cast<size_t>(b) * (g + 1) + i, o0 = static_cast<size_t>(b) * g + i;
                    float pv, hv, Sv = nanf_;
                    if (tv) {
                        pv = nanf_;
                        hv = i == 0 ? 1.f : static_cast<float>(fmin(sh.ratio[b * (g + 1) + i - 1], 1.0));
                        if (i == tau && i < g) Sv = static_cast<float>(sh.cS[i]);
                    } else {
                        const double p = sh.pch[b * (g + 1) + i];
                        pv = static_cast<float>(p);
                        hv = static_cast<float>(i == 0 ? 1.0 : (i == g ? p : f_weight(p, sh.cS[i])));
                        if (i < g) Sv = static_cast<float>(sh.cS[i]);
                    }
                    if (prm.out_p) prm.out_p[o1] = pv;
                    if (prm.out_h) prm.out_h[o1] = hv;
                    if (prm.out_lse_t) prm.out_lse_t[o1] = static_cast<float>((static_cast<double>(sh.rowM[b * rpb + i]) + log2(sh.rowZ[b * rpb + i])) * ln2);
                    if (i < g && prm.out_S) prm.out_S[o0] = Sv;
                    if (i < g && prm.out_lse_d) prm.out_lse_d[o0] = static_cast<float>((static_cast<double>(sh.rowM[b * rpb + g + 1 + i]) + log2(sh.rowZ[b * rpb + g + 1 + i])) * ln2);
                }
            }
        }
        __syncthreads();
    };

    // ---------------- phase 2b: per-segment sums of the residual terms of every candidate position ----------------
    unsigned ends = 0;                    // sequences whose last item was this CTA's
    if (alive) {
        const int total = sh.item0[B];
        for (int item = blockIdx.x; item < total; item += gridDim.x) {
            const int b = __popc(__ballot_sync(0xffffffffu, lane < B && item >= sh.item0[lane < B ? lane + 1 : 0]));
            const int k = (item - sh.item0[b]) / np, piece = (item - sh.item0[b]) % np;
            // the k-th candidate of the sequence, from position 0 up; position gamma last
            const unsigned c_lo = sh.mask_lo[b], c_hi = sh.mask_hi[b], below = (1u << lane) - 1u;
            const unsigned in_lo = __ballot_sync(0xffffffffu, (c_lo >> lane & 1u) && __popc(c_lo & below) == k);
            const unsigned in_hi = __ballot_sync(0xffffffffu, (c_hi >> lane & 1u) && __popc(c_lo) + __popc(c_hi & below) == k);
            const int i = in_lo ? __ffs(in_lo) - 1 : in_hi ? 31 + __ffs(in_hi) : g;
            const bool have_q = i < g;
            const char* rowP = small_row(prm, row_bytes, b, i);
            const char* rowQ = have_q ? small_row(prm, row_bytes, b, g + 1 + i) : nullptr;
            const float cp = sh.csc[b * (g + 1) + i];
            const float nMP = -sh.rowM[b * rpb + i], nMQ = have_q ? -sh.rowM[b * rpb + g + 1 + i] : 0.f;
            int s0, s1, hP, nvP, hQ = 0, nvQ = 0;
            const char* baseP;
            const char* baseQ = nullptr;
            row_grid<DT, AL>(rowP, V, baseP, hP, nvP);
            if (have_q) row_grid<DT, AL>(rowQ, V, baseQ, hQ, nvQ);
            int shift = hQ - hP, dq = 0;                      // the draft row's elements against the target row's grid
            if (!AL && shift < 0) { shift += EPV; dq = -1; }
            const int sq = shift * static_cast<int>(ESZ) >> 2, sbits = (shift * static_cast<int>(ESZ) & 3) * 8;
            small_seg_range(nvP, nseg, piece * kSmWarps + (warp < kSmWarps ? warp : 0), s0, s1);
            // (AL: all of a segment's vectors; otherwise the target row's outer two are put together from elements, and so are
            // the draft row's elements under them)
            const int i0 = AL ? s0 : max(s0, 1), i1 = AL ? s1 : min(s1, nvP - 1);
            double acc = 0.0;
            uint4 edge_p = make_uint4(kPad, kPad, kPad, kPad), edge_q = edge_p;
            const bool edges = !AL && warp < kSmWarps && (s0 == 0 || s1 == nvP) && s0 < s1;      // (warp-uniform)
            if (edges) {
                const int i = lane == 0 && s0 == 0 ? 0 : (lane == 1 && s1 == nvP && nvP > 1 ? nvP - 1 : -1);
                if (i >= 0) {
                    edge_p = small_edge<DT>(rowP, i, hP, V, kPad);
                    if (have_q) edge_q = small_edge<DT>(rowQ, i, hP, V, kPad);
                }
            }
            // a draft vector that holds a whole target vector's elements, or some of them, lies in the draft row's tensor: all but
            // its outer two do, and the neighbour of one that is shifted is the next lane's
            for (int base = i0; warp < kSmWarps && base < i1; base += 32 * kPairs) {
                uint4 rp[kPairs], rq[kPairs], rx[AL ? 1 : kPairs];
#pragma unroll
                for (int j = 0; j < kPairs; ++j) {
                    const int v = base + 32 * j + lane;
                    rp[j] = small_load(baseP, v, i0, i1, kPad);
                    if (AL) {
                        rq[j] = small_load(baseQ, v, i0, have_q ? i1 : 0, kPad);
                    } else {
                        const int q1 = have_q && v < i1 ? nvQ : 0;
                        rq[j] = row_vector<DT>(baseQ, v + dq, q1, rowQ, hQ, V, kPad);
                        // (the last lane has nobody to ask, and neither has the one before the end)
                        rx[AL ? 0 : j] = lane == 31 || v + 1 >= i1 ? row_vector<DT>(baseQ, v + dq + 1, q1, rowQ, hQ, V, kPad) : make_uint4(0u, 0u, 0u, 0u);
                    }
                }
#pragma unroll
                for (int j = 0; j < kPairs; ++j) {
                    const int v = base + 32 * j + lane;
                    float vp[EPV], vq[EPV], t[EPV];
                    R::unpack(rp[j], vp);
                    if (AL) {
                        R::unpack(rq[j], vq);
                    } else {
                        const uint4 n = make_uint4(__shfl_down_sync(0xffffffffu, rq[j].x, 1), __shfl_down_sync(0xffffffffu, rq[j].y, 1),
                                                   __shfl_down_sync(0xffffffffu, rq[j].z, 1), __shfl_down_sync(0xffffffffu, rq[j].w, 1));
                        R::unpack(vector_shift(rq[j], lane == 31 || v + 1 >= i1 ? rx[AL ? 0 : j] : n, sq, sbits), vq);
                    }
                    if (have_q) acc += static_cast<double>(f_pair_sum<EPV, true, PROBS>(vp, vq, kf, cp, nMP, nMQ, t));
                    else acc += static_cast<double>(f_pair_sum<EPV, false, PROBS>(vp, vq, kf, cp, nMP, nMQ, t));
                }
            }
            if (edges) {
                float vp[EPV], vq[EPV], t[EPV];
                R::unpack(edge_p, vp);
                R::unpack(edge_q, vq);
                if (have_q) acc += static_cast<double>(f_pair_sum<EPV, true, PROBS>(vp, vq, kf, cp, nMP, nMQ, t));
                else acc += static_cast<double>(f_pair_sum<EPV, false, PROBS>(vp, vq, kf, cp, nMP, nMQ, t));
            }
            acc = warp_sum_d(acc);
            if (lane == 0 && warp < kSmWarps) __stcg(&sc.seg[(static_cast<size_t>(b) * (g + 1) + i) * (sc.np * kSmWarps) + piece * kSmWarps + warp], acc);
        }
        // This CTA's items are in: said of all of them together, so that none waits for another's answer.
        __syncthreads();
        if (warp == 0) {
            __threadfence();
            for (int item = blockIdx.x + lane * static_cast<int>(gridDim.x); __any_sync(0xffffffffu, item < total); item += 32 * static_cast<int>(gridDim.x)) {
                unsigned mine = 0;
                if (item < total) {
                    int b = 0;
                    while (item >= sh.item0[b + 1]) ++b;
                    if (atomicAdd(&sc.seq[b], 1u) + 1u == static_cast<unsigned>(sh.item0[b + 1] - sh.item0[b])) mine = 1u << b;
                }
                ends |= __reduce_or_sync(0xffffffffu, mine);
            }
            __threadfence();
            if (lane == 0) sh.ends = ends;
        }
        __syncthreads();
        ends = sh.ends;
    }

    // No CTA looks at the barrier word or a sequence's counter any more once all have come by here, whatever became of the wait:
    // the last one puts them back to zero.  (A warp that is not on the way to the result does it: the fence, the atomic and its
    // answer at the end of the kernel were 1 us of the 20 that a single sequence takes.)
    if (warp == kSmWarps - 1) {
        unsigned gone = 0;
        if (lane == 0) gone = atomicAdd(sc.barrier + 16, 1u);
        if (__shfl_sync(0xffffffffu, gone, 0) == gridDim.x - 1) {
            if (lane < B) atomicExch(&sc.seq[lane], 0u);
            if (lane == 0) { atomicExch(sc.barrier, 0u); atomicExch(sc.barrier + 16, 0u); }
        }
    }
    for (; ends != 0u; ends &= ends - 1u) finish(__ffs(ends) - 1);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static size_t up256s(size_t x) { return (x + 255) / 256 * 256; }

bool small_fits(int B, int gamma) {
    return B >= 1 && B <= kSmallMaxB && static_cast<long long>(B) * (2 * gamma + 1) <= kSmMaxRows &&
           static_cast<long long>(B) * (gamma + 1) <= kSmMaxPos;
}

// Chunks per row in the first phase.  A CTA goes through its
// items one after the other, each costing its share of the row plus a fixed part (the reduction
// across the CTA and its barriers: about as long as streaming 2500 vectors), so the count is the
// one that minimises rounds x (vectors per item + 2500); no chunk below 512 vectors.
static int small_best_split(long long units, long long rows, int nctas, int most) {
    int best = 1;
    long long best_cost = -1;
    for (int n = 1; n <= most && units / n >= 512; ++n) {
        const long long rounds = (rows * n + nctas - 1) / nctas;
        const long long cost = rounds * (units / n + 2500);
        if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = n; }
    }
    return best;
}

SmallPlan small_plan(long long units, int B, int gamma, int nctas) {
    SmallPlan pl{};
    pl.nch = small_best_split(units, static_cast<long long>(B) * (2 * gamma + 1), nctas, kSmallMaxChunks);
    // Loads ahead of the arithmetic: where a CTA has more than one item, or one of more than 16 vectors a thread (B = 20, gamma = 6,
    // V = 65536, Algorithm 1, 30.7 us without, 28.6 with; B = 12, gamma = 8, V = 32000, all positions, 30.7 / 28.7; B = 24, gamma = 5,
    // V = 50257 alike).  A single item of fewer waits for memory once or twice either way, and the ring only costs: B = 1, gamma = 8,
    // V = 152064 7 % more, B = 3, gamma = 3, V = 256000 2 %, B = 8, V = 32000 in 32 bits 1.5 %.
    pl.ahead = static_cast<long long>(B) * (2 * gamma + 1) * pl.nch > nctas || units / pl.nch > 16 * kSmThreads;
    pl.np = 8;           // (the most: the kernel knows how many positions there are)
    return pl;
}

size_t small_scratch_bytes(int B, int gamma, const SmallPlan& pl) {
    const size_t rows = static_cast<size_t>(B) * (2 * gamma + 1), pos = static_cast<size_t>(B) * (gamma + 1);
    return up256s(rows * pl.nch * sizeof(double2)) + up256s(pos * pl.np * kSmWarps * sizeof(double));
}

// barrier: two words 64 bytes apart; seq: a word a sequence; all zero between launches (the kernel leaves them so)
void small_scratch_layout(void* base, unsigned* barrier, unsigned* seq, int B, int gamma, const SmallPlan& pl, SmallScratch* sc) {
    char* p = static_cast<char*>(base);
    const size_t rows = static_cast<size_t>(B) * (2 * gamma + 1);
    sc->barrier = barrier;
    sc->seq = seq;
    sc->part = reinterpret_cast<double2*>(p);
    sc->seg = reinterpret_cast<double*>(p + up256s(rows * pl.nch * sizeof(double2)));
    sc->nch = pl.nch;
    sc->ahead = pl.ahead;
    sc->np = pl.np;
}

using SKernelFn = void (*)(const Params, const SmallScratch);
static SKernelFn pick_small(int dtype, bool probs, bool aligned) {
    if (probs) return dtype == kF32 ? verify_small_kernel<kF32, true, true> : verify_small_kernel<kBF16, true, true>;
    if (aligned) return dtype == kF32 ? verify_small_kernel<kF32, false, true> : verify_small_kernel<kBF16, false, true>;
    return dtype == kF32 ? verify_small_kernel<kF32, false, false> : verify_small_kernel<kBF16, false, false>;
}

int small_max_ctas(int dtype, int sm_count) {
    for (int v = 0; v < 3; ++v) {
        int n = 0;
        if (cudaFuncSetAttribute(reinterpret_cast<const void*>(pick_small(dtype, v == 2, v != 1)), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmRingBytes) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pick_small(dtype, v == 2, v != 1), kSmAllThreads, kSmRingBytes) != cudaSuccess || n < 1) {
            cudaGetLastError();
            return 0;
        }
    }
    return sm_count;          // one CTA per SM: all of them resident at once, as the barriers need
}

cudaError_t launch_small(const Params& prm, const SmallScratch& sc, int dtype, bool aligned, int nctas, cudaStream_t stream) {
    Params p = prm;
    SmallScratch s = sc;
    if (prm.probs) s.ahead = 0;
    void* args[] = {&p, &s};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(pick_small(dtype, prm.probs != 0, aligned)), dim3(nctas), dim3(kSmAllThreads), args,
                                       s.ahead ? kSmRingBytes : 0, stream);
}

}  // namespace bv
