// C-ABI layer: argument checks, per-device and per-stream workspace, launch-shape selection and
// the host-buffer entry points.  Declarations and contracts are in include/bv.h.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "../../include/bv.h"
#include "bv_launch.h"

namespace {

constexpr int kMaxDevices = 64;
constexpr int kTicketSlots = 64;  // concurrent calls of the cluster kernels on one device each need their own slot
// Logit bytes up to which the small-batch kernel is the default (against the flow kernel, drafts of noise 0.1 / 0.7: Algorithm 2,
// V = 256000, gamma = 16, B = 5 (81 MB) 72 / 55 us against 72 / 66, 6 (97 MB) 84 / 52 against 73 / 67; Algorithm 1, gamma = 8, noise
// 0.1 / 0.7 / 3, B = 18 (149 MB) 73 / 74 / 74 against 85 / 77 / 51, 22 (183 MB) 73 / 74 / 74 against 87 / 81 / 66).  The phase kernel
// takes over below that, but for few sequences or many positions swept (phase_pays).
constexpr long long kSmallBytes[2] = {160LL << 20, 90LL << 20};   // [algo]
// Logit bytes between which the phase kernel is the default for rows of 16-byte vectors ({Algorithm 1, Algorithms 2 and 4,
// Algorithm 2 with supplied normalisers}), and the sequences from which it is on probabilities.  Measured at V = 128256 bf16,
// gamma = 8, drafts of noise 0.1 / 0.7 / 1.5, against the small-batch kernel (as it is) and the flow kernel:
//   Algorithm 2, B = 8 (35 MB): 42 / 41 / 39 us against 38 / 31 / 27 (small-batch); 12: 44 / 44 / 42 against 58 / 45 / 38; 14: 45 / 46 / 43
//   against 60 / 47 / 40; 16: 49 / 48 / 45 against 60 / 48 / 40; in 32 bits 8 (70 MB): 50 / 48 / 46 against 46 / 35 / 32, 10: 57 / 51 / 49
//   against 67 / 51 / 45 (the line was drawn for 16 bits and for a small-batch kernel with two barriers: it could lie 15 MB lower there, and higher here);
//   33: 65 / 62 / 60 against 86 / 80 / 77 (flow); 128: 144 / 145 / 136 against 168 / 154 / 140; 200 (874 MB): 202 / 208 / 194
//   against 230 / 218 / 195; the 2.2 GB of B = 256, V = 256000: 432 against 416 (the flow kernel overlaps the two sweeps)
//   supplied normalisers, noise 0.7, B = 8 / 10 / 12 / 16 (small-batch): 43 / 44 / 43 / 46 us against 31 / 44 / 41 / 50, 0.1: 44 / 47 / 43 / 46
//   against 40 / 58 / 54 / 63; 33 / 128 / 256 (flow): 52 / 101 / 164 against 67 / 121 / 184
//   Algorithm 1, noise 0.7, B = 12 / 16 / 18 / 24 (small-batch): 40 / 42 / 44 / 49 us against 35 / 35 / 49 / 53; 33 / 64 / 128 (flow): 57 / 82 / 132
//   against 77 / 90 / 115 (it reads all rows, the flow kernel the ones the tests need)
//   probabilities, noise 0.7, B = 33 / 128 / 256 (flow): 31 / 49 / 72 us against 39 / 65 / 120
// The upper ends are lower for 32-bit logits, of which the flow kernel streams the more (half the arithmetic a byte; V = 256000,
// gamma = 2, 312 MB: 103 us against 100; Algorithm 1, 296 MB: 81 against 73), and the one of Algorithm 1 is where a draft that
// is hardly accepted leaves the flow kernel an eighth of the rows to read (23 sequences, noise 3, 238 MB: 53 us against 46).
// On probabilities Algorithm 1 sweeps one row pair a sequence: 33 MB of them 1.2 times faster, 129 MB 51 us against 44;
// Algorithm 2 at 131 MB 72 us against 120.
constexpr long long kPhaseBytes[3][2] = {{72LL << 20, 180LL << 20}, {64LL << 20, 860LL << 20}, {48LL << 20, 1400LL << 20}};
constexpr long long kPhaseBytesF32[3] = {120LL << 20, 280LL << 20, 280LL << 20};
constexpr long long kPhaseProbsPairs[2] = {36LL << 20, 140LL << 20}, kPhaseProbsPairsF32[2] = {24LL << 20, 110LL << 20};   // [algo] bytes of one row pair of every sequence
// (Fewer sequences than this: small-batch kernel.  One line for rows of any length and any gamma, noise 0.1 / 0.7, us against the phase
// kernel's: V = 8192, gamma = 4, B = 12 15 / 14 against 23 / 22, 32 20 / 19 against 23 / 23; gamma = 8, 16 17 / 17 against 25 / 23, 24 27 / 21 against 25 / 24;
// V = 32768, gamma = 8, 16 23 / 19 against 27 / 24, 24 36 / 27 against 28 / 26; V = 128256, gamma = 8, 12 37 / 26 against 26 / 27, 16 40 / 29 against 30 / 29, 24 63 / 40
// against 32 / 29; Algorithm 1, gamma = 8, V = 128256, 16 17 / 19 against 23 / 23, 32 24 / 26 against 25 / 25.)
constexpr int kPhaseProbsB = 17;
// On probabilities, Algorithm 1 on more sequences than SMs: 256 of V = 32768 (34 MB of pairs) takes 1.09 times as long as in the
// flow kernel, 250 of V = 8192 in 32 bits (16 MB) 1.19, 256 of V = 8192 in 16 (8 MB) as long.  Algorithm 2 with many positions:
// gamma = 16, noise 0.1 / 1, B = 17 of V = 8192: 34 against 30 / 25 against 27 us (flow); of V = 32768: even / 1.29 times faster;
// gamma = 64, B = 40 of V = 8192: 71 against 49.
constexpr long long kPhaseProbsMany = 12LL << 20, kPhaseProbsRow = 60000;
// Fewer sequences than this leave the phase kernel with rows in many pieces: V = 152064, gamma = 8, 32-bit logits with supplied
// normalisers, B = 6 (62 MB) 53 / 50 / 46 us against 47 / 38 / 35 in the small-batch kernel, 7 50 / 50 / 47 against 54 / 39 / 36, without 52 / 52 / 49 against 51 / 37 / 34;
// B = 10 (bf16, V = 128256, 44 MB) 47 / 44 / 42 against 58 / 44 / 39;
// beyond its sizes V = 256000, 32-bit, gamma = 16, B = 3 (101 MB) 93 / 83 us (noise 0.1 / 1) against 75 / 66 (flow).  Algorithm 1, whose tests
// the small-batch kernel makes as fast for any outcome: V = 256000, gamma = 8 (bf16), B = 10 (87 MB) 50 / 47 / 47 us (noise 0.1 / 0.7 / 3) against
// 49 / 49 / 50; V = 152064, gamma = 12, B = 10 44 / 42 / 42 against 38 / 39 / 39, 12 47 / 45 / 45 against 52 / 52 / 52.
constexpr int kPhaseFew = 8, kPhaseFewTv = 12;
constexpr long long kPhaseFewRow = 700000;
// With every position swept (diagnostic outputs): bytes of logits, for gamma below 12 and from there on, and bytes of one
// sequence's target rows, [32-bit logits].  bf16, against the flow kernel: V = 256000 gamma = 8, B = 40 (348 MB) 166 against 148 us;
// gamma = 4, B = 24 85 against 89; V = 152064 gamma = 16, B = 24 (241 MB) 141 against 125; V = 65536 gamma = 16, B = 64 1.05 times
// faster.  32-bit: V = 152064 gamma = 4, B = 24 (131 MB) 0.88 times as fast; V = 32768 gamma = 4, B = 128 (151 MB) 1.07, gamma = 8 0.93
// (285 MB); gamma = 12, V = 8192, B = 128 (105 MB) 0.95, B = 64 1.11.  Against the small-batch kernel: V = 152064 gamma = 8, B = 16
// (bf16, 83 MB) 76 against 68 us; gamma = 4, B = 24 64 against 67, 32 69 against 88.
constexpr long long kPhaseAllBytes[2] = {360LL << 20, 144LL << 20}, kPhaseAllBytesLong[2] = {360LL << 20, 60LL << 20};
constexpr long long kPhaseAllRows[2] = {2500000, 2200000}, kPhaseAllSmall = 1300000;
constexpr size_t kSlotHead = 16384;   // first area of a stream's workspace: status word, barrier words, the phase kernel's counters
constexpr size_t kSlotPhase = 256, kSlotSmall = 8192;    // ... the phase kernel's from here on, the small-batch kernel's counters of its sequences
static_assert(kSlotPhase + bv::kPhaseCounterWords * sizeof(unsigned) <= kSlotSmall && kSlotSmall + bv::kSmallMaxB * sizeof(unsigned) <= kSlotHead, "the counters fit in the head");
constexpr int kStreamSlots = 32;  // streams per device that keep a workspace of their own

// Tuning and test options (bv_set_option); their first values come from the environment, read once.
struct Options {
    int kernel = 0;        // 0: chosen by shape; 1 flow, 2 cluster, 3 stream, 4 small-batch, 5 phase
    int loop = 0;          // the decoding loop: 0 by shape, 1 in one kernel wherever two rows fit in shared memory, 2 in two launches an iteration
    int small_bytes = 0;   // logit bytes (in MB) up to which the small-batch kernel is chosen; 0: the built-in limit
    int cluster = 0;       // cluster width of the cluster / stream kernels (1, 2, 4, 8); 0: chosen by shape
    int max_clusters = 0;  // cap on the clusters launched; 0: none
    int flow_chunks = 0, flow_pieces = 0, flow_ctas = 0, flow_depth = 0;   // 0: chosen by shape
    int flow_fine = 0;     // > 0: this many blocks at the end of the batch have their rows cut into the finer chunks
    int flow_keep_l2 = 0;  // 1: the lines of a first sweep stay in L2 at normal priority; 0: every load streams past L2
    int wait_limit = 0;    // polls after which a bounded device-side wait gives up; 0: the built-in limits
    int never_signal = 0;  // test switch: 1 the kernels' workers never report what they have swept; 2 only the phase kernel's second sweeps
};
Options g_opt;
std::once_flag g_opt_once;

int env_int(const char* name) {
    const char* v = std::getenv(name);
    return v ? std::atoi(v) : 0;
}
int kernel_code(const char* v) {
    if (!v) return 0;
    if (!std::strcmp(v, "flow")) return 1;
    if (!std::strcmp(v, "cluster")) return 2;
    if (!std::strcmp(v, "stream")) return 3;
    if (!std::strcmp(v, "small")) return 4;
    if (!std::strcmp(v, "phase")) return 5;
    return 0;
}
void load_env_options() {
    g_opt.kernel = kernel_code(std::getenv("BV_KERNEL"));
    g_opt.cluster = env_int("BV_CLUSTER");
    g_opt.max_clusters = env_int("BV_MAX_CLUSTERS");
    g_opt.flow_chunks = env_int("BV_FLOW_CHUNKS");
    g_opt.flow_pieces = env_int("BV_FLOW_PIECES");
    g_opt.flow_ctas = env_int("BV_FLOW_CTAS");
    g_opt.flow_depth = env_int("BV_FLOW_DEPTH");
}

// The workspace a stream's calls share.  Calls on one stream run one after the other, and the kernels
// leave their counters at zero, so one set of areas per stream serves any number of calls in flight.
// What has to be zero when a kernel starts lies apart from what kernels write as they like: a call that
// a graph replays comes between others without the library knowing, and finds its counters at zero all
// the same.  For the same reason an area that is outgrown stays allocated until the workspace is given
// back (each is at least twice the size of the one before, so they add up to less than the last one).
struct Area {
    char* p = nullptr;
    size_t bytes = 0;
};
struct StreamSlot {
    cudaStream_t stream = nullptr;
    bool used = false;
    Area head;                 // kSlotHead bytes, zero between calls but for the status word
    Area zeros;                // the flow kernel's counters and flags, zero between calls
    Area scratch;              // anything
    std::vector<char*> outgrown;
    unsigned long long stamp = 0;
};

struct DeviceState {
    bool ready = false;
    int sm_count = 0;
    int cc_major = 0;
    unsigned int* tickets = nullptr;  // [kTicketSlots][2], zero when idle
    unsigned long long calls = 0;
    int max_clusters[2][2][2][bv::kMaxCluster + 1] = {};  // [algo][dtype][vec][cluster], 0 = not asked yet
    int clu_clusters[2][2][bv::kMaxCluster + 1] = {};     // cluster kernel: [algo][dtype][cluster]
    StreamSlot slots[kStreamSlots];
    unsigned long long clock = 0;
    int flow_ctas_per_sm[2] = {};
    int small_ctas[2] = {};            // small-batch kernel: CTAs of a launch per dtype (0: not asked yet)
    int phase_ctas[2] = {};            // the phase kernel's
    // staging for the host-buffer entry points, on the device and, for what is small, in pinned host memory
    void* stage = nullptr;
    size_t stage_bytes = 0;
    char* pinned = nullptr;
    size_t pinned_bytes = 0;
    cudaStream_t stream = nullptr;     // theirs, and where memory is obtained while a caller's stream is captured
};

DeviceState g_dev[kMaxDevices];
std::mutex g_mu;
// Held for the whole of a call on host buffers: a device's calls share its staging areas and stream.  (One each, taken before g_mu:
// calls on different devices run side by side.)
std::mutex g_host_mu[kMaxDevices];

thread_local int t_last_launches = 0;
thread_local int t_last_kernel = 0;     // which kernel the last verification call on this thread launched (the "kernel" option's codes)
thread_local int t_last_cuda_error = 0;

int cuda_fail(cudaError_t e) { return bv::note_cuda_error(e); }

// Per-device set-up on first use: device attributes and the ticket slots.
int device_state(DeviceState** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    if (dev < 0 || dev >= kMaxDevices) return BV_ERR_UNSUPPORTED;
    DeviceState& d = g_dev[dev];
    if (!d.ready) {
        if ((e = cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
            return cuda_fail(e);
        if ((e = cudaDeviceGetAttribute(&d.cc_major, cudaDevAttrComputeCapabilityMajor, dev)) != cudaSuccess)
            return cuda_fail(e);
        if (d.cc_major < 10) return BV_ERR_UNSUPPORTED;
        if ((e = cudaMalloc(&d.tickets, sizeof(unsigned int) * 2 * kTicketSlots)) != cudaSuccess)
            return cuda_fail(e);
        if ((e = cudaMemset(d.tickets, 0, sizeof(unsigned int) * 2 * kTicketSlots)) != cudaSuccess)
            return cuda_fail(e);
        d.ready = true;
    }
    *out = &d;
    return BV_OK;
}

int own_stream(DeviceState& d) {
    const cudaError_t e = d.stream ? cudaSuccess : cudaStreamCreateWithFlags(&d.stream, cudaStreamNonBlocking);
    return e == cudaSuccess ? BV_OK : cuda_fail(e);
}

// `want` bytes on `stream` (or `need`, if there are not as many), set to zero if `zero`.
cudaError_t obtain(Area* a, size_t want, size_t need, bool zero, cudaStream_t stream) {
    void* p = nullptr;
    cudaError_t e = cudaMallocAsync(&p, want, stream);
    if (e == cudaErrorMemoryAllocation && want > need) {
        cudaGetLastError();
        e = cudaMallocAsync(&p, want = need, stream);
    }
    if (e != cudaSuccess) return e;
    if (zero && (e = cudaMemsetAsync(p, 0, want, stream)) != cudaSuccess) {
        cudaFreeAsync(p, stream);
        return e;
    }
    a->p = static_cast<char*>(p);
    a->bytes = want;
    return e;
}
// Makes room for `need` bytes in one of the areas of `s`.
int grow(DeviceState& d, StreamSlot& s, Area* a, size_t need, bool zero) {
    if (a->bytes >= need) return BV_OK;
    const size_t want = need > 2 * a->bytes ? need : 2 * a->bytes;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(s.stream, &cap);
    if (e != cudaSuccess) return cuda_fail(e);
    Area fresh;
    if (cap == cudaStreamCaptureStatusNone) {
        e = obtain(&fresh, want, need, zero, s.stream);
    } else {
        // What is allocated on a stream that is captured belongs to the graph: it is obtained on another one, and there
        // before the graph can run.
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        if ((e = cudaThreadExchangeStreamCaptureMode(&mode)) != cudaSuccess) return cuda_fail(e);
        const int rc = own_stream(d);
        if (rc == BV_OK && (e = obtain(&fresh, want, need, zero, d.stream)) == cudaSuccess) e = cudaStreamSynchronize(d.stream);
        cudaThreadExchangeStreamCaptureMode(&mode);
        if (rc != BV_OK) return rc;
    }
    if (e != cudaSuccess) return cuda_fail(e);
    if (a->p) s.outgrown.push_back(a->p);
    *a = fresh;
    return BV_OK;
}

// The workspace of `stream` with room for `zeros` bytes that are zero and `scratch` bytes that are anything.
// A stream seen for the first time takes a free entry, or the one used longest ago (whose areas are
// freed in its own stream's order).
int stream_slot(DeviceState& d, cudaStream_t stream, size_t zeros, size_t scratch, StreamSlot** out) {
    StreamSlot* s = nullptr;
    StreamSlot* victim = nullptr;
    for (StreamSlot& c : d.slots) {
        if (c.used && c.stream == stream) { s = &c; break; }
        if (!victim || (victim->used && (!c.used || c.stamp < victim->stamp))) victim = &c;
    }
    if (!s) {
        s = victim;
        if (s->used) {
            cudaError_t e = cudaSuccess;
            for (char* p : s->outgrown) if (e == cudaSuccess) e = cudaFreeAsync(p, s->stream);
            for (const Area* a : {&s->head, &s->zeros, &s->scratch}) if (e == cudaSuccess && a->p) e = cudaFreeAsync(a->p, s->stream);
            *s = StreamSlot{};
            if (e != cudaSuccess) return cuda_fail(e);
        }
        s->used = true;
        s->stream = stream;
    }
    s->stamp = ++d.clock;
    int rc = grow(d, *s, &s->head, kSlotHead, true);
    if (rc == BV_OK) rc = grow(d, *s, &s->zeros, zeros, true);
    if (rc == BV_OK) rc = grow(d, *s, &s->scratch, scratch, false);
    *out = s;
    return rc;
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Cluster width for the streaming kernel: wide enough that a CTA's slice of a row
// is at most 64 KB, widened further while the batch alone cannot fill the SMs.
int pick_cluster(const DeviceState& d, const Options& opt, int B, size_t row_bytes) {
    if (opt.cluster == 1 || opt.cluster == 2 || opt.cluster == 4 || opt.cluster == 8) return opt.cluster;
    int c = 1;
    while (c < bv::kMaxCluster && row_bytes / c > (64u << 10)) c *= 2;
    while (c < bv::kMaxCluster && static_cast<long long>(B) * c < d.sm_count && row_bytes / (2 * c) >= (8u << 10))
        c *= 2;
    // With several sequences per cluster to go through, narrower clusters (more sequences at a time,
    // cheaper exchanges) win: measured 0.43 against 0.57 ms at B = 256, gamma = 8, V = 152064.
    if (c == 8 && static_cast<long long>(B) * c >= 8LL * d.sm_count) c = 4;
    return c;
}

// Did a kernel that needs a CTA on every SM at once find fewer (a process that is given a part of the GPU)?  The kernels
// that need no such thing take the call.
bool not_all_sms(cudaError_t e) {
    if (e != cudaErrorCooperativeLaunchTooLarge) return false;
    cudaGetLastError();
    return true;
}

// Where the element-wise kernel is the default for rows that are not whole 16-byte vectors: a few short ones a sequence, whose
// dependent steps cost less than the phase kernel's waits for the whole batch.  What a step costs it depends on the part of a
// row, in elements, that one CTA of a sequence's cluster goes through, and on whether all sequences are at work at once.
// Measured, bf16, time over the phase kernel's:
//   Algorithm 1, drafts of noise 0.3 / 1 / 3, all at once, 1000 to 4100 a CTA: gamma = 1 (B = 33 .. 148) 0.50 / 0.49 / 0.48 to 0.67,
//   3: 0.68 to 0.82, 5: 0.96 / 1.01 / 0.78, 6: 1.10 / 1.09 / 0.83; 8200 (B = 148): gamma = 1 0.70, 3: 0.99 / 0.97 / 0.93,
//   4: 1.12 / 1.11 / 1.03; two rounds of sequences (B = 200): gamma = 1 0.84 / 0.82 / 0.79, 2: 0.91 / 0.80 / 0.76 (2050), 1.07 / 0.93 / 0.87 (4100)
//   Algorithm 2, all at once: gamma = 1 0.55 to 0.70 (1000 to 4100), 0.92 (8200); 2: 0.74 to 0.93 (1000 to 4100); 3: 0.90 to 0.99
//   (1000 to 2050), 1.11 (4100); two rounds: 0.90 to 1.15
// and 32-bit logits, B = 148, 8200 elements a CTA, Algorithm 1: gamma = 1 0.69, 2: 0.86, 3: 0.98 / - / 0.92; two rounds (B = 40, 2050) 2: 0.89 /
// 0.80 / 0.81; Algorithm 2: gamma = 1 0.90.
// Drafts that are hardly accepted at all, which Algorithm 1 leaves after a row, are up to a third faster here at any gamma, the
// others up to seven times slower: the lines lie where the three noises together are even.  Against the small-batch kernel:
//   Algorithm 1, B = 32: V = 1003 gamma = 1 0.85 / 0.82 / 0.76, 2: 0.82 / 0.82 / 0.78; V = 4099 0.95 / 0.93 / 0.91, 1.02 / 1.01 / 0.96; V = 16421
//   0.99 / 0.98 / 0.92, 0.99 / 0.96 / 0.85; V = 8209 in 32 bits, gamma = 1, 0.93 / 0.91 / 0.90;  B = 24: V = 16421 0.97 / 0.96 / 0.91, 1.18 / 1.14 / 1.01
bool elements_pay(int algo, const bv::Params& prm, const DeviceState& d, const Options& opt, size_t row_bytes) {
    const int g = prm.gamma;
    if (bv::small_fits(prm.B, g)) return algo == bv::kTokenVerify && g <= 2 && (row_bytes <= 4200 || (prm.B >= 24 && row_bytes > 16500 && row_bytes <= 33000));
    const int cluster = pick_cluster(d, opt, prm.B, row_bytes);
    const int part = prm.V / cluster;
    const long long ctas = static_cast<long long>(prm.B) * cluster;
    if (algo == bv::kTokenVerify) {
        if (ctas <= d.sm_count) return g <= (part <= 4250 ? 5 : part <= 8250 ? 3 : 0);
        return ctas <= 2LL * d.sm_count && prm.V <= 16500 && g <= (part <= 2100 ? 2 : part <= 4250 ? 1 : 0);
    }
    return ctas <= d.sm_count && g <= (part <= 2100 ? 3 : part <= 4250 ? 2 : part <= 8250 ? 1 : 0);
}

// Where the phase kernel is the default.  (Rows that are not whole 16-byte vectors: wherever the kernels above and below are not.)
bool phase_pays(int algo, const bv::Params& prm, const Options& opt, const DeviceState& d, int dtype, bool vec, long long logit_bytes) {
    const bool small = bv::small_fits(prm.B, prm.gamma), f32 = dtype == BV_DTYPE_F32;
    const int a = algo == bv::kBlockVerify ? 1 : 0;
    const long long one_row = logit_bytes / (2 * prm.gamma + 1);      // of every sequence
    if (prm.probs) {
        if (small && prm.B < kPhaseProbsB) return false;
        if (a == 0) return 2 * one_row <= (prm.B > d.sm_count ? kPhaseProbsMany : f32 ? kPhaseProbsPairsF32[a] : kPhaseProbsPairs[a]);
        // (few short rows with many candidates each: the ends of sequences, one candidate after the other)
        if (prm.gamma >= 14 && prm.B < 48 && one_row < prm.gamma * kPhaseProbsRow) return false;
        return 2 * one_row <= (f32 ? kPhaseProbsPairsF32[a] : kPhaseProbsPairs[a]);
    }
    const int which = a == 0 ? 0 : (prm.lse_d != nullptr ? 2 : 1);
    if (prm.first != nullptr) return !bv::small_takes_tables(algo, prm.lse_d != nullptr, prm.B, prm.gamma, static_cast<size_t>(one_row / prm.B));      // (no other kernel takes larger ones)
    const long long small_limit = opt.small_bytes > 0 ? static_cast<long long>(opt.small_bytes) << 20 : kSmallBytes[a];
    if (small && prm.B < kPhaseFew && logit_bytes <= small_limit) return false;
    if (vec && f32 && prm.B < kPhaseFew && one_row / prm.B > kPhaseFewRow) return false;
    if (small && a == 0 && prm.B < kPhaseFewTv && prm.gamma <= 8 && logit_bytes <= small_limit) return false;
    if (vec && (prm.out_p || prm.out_S || prm.out_h || prm.out_lse_t || prm.out_lse_d)) {
        // (every position is swept, and the flow kernel overlaps its two sweeps)
        const long long positions = one_row / prm.B * prm.gamma;                          // bytes of a sequence's target rows
        if (positions > (small && logit_bytes <= small_limit ? kPhaseAllSmall : kPhaseAllRows[f32]) ||
            logit_bytes > (prm.gamma < 12 ? kPhaseAllBytes[f32] : kPhaseAllBytesLong[f32])) return false;
    }
    const long long least = opt.small_bytes > 0 ? small_limit : kPhaseBytes[which][0];
    return (!small || logit_bytes > least) && (!vec || logit_bytes <= (f32 ? kPhaseBytesF32[which] : kPhaseBytes[which][1]));
}

// The phase kernel for the call in `prm`: BV_OK, an error, or 1 if it does not take the call.  Rows at any alignment have no
// other kernel of this speed, so a batch of more sequences than it takes goes through it in parts.
int run_phase(DeviceState& d, const bv::Params& prm, int dtype, bool vec, bool probe, cudaStream_t stream) {
    int& nc = d.phase_ctas[dtype];
    if (nc == 0) {
        nc = bv::phase_max_ctas(dtype, d.sm_count);
        if (nc <= 0) nc = -1;
    }
    if (nc < 0) return 1;
    const int g = prm.gamma;
    int part = prm.B;
    bv::PhasePlan plan = bv::phase_plan(prm.V, dtype, vec, part, g, prm.lse_d != nullptr, nc);
    while (!plan.fits && !vec && part > 1) {
        part = part > bv::kPhaseMaxB ? bv::kPhaseMaxB : part / 2;
        plan = bv::phase_plan(prm.V, dtype, vec, part, g, prm.lse_d != nullptr, nc);
    }
    if (!plan.fits) return 1;
    bv::PhaseScratch ps;
    size_t need = bv::phase_scratch(nullptr, nullptr, part, g, plan, &ps);
    if (prm.B % part != 0) {
        // (the last part is planned for its own size: fewer sequences, but the warps' parts of the list are shorter too, so a
        // row may lie in more pieces and the whole take more)
        const int rest = prm.B % part;
        const size_t n = bv::phase_scratch(nullptr, nullptr, rest, g, bv::phase_plan(prm.V, dtype, vec, rest, g, prm.lse_d != nullptr, nc), &ps);
        if (n > need) need = n;
    }
    StreamSlot* slot = nullptr;
    const int rc = stream_slot(d, stream, 0, need, &slot);
    if (rc != BV_OK || probe) return rc;
    const size_t row_bytes = static_cast<size_t>(prm.V) * (dtype == BV_DTYPE_F32 ? 4 : 2);
    int launches = 0;
    for (int b0 = 0; b0 < prm.B; b0 += part, ++launches) {
        bv::Params p = prm;
        const size_t b = static_cast<size_t>(b0);
        p.B = prm.B - b0 < part ? prm.B - b0 : part;
        p.tgt = static_cast<const char*>(prm.tgt) + b * (g + 1) * row_bytes;
        p.drf = static_cast<const char*>(prm.drf) + b * g * row_bytes;
        p.tok = prm.tok + b * g;
        p.uni = prm.uni + b * (g + 2);
        if (prm.lse_d) p.lse_d = prm.lse_d + b * g;
        p.out_tokens = prm.out_tokens + b * (g + 1);
        p.out_len = prm.out_len + b;
        if (prm.out_p) p.out_p = prm.out_p + b * (g + 1);
        if (prm.out_S) p.out_S = prm.out_S + b * g;
        if (prm.out_h) p.out_h = prm.out_h + b * (g + 1);
        if (prm.out_lse_t) p.out_lse_t = prm.out_lse_t + b * (g + 1);
        if (prm.out_lse_d) p.out_lse_d = prm.out_lse_d + b * g;
        if (p.status == nullptr) p.status = reinterpret_cast<int*>(slot->head.p);
        if (p.B != part) plan = bv::phase_plan(p.V, dtype, vec, p.B, g, p.lse_d != nullptr, nc);
        bv::phase_scratch(slot->scratch.p, reinterpret_cast<unsigned*>(slot->head.p + kSlotPhase), p.B, g, plan, &ps);
        const cudaError_t e = bv::launch_phase(p, ps, dtype, vec, nc, stream);
        if (launches == 0 && not_all_sms(e)) return 1;
        if (e != cudaSuccess) return cuda_fail(e);
    }
    t_last_launches = launches; t_last_kernel = 5;
    return BV_OK;
}

struct Extra {              // what only some entry points pass
    const float* lse_d = nullptr;   // supplied draft log-normalisers (bv_verify_lse)
    int greedy = 0;                 // Algorithm 4 instead of Algorithm 2 (gbv_verify)
    const int32_t* first = nullptr; // the rows are those of two tables (Params::first)
    int* status = nullptr;          // where a wait that gives up is recorded (null: the stream's status word)
    bool probe = false;             // find the kernel and its workspace, launch nothing
    int probs = 0;                  // the rows hold probabilities, not logits (bv_verify_probs, tv_verify_probs)
    float* out_p = nullptr; float* out_S = nullptr; float* out_h = nullptr;
    float* out_lse_t = nullptr; float* out_lse_d = nullptr;
};

int run_device(int algo, const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B,
               int gamma, int V, int dtype, float T, int32_t* ot, int32_t* ol, const Extra& ex, cudaStream_t stream) {
    t_last_launches = 0;
    t_last_kernel = 0;
    int rc = bv::check_verify_args(tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol);
    if (rc != BV_OK) return rc;
    if (B == 0) return BV_OK;
    std::call_once(g_opt_once, load_env_options);

    std::lock_guard<std::mutex> lock(g_mu);
    const Options opt = g_opt;
    DeviceState* d = nullptr;
    if ((rc = device_state(&d)) != BV_OK) return rc;

    const size_t esz = dtype == BV_DTYPE_F32 ? 4 : 2;
    const size_t row_bytes = static_cast<size_t>(V) * esz;
    const bool vec = (row_bytes % 16 == 0) && aligned(tgt, 16) && aligned(drf, 16);

    bv::Params prm{};
    prm.tgt = tgt; prm.drf = drf; prm.tok = tok; prm.uni = uni;
    prm.lse_d = ex.lse_d;
    prm.greedy = ex.greedy;
    prm.probs = ex.probs;
    prm.first = ex.first;
    prm.B = B; prm.gamma = gamma; prm.V = V;
    const double kd = 1.4426950408889634073599246810019 / static_cast<double>(T);
    prm.kd = kd;
    prm.kf = static_cast<float>(kd);
    prm.out_tokens = ot; prm.out_len = ol;
    prm.out_p = ex.out_p; prm.out_S = ex.out_S; prm.out_h = ex.out_h;
    prm.out_lse_t = ex.out_lse_t; prm.out_lse_d = ex.out_lse_d;
    prm.wait_limit = opt.wait_limit > 0 ? static_cast<unsigned>(opt.wait_limit) : 0u;
    prm.never_signal = opt.never_signal;
    prm.status = ex.status;

    prm.algo = algo;
    const long long logit_bytes = static_cast<long long>(B) * (2 * gamma + 1) * static_cast<long long>(row_bytes);
    const bool flow_ok = vec && (opt.kernel == 0 || opt.kernel == 1);

    // Both sweeps split over all warps, with the folds between them: between the small-batch kernel's sizes and the flow
    // kernel's, and for rows at any alignment.
    const bool only_vec = prm.lse_d != nullptr || prm.greedy || prm.probs;      // (entry points without an element-wise path)
    if (prm.first != nullptr && !vec) return BV_ERR_UNSUPPORTED;
    const bool elements = !vec && !only_vec && opt.kernel == 0 && elements_pay(algo, prm, *d, opt, row_bytes);
    if ((vec || !only_vec) && !elements && (opt.kernel == 5 || ((opt.kernel == 0 || prm.first != nullptr) && phase_pays(algo, prm, opt, *d, dtype, vec, logit_bytes)))) {
        if ((rc = run_phase(*d, prm, dtype, vec, ex.probe, stream)) <= BV_OK) return rc;
    }

    // A few sequences whose logits fit in L2: the launch is a matter of latency, and the kernel with one grid-wide
    // barrier (none on probabilities) instead of queues takes half the time of the flow kernel or less.
    const long long small_limit = opt.small_bytes > 0 ? static_cast<long long>(opt.small_bytes) << 20 : kSmallBytes[algo == bv::kBlockVerify ? 1 : 0];
    // (given probabilities only a few row pairs per sequence are read whatever the size of the rest: kPhaseProbsB)
    if ((vec || !only_vec) && !elements && bv::small_fits(B, gamma) &&
        (opt.kernel == 4 || ((opt.kernel == 0 || prm.first != nullptr) && (prm.probs ? B <= 16 : logit_bytes <= small_limit)))) {
        int& nc = d->small_ctas[dtype];
        if (nc == 0) {
            nc = bv::small_max_ctas(dtype, d->sm_count);
            if (nc <= 0) nc = -1;
        }
        // (a row that starts inside a vector lies in one more)
        const long long vecs = vec ? static_cast<long long>(row_bytes / 16) : (static_cast<long long>(row_bytes) + 30) / 16;
        const bv::SmallPlan plan = bv::small_plan(vecs, B, gamma, nc > 0 ? nc : 1);
        if (nc > 0 && (vec || V <= (1 << 30))) {
            StreamSlot* slot = nullptr;
            rc = stream_slot(*d, stream, 0, bv::small_scratch_bytes(B, gamma, plan), &slot);
            if (rc != BV_OK || ex.probe) return rc;
            bv::SmallScratch sc;
            // the barrier words are in the head: zero since it was allocated
            bv::small_scratch_layout(slot->scratch.p, reinterpret_cast<unsigned*>(slot->head.p + 128), reinterpret_cast<unsigned*>(slot->head.p + kSlotSmall),
                                     B, gamma, plan, &sc);
            prm.ticket = nullptr;
            prm.nclusters = 0;
            prm.status = ex.status ? ex.status : reinterpret_cast<int*>(slot->head.p);
            const cudaError_t e = bv::launch_small(prm, sc, dtype, vec, nc, stream);
            if (e == cudaSuccess) {
                t_last_launches = 1; t_last_kernel = 4;
                return BV_OK;
            }
            if (!not_all_sms(e)) return cuda_fail(e);
        }
    }

    if (prm.first != nullptr) return BV_ERR_UNSUPPORTED;      // (the kernels below take whole tensors)
    // (only the kernels above and below serve these entry points)
    if ((prm.lse_d != nullptr || prm.greedy || prm.probs) && !flow_ok) return BV_ERR_UNSUPPORTED;

    // 16-byte rows: the flow of independent work items (both algorithms)
    if (flow_ok) {
        int& per_sm = d->flow_ctas_per_sm[dtype];
        if (per_sm == 0) {
            per_sm = bv::flow_max_ctas_per_sm(dtype);
            if (per_sm <= 0) per_sm = -1;
        }
        if (per_sm > 0) {
            const long long units = static_cast<long long>(row_bytes / 16);
            long long nctas = static_cast<long long>(d->sm_count) * per_sm;
            if (opt.flow_ctas >= 1 && opt.flow_ctas < nctas) nctas = opt.flow_ctas;
            const int chunks = (opt.flow_chunks >= 1 && opt.flow_chunks <= bv::kFlowMaxChunks) ? opt.flow_chunks : 0;
            const int pieces = (opt.flow_pieces >= 1 && opt.flow_pieces <= 8) ? opt.flow_pieces : 0;
            // (with supplied draft normalisers a first-sweep item streams one row, not two)
            bv::FlowPlan plan = bv::flow_plan(units, B, gamma, nctas, prm.lse_d == nullptr, chunks, pieces, algo == bv::kTokenVerify, prm.probs != 0);
            if (opt.flow_fine > 0 && algo != bv::kTokenVerify && !prm.probs && plan.nch_late > plan.nch) plan.fine_from = opt.flow_fine < B ? B - opt.flow_fine : 0;
            size_t zero_bytes = 0;
            const size_t need = bv::flow_scratch_bytes(B, gamma, plan, &zero_bytes);
            StreamSlot* slot = nullptr;
            if ((rc = stream_slot(*d, stream, zero_bytes, need, &slot)) != BV_OK) return rc;
            bv::FlowScratch fl;
            bv::flow_scratch_layout(slot->zeros.p, slot->scratch.p, B, gamma, plan, &fl);
            // (with every position swept the second sweeps are the larger half of the launch and never wait for one another: deeper measured better)
            if (prm.out_p || prm.out_S || prm.out_h || prm.out_lse_t || prm.out_lse_d) fl.depth = 3;
            if (opt.flow_depth >= 2 && opt.flow_depth <= 6) fl.depth = opt.flow_depth;
            fl.keep_l2 = opt.flow_keep_l2 == 1;
            // (the kernel leaves its counters and flags at zero when it ends: they have been since their area was obtained)
            // (given probabilities the items are the pieces of the positions swept: at most all of them)
            long long items = prm.probs ? static_cast<long long>(B) * (gamma + 1) * fl.np : static_cast<long long>(fl.total_s1);
            if (nctas > items) nctas = items;
            prm.ticket = nullptr;
            prm.nclusters = 0;
            prm.status = ex.status ? ex.status : reinterpret_cast<int*>(slot->head.p);
            const cudaError_t e = bv::launch_flow(prm, fl, dtype, static_cast<int>(nctas), stream);
            if (e != cudaSuccess) return cuda_fail(e);
            t_last_launches = 1; t_last_kernel = 1;
            return BV_OK;
        }
    }

    if (prm.lse_d != nullptr || prm.greedy || prm.probs) return BV_ERR_UNSUPPORTED;   // (the flow kernel could not be launched)

    StreamSlot* slot = nullptr;
    if ((rc = stream_slot(*d, stream, 0, 0, &slot)) != BV_OK) return rc;
    prm.status = ex.status ? ex.status : reinterpret_cast<int*>(slot->head.p);

    int cluster = pick_cluster(*d, opt, B, row_bytes);
    if (vec && opt.kernel != 3) {
        int& cc = d->clu_clusters[algo][dtype][cluster];
        if (cc == 0) {
            cc = bv::cluster_max_clusters(algo, dtype, cluster);
            if (cc <= 0) cc = -1;
        }
        if (cc > 0) {
            int n = B < cc ? B : cc;
            if (opt.max_clusters > 0 && opt.max_clusters < n) n = opt.max_clusters;
            prm.ticket = d->tickets + 2 * (d->calls++ % kTicketSlots);
            prm.nclusters = n;
            cudaError_t e = bv::launch_cluster(prm, algo, dtype, cluster, n, stream);
            if (e != cudaSuccess) return cuda_fail(e);
            t_last_launches = 1; t_last_kernel = 2;
            return BV_OK;
        }
    }
    int& cached = d->max_clusters[algo][dtype][vec ? 1 : 0][cluster];
    if (cached == 0) {
        cached = bv::stream_max_clusters(algo, dtype, vec, cluster);
        if (cached <= 0) cached = -1;
    }
    if (cached < 0) return BV_ERR_UNSUPPORTED;
    const int nclusters = B < cached ? B : cached;

    prm.ticket = d->tickets + 2 * (d->calls++ % kTicketSlots);
    prm.nclusters = nclusters;

    cudaError_t e = bv::launch_stream(prm, algo, dtype, vec, cluster, nclusters, stream);
    if (e != cudaSuccess) return cuda_fail(e);
    t_last_launches = 1; t_last_kernel = 3;
    return BV_OK;
}

// Reads and clears the status word of `stream`'s workspace; waits for the stream.
int take_stream_status(cudaStream_t stream) {
    int* word = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        DeviceState* d = nullptr;
        const int rc = device_state(&d);
        if (rc != BV_OK) return rc;
        for (StreamSlot& c : d->slots)
            if (c.used && c.stream == stream) word = reinterpret_cast<int*>(c.head.p);
    }
    cudaError_t e;
    if (!word) {
        if ((e = cudaStreamSynchronize(stream)) != cudaSuccess) return cuda_fail(e);
        return BV_OK;
    }
    int status = 0;
    if ((e = cudaMemcpyAsync(&status, word, sizeof(int), cudaMemcpyDeviceToHost, stream)) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMemsetAsync(word, 0, sizeof(int), stream)) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaStreamSynchronize(stream)) != cudaSuccess) return cuda_fail(e);
    return status ? BV_ERR_TIMEOUT : BV_OK;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

int run_host(int algo, const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B,
             int gamma, int V, int dtype, float T, int32_t* ot, int32_t* ol) {
    int rc = bv::check_verify_args(tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol);
    if (rc != BV_OK) return rc;
    if (B == 0) return BV_OK;
    const size_t esz = dtype == BV_DTYPE_F32 ? 4 : 2;
    const size_t n_t = static_cast<size_t>(B) * (gamma + 1) * V * esz;
    const size_t n_d = static_cast<size_t>(B) * gamma * V * esz;
    const size_t n_tok = static_cast<size_t>(B) * gamma * 4, n_uni = static_cast<size_t>(B) * (gamma + 2) * 4;
    const size_t n_ot = static_cast<size_t>(B) * (gamma + 1) * 4, n_ol = static_cast<size_t>(B) * 4;
    // The small arrays travel together, in with the status word behind them and out with it in front: one copy each way beside
    // the two of the logits.  (A copy more costs some 5 us in the stream's order: 8 sequences of gamma = 8, V = 32000 in 32 bits,
    // 17 MB, with seven copies and a memset 391 us a call, 311 of them the logits' on the link.)
    const size_t o_t = 0, o_d = align_up(o_t + n_t, 256), o_in = align_up(o_d + n_d, 256);
    const size_t i_uni = align_up(n_tok, 16), i_status = align_up(i_uni + n_uni, 16), i_ot = i_status + 16, i_ol = align_up(i_ot + n_ot, 16);
    const size_t n_in = i_ot, n_small = i_ol + n_ol, total = o_in + n_small;

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    if (dev < 0 || dev >= kMaxDevices) return BV_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> host_lock(g_host_mu[dev]);
    char* base = nullptr;
    char* pin = nullptr;
    cudaStream_t s = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        DeviceState* d = nullptr;
        if ((rc = device_state(&d)) != BV_OK) return rc;
        if ((rc = own_stream(*d)) != BV_OK) return rc;
        // (this entry point waits for its result anyway, so its staging buffers grow with plain cudaMalloc)
        if (d->stage_bytes < total) {
            if (d->stage) cudaFree(d->stage);
            d->stage = nullptr;
            d->stage_bytes = 0;
            if ((e = cudaMalloc(&d->stage, total)) != cudaSuccess) return cuda_fail(e);
            d->stage_bytes = total;
        }
        if (d->pinned_bytes < n_small) {
            if (d->pinned) cudaFreeHost(d->pinned);
            d->pinned = nullptr;
            d->pinned_bytes = 0;
            if ((e = cudaHostAlloc(reinterpret_cast<void**>(&d->pinned), n_small, cudaHostAllocPortable)) != cudaSuccess) return cuda_fail(e);
            d->pinned_bytes = n_small;
        }
        base = static_cast<char*>(d->stage);
        pin = d->pinned;
        s = d->stream;
    }
    char* const in = base + o_in;
    std::memcpy(pin, tok, n_tok);
    std::memcpy(pin + i_uni, uni, n_uni);
    std::memset(pin + i_status, 0, 16);
    // (whatever fails below, nothing of this call is under way any more when the buffers are let go)
    auto enqueue = [&]() -> int {
        if ((e = cudaMemcpyAsync(in, pin, n_in, cudaMemcpyHostToDevice, s)) != cudaSuccess) return cuda_fail(e);
        if ((e = cudaMemcpyAsync(base + o_t, tgt, n_t, cudaMemcpyHostToDevice, s)) != cudaSuccess) return cuda_fail(e);
        if ((e = cudaMemcpyAsync(base + o_d, drf, n_d, cudaMemcpyHostToDevice, s)) != cudaSuccess) return cuda_fail(e);
        Extra ex;
        ex.status = reinterpret_cast<int*>(in + i_status);
        const int done = run_device(algo, base + o_t, base + o_d, reinterpret_cast<const int32_t*>(in), reinterpret_cast<const float*>(in + i_uni),
                                    B, gamma, V, dtype, T, reinterpret_cast<int32_t*>(in + i_ot), reinterpret_cast<int32_t*>(in + i_ol), ex, s);
        if (done != BV_OK) return done;
        if ((e = cudaMemcpyAsync(pin + i_status, in + i_status, n_small - i_status, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return cuda_fail(e);
        return BV_OK;
    };
    rc = enqueue();
    e = cudaStreamSynchronize(s);
    if (rc != BV_OK) return rc;
    if (e != cudaSuccess) return cuda_fail(e);
    std::memcpy(ot, pin + i_ot, n_ot);
    std::memcpy(ol, pin + i_ol, n_ol);
    int status = 0;
    std::memcpy(&status, pin + i_status, sizeof(int));
    return status ? BV_ERR_TIMEOUT : BV_OK;
}

Extra diagnostics(float* out_p, float* out_S, float* out_h, float* out_lse_t, float* out_lse_d) {
    Extra ex;
    ex.out_p = out_p; ex.out_S = out_S; ex.out_h = out_h; ex.out_lse_t = out_lse_t; ex.out_lse_d = out_lse_d;
    return ex;
}

}  // namespace

namespace bv {

int note_cuda_error(cudaError_t e) {
    t_last_cuda_error = static_cast<int>(e);
    cudaGetLastError();
    return BV_ERR_CUDA;
}
void note_launches(int n) { t_last_launches = n; }
bool small_takes_tables(int algo, bool lse, int B, int gamma, size_t row_bytes) {
    return small_fits(B, gamma) &&
           static_cast<long long>(B) * (2 * gamma + 1) * static_cast<long long>(row_bytes) <= kPhaseBytes[algo != kBlockVerify ? 0 : lse ? 2 : 1][0];
}
int loop_option() {
    std::call_once(g_opt_once, load_env_options);
    std::lock_guard<std::mutex> lock(g_mu);
    return g_opt.loop ? g_opt.loop : g_opt.kernel ? 2 : 0;
}

int run_tables(int algo, const void* tgt_table, const void* drf_table, const int32_t* first, const int32_t* tok, const float* uni,
               const float* lse_d, int B, int gamma, int V, int dtype, float T, int32_t* ot, int32_t* ol, bool probe, cudaStream_t stream) {
    Extra ex;
    ex.lse_d = lse_d;
    ex.first = first;
    ex.probe = probe;
    return run_device(algo, tgt_table, drf_table, tok, uni, B, gamma, V, dtype, T, ot, ol, ex, stream);
}

int check_verify_args(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B, int gamma,
                      int V, int dtype, float T, const int32_t* ot, const int32_t* ol) {
    if (!tgt || !drf || !tok || !uni || !ot || !ol) return BV_ERR_INVALID_ARG;
    if (B < 0 || gamma < 1 || V < 1) return BV_ERR_INVALID_ARG;
    if (!(T > 0.f) || !std::isfinite(T)) return BV_ERR_INVALID_ARG;
    if (dtype != BV_DTYPE_F32 && dtype != BV_DTYPE_BF16) return BV_ERR_INVALID_ARG;
    const size_t esz = dtype == BV_DTYPE_F32 ? 4 : 2;
    if (!aligned(tgt, esz) || !aligned(drf, esz) || !aligned(tok, 4) || !aligned(uni, 4) ||
        !aligned(ot, 4) || !aligned(ol, 4))
        return BV_ERR_INVALID_ARG;
    if (gamma > BV_MAX_GAMMA) return BV_ERR_UNSUPPORTED;
    return BV_OK;
}

}  // namespace bv

extern "C" {

int bv_verify(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B, int gamma,
              int V, int dtype, float T, int32_t* ot, int32_t* ol, void* stream) {
    return run_device(bv::kBlockVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol, Extra{},
                      static_cast<cudaStream_t>(stream));
}

int bv_verify_lse(const void* tgt, const void* drf, const int32_t* tok, const float* uni, const float* draft_lse,
                  int B, int gamma, int V, int dtype, float T, int32_t* ot, int32_t* ol, void* stream) {
    if (!draft_lse) return BV_ERR_INVALID_ARG;
    Extra ex;
    ex.lse_d = draft_lse;
    return run_device(bv::kBlockVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol, ex, static_cast<cudaStream_t>(stream));
}

int bv_verify_lse_ex(const void* tgt, const void* drf, const int32_t* tok, const float* uni, const float* draft_lse,
                     int B, int gamma, int V, int dtype, float T, int32_t* ot, int32_t* ol, float* out_p,
                     float* out_S, float* out_h, float* out_lse_t, float* out_lse_d, void* stream) {
    if (!draft_lse) return BV_ERR_INVALID_ARG;
    Extra ex = diagnostics(out_p, out_S, out_h, out_lse_t, out_lse_d);
    ex.lse_d = draft_lse;
    return run_device(bv::kBlockVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol, ex, static_cast<cudaStream_t>(stream));
}

int tv_verify_lse(const void* tgt, const void* drf, const int32_t* tok, const float* uni, const float* draft_lse,
                  int B, int gamma, int V, int dtype, float T, int32_t* ot, int32_t* ol, void* stream) {
    if (!draft_lse) return BV_ERR_INVALID_ARG;
    Extra ex;
    ex.lse_d = draft_lse;
    return run_device(bv::kTokenVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol, ex, static_cast<cudaStream_t>(stream));
}

int tv_verify_lse_ex(const void* tgt, const void* drf, const int32_t* tok, const float* uni, const float* draft_lse,
                     int B, int gamma, int V, int dtype, float T, int32_t* ot, int32_t* ol, float* out_p,
                     float* out_S, float* out_h, float* out_lse_t, float* out_lse_d, void* stream) {
    if (!draft_lse) return BV_ERR_INVALID_ARG;
    Extra ex = diagnostics(out_p, out_S, out_h, out_lse_t, out_lse_d);
    ex.lse_d = draft_lse;
    return run_device(bv::kTokenVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol, ex, static_cast<cudaStream_t>(stream));
}

int bv_verify_probs(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B, int gamma,
                    int V, int dtype, int32_t* ot, int32_t* ol, float* out_p, float* out_S, float* out_h, void* stream) {
    Extra ex = diagnostics(out_p, out_S, out_h, nullptr, nullptr);
    ex.probs = 1;
    return run_device(bv::kBlockVerify, tgt, drf, tok, uni, B, gamma, V, dtype, 1.f, ot, ol, ex, static_cast<cudaStream_t>(stream));
}

int tv_verify_probs(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B, int gamma,
                    int V, int dtype, int32_t* ot, int32_t* ol, float* out_p, float* out_S, float* out_h, void* stream) {
    Extra ex = diagnostics(out_p, out_S, out_h, nullptr, nullptr);
    ex.probs = 1;
    return run_device(bv::kTokenVerify, tgt, drf, tok, uni, B, gamma, V, dtype, 1.f, ot, ol, ex, static_cast<cudaStream_t>(stream));
}

int gbv_verify(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B, int gamma,
               int V, int dtype, float T, int32_t* ot, int32_t* ol, void* stream) {
    Extra ex;
    ex.greedy = 1;
    return run_device(bv::kBlockVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol, ex, static_cast<cudaStream_t>(stream));
}

int gbv_verify_ex(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B, int gamma,
                  int V, int dtype, float T, int32_t* ot, int32_t* ol, float* out_p, float* out_S,
                  float* out_h, float* out_lse_t, float* out_lse_d, void* stream) {
    Extra ex = diagnostics(out_p, out_S, out_h, out_lse_t, out_lse_d);
    ex.greedy = 1;
    return run_device(bv::kBlockVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol, ex, static_cast<cudaStream_t>(stream));
}

int tv_verify(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B, int gamma,
              int V, int dtype, float T, int32_t* ot, int32_t* ol, void* stream) {
    return run_device(bv::kTokenVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol, Extra{},
                      static_cast<cudaStream_t>(stream));
}

int bv_verify_ex(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B, int gamma,
                 int V, int dtype, float T, int32_t* ot, int32_t* ol, float* out_p, float* out_S,
                 float* out_h, float* out_lse_t, float* out_lse_d, void* stream) {
    return run_device(bv::kBlockVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol,
                      diagnostics(out_p, out_S, out_h, out_lse_t, out_lse_d), static_cast<cudaStream_t>(stream));
}

int tv_verify_ex(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B, int gamma,
                 int V, int dtype, float T, int32_t* ot, int32_t* ol, float* out_p, float* out_S,
                 float* out_h, float* out_lse_t, float* out_lse_d, void* stream) {
    return run_device(bv::kTokenVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol,
                      diagnostics(out_p, out_S, out_h, out_lse_t, out_lse_d), static_cast<cudaStream_t>(stream));
}

int bv_verify_host(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B,
                   int gamma, int V, int dtype, float T, int32_t* ot, int32_t* ol) {
    return run_host(bv::kBlockVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol);
}

int tv_verify_host(const void* tgt, const void* drf, const int32_t* tok, const float* uni, int B,
                   int gamma, int V, int dtype, float T, int32_t* ot, int32_t* ol) {
    return run_host(bv::kTokenVerify, tgt, drf, tok, uni, B, gamma, V, dtype, T, ot, ol);
}

int bv_stream_status(void* stream) { return take_stream_status(static_cast<cudaStream_t>(stream)); }

int bv_set_option(const char* name, int value) {
    if (!name) return BV_ERR_INVALID_ARG;
    std::call_once(g_opt_once, load_env_options);
    std::lock_guard<std::mutex> lock(g_mu);
    if (!std::strcmp(name, "kernel")) g_opt.kernel = value;
    else if (!std::strcmp(name, "loop")) g_opt.loop = value;
    else if (!std::strcmp(name, "small_bytes")) g_opt.small_bytes = value;
    else if (!std::strcmp(name, "cluster")) g_opt.cluster = value;
    else if (!std::strcmp(name, "max_clusters")) g_opt.max_clusters = value;
    else if (!std::strcmp(name, "flow_chunks")) g_opt.flow_chunks = value;
    else if (!std::strcmp(name, "flow_pieces")) g_opt.flow_pieces = value;
    else if (!std::strcmp(name, "flow_ctas")) g_opt.flow_ctas = value;
    else if (!std::strcmp(name, "flow_depth")) g_opt.flow_depth = value;
    else if (!std::strcmp(name, "flow_keep_l2")) g_opt.flow_keep_l2 = value;
    else if (!std::strcmp(name, "flow_fine")) g_opt.flow_fine = value;
    else if (!std::strcmp(name, "wait_limit")) g_opt.wait_limit = value;
    else if (!std::strcmp(name, "never_signal")) g_opt.never_signal = value;
    else return BV_ERR_INVALID_ARG;
    return BV_OK;
}

int bv_release(void) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    if (dev < 0 || dev >= kMaxDevices) return BV_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> host_lock(g_host_mu[dev]);
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState& d = g_dev[dev];
    if ((e = cudaDeviceSynchronize()) != cudaSuccess) return cuda_fail(e);
    if (d.stage) cudaFree(d.stage);
    if (d.pinned) cudaFreeHost(d.pinned);
    if (d.tickets) cudaFree(d.tickets);
    for (StreamSlot& c : d.slots) {
        for (char* p : c.outgrown) cudaFree(p);
        for (const Area* a : {&c.head, &c.zeros, &c.scratch}) if (a->p) cudaFree(a->p);
    }
    if (d.stream) cudaStreamDestroy(d.stream);
    d = DeviceState{};
    return BV_OK;
}

int bv_last_launch_count(void) { return t_last_launches; }
int bv_last_kernel(void) { return t_last_kernel; }
int bv_last_cuda_error(void) { return t_last_cuda_error; }

const char* bv_status_string(int status) {
    switch (status) {
        case BV_OK: return "ok";
        case BV_ERR_INVALID_ARG: return "invalid argument";
        case BV_ERR_UNSUPPORTED: return "unsupported shape or device";
        case BV_ERR_CUDA: return "CUDA runtime error";
        case BV_ERR_TIMEOUT: return "device-side wait timed out";
        case BV_ERR_TOO_LARGE: return "problem needs more scratch than the no-allocation entry point has";
        default: return "unknown status";
    }
}

int bv_version(void) { return 200; }

}  // extern "C"
