// The dispatch layer (bv_api.cu) on a runtime that only keeps books, for tests without a GPU: every allocation is host
// memory of exactly the size asked for, launches check the memory they are handed and leave in it what the kernels leave
// (scratch: anything; counters: zero), and a captured stream records its work for replays.  Plans come from the library itself.
#include <cuda_runtime.h>

#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "bv_flow_common.cuh"

namespace {

struct Block { size_t bytes; bool live; };
std::map<char*, Block> g_blocks;
std::vector<std::vector<std::function<void()>>> g_graphs;
bool g_capturing = false;
cudaStream_t g_captured = nullptr;       // the stream that is captured
int g_refuse_cooperative = 0;
int g_launches = 0;
std::string g_errors;

void complain(const std::string& what) { g_errors += what + "\n"; }
cudaError_t give(void** p, size_t bytes) {
    char* c = static_cast<char*>(std::malloc(bytes));
    std::memset(c, 0xcd, bytes);
    g_blocks[c] = Block{bytes, true};
    *p = c;
    return cudaSuccess;
}
cudaError_t take_back(void* p) {
    auto it = g_blocks.find(static_cast<char*>(p));
    if (it == g_blocks.end() || !it->second.live) complain("free of what is not allocated");
    else it->second.live = false;               // (kept: what still points into it is found out, not crashed on)
    return cudaSuccess;
}
bool inside(const char* what, const void* p, size_t bytes) {
    const char* c = static_cast<const char*>(p);
    auto it = g_blocks.upper_bound(const_cast<char*>(c));
    if (it == g_blocks.begin()) { complain(std::string(what) + ": no allocation"); return false; }
    --it;
    if (c + bytes > it->first + it->second.bytes) { complain(std::string(what) + ": outside its allocation"); return false; }
    if (!it->second.live) { complain(std::string(what) + ": memory was given back"); return false; }
    return true;
}
void scratch(const char* what, void* p, size_t bytes) { if (bytes && inside(what, p, bytes)) std::memset(p, 0xab, bytes); }
void zeros(const char* what, const void* p, size_t bytes) {
    if (!inside(what, p, bytes)) return;
    for (size_t i = 0; i < bytes; ++i)
        if (static_cast<const char*>(p)[i]) { complain(std::string(what) + ": not zero at the launch"); return; }
}
bool captured(cudaStream_t s) { return g_capturing && s == g_captured; }
cudaError_t enqueue(cudaStream_t s, std::function<void()> f) {
    if (captured(s)) g_graphs.back().push_back(f); else f();
    return cudaSuccess;
}

thread_local int t_device = 0;
cudaError_t fake_cudaGetDevice(int* d) { *d = t_device; return cudaSuccess; }
cudaError_t fake_cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 148 : 10;
    return cudaSuccess;
}
cudaError_t fake_cudaMalloc(void** p, size_t n) { return give(p, n); }
template <class T> cudaError_t fake_cudaMalloc(T** p, size_t n) { return give(reinterpret_cast<void**>(p), n); }
cudaError_t fake_cudaMallocAsync(void** p, size_t n, cudaStream_t s) {
    if (captured(s)) complain("memory that would belong to a graph");
    return give(p, n);
}
cudaError_t fake_cudaFree(void* p) { return take_back(p); }
cudaError_t fake_cudaFreeAsync(void* p, cudaStream_t s) {
    if (captured(s)) complain("memory freed by a graph");
    return take_back(p);
}
cudaError_t fake_cudaMemset(void* p, int v, size_t n) { if (inside("memset", p, n)) std::memset(p, v, n); return cudaSuccess; }
cudaError_t fake_cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) { return enqueue(s, [=] { fake_cudaMemset(p, v, n); }); }
cudaError_t fake_cudaMemcpyAsync(void* d, const void* src, size_t n, cudaMemcpyKind, cudaStream_t s) { return enqueue(s, [=] { std::memcpy(d, src, n); }); }
cudaError_t fake_cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t fake_cudaStreamIsCapturing(cudaStream_t st, cudaStreamCaptureStatus* s) {
    *s = captured(st) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t fake_cudaGetLastError() { return cudaSuccess; }
// threads that wait for a stream at the same time: each waits for as many as are asked for, or for a while
std::mutex g_meet_mu;
std::condition_variable g_meet_cv;
int g_meet_want = 0, g_meet_now = 0, g_meet_most = 0;
cudaError_t fake_cudaStreamSynchronize(cudaStream_t s) {
    if (captured(s)) complain("a captured stream is waited for");
    std::unique_lock<std::mutex> lock(g_meet_mu);
    if (g_meet_want > 0) {
        if (++g_meet_now > g_meet_most) { g_meet_most = g_meet_now; g_meet_cv.notify_all(); }
        g_meet_cv.wait_for(lock, std::chrono::milliseconds(500), [] { return g_meet_most >= g_meet_want; });
        --g_meet_now;
    }
    return cudaSuccess;
}
cudaError_t fake_cudaHostAlloc(void** p, size_t n, unsigned) { return give(p, n); }
cudaError_t fake_cudaFreeHost(void* p) { return take_back(p); }
cudaError_t fake_cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t fake_cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = reinterpret_cast<cudaStream_t>(7); return cudaSuccess; }
cudaError_t fake_cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }

}  // namespace

namespace bv {

int fake_phase_max_ctas(int, int sms) { return sms; }
int fake_small_max_ctas(int, int sms) { return sms; }
int fake_flow_max_ctas_per_sm(int) { return 1; }
int fake_cluster_max_clusters(int, int, int c) { return 148 / c; }
int fake_stream_max_clusters(int, int, bool, int c) { return 148 / c; }

cudaError_t fake_launch_phase(const Params& prm, const PhaseScratch& ps, int, bool, int, cudaStream_t st) {
    if (g_refuse_cooperative) return cudaErrorCooperativeLaunchTooLarge;
    const size_t B = prm.B, g = prm.gamma;
    ++g_launches;
    return enqueue(st, [=] {
        inside("status word", prm.status, 4);
        zeros("phase counters", ps.ctr, ps.zero_words * 4);
        scratch("phase pieces", ps.part, B * ps.rows * ps.slots * sizeof(double2));
        scratch("drafted logits", ps.drafted, B * g * sizeof(float2));
        scratch("positions", ps.pos, B * (g + 1) * sizeof(PhPos));
        scratch("candidates", ps.sel, B * 3 * sizeof(uint4));
        scratch("later candidates", ps.rest, B * sizeof(uint2));
        scratch("unit references", ps.seg_M, B * ps.units * sizeof(float));
        scratch("unit totals", ps.seg, B * (g + 1) * ps.units * sizeof(double));
        zeros("phase counters beside the scratch", ps.ctr, ps.zero_words * 4);
    });
}
cudaError_t fake_launch_small(const Params& prm, const SmallScratch& sc, int, bool, int, cudaStream_t st) {
    if (g_refuse_cooperative) return cudaErrorCooperativeLaunchTooLarge;
    const size_t B = prm.B, g = prm.gamma;
    ++g_launches;
    return enqueue(st, [=] {
        inside("status word", prm.status, 4);
        zeros("barrier words", sc.barrier, 17 * 4);
        zeros("counters of the sequences", sc.seq, kSmallMaxB * 4);
        scratch("chunk pairs", sc.part, B * (2 * g + 1) * sc.nch * sizeof(double2));
        scratch("segment totals", sc.seg, B * (g + 1) * sc.np * 16 * sizeof(double));
        zeros("barrier words beside the scratch", sc.barrier, 17 * 4);
        zeros("counters of the sequences beside the scratch", sc.seq, kSmallMaxB * 4);
    });
}
cudaError_t fake_launch_flow(const Params& prm, const FlowScratch& fl, int, int, cudaStream_t st) {
    const size_t B = prm.B, g = prm.gamma, rows = B * (g + 1);
    ++g_launches;
    return enqueue(st, [=] {
        inside("status word", prm.status, 4);
        zeros("flow counters", fl.counters, static_cast<size_t>(fl.zero_words) * 4);
        scratch("chunk pairs", fl.part, rows * fl.part_stride * sizeof(RowZ));
        scratch("normalisers", fl.rowZ, rows * sizeof(RowZ));
        scratch("prefix chain", fl.pchain, B * (g + 2) * sizeof(double));
        scratch("scales", fl.cscale, rows * sizeof(float));
        scratch("ratios", fl.ratio, rows * sizeof(double));
        scratch("normaliser ratios", fl.zratio, rows * sizeof(double));
        scratch("segment totals", fl.seg_tot, rows * fl.segs * sizeof(double));
        scratch("residual masses", fl.S, rows * sizeof(double));
        scratch("candidates", fl.cand, rows * sizeof(int));
        scratch("tau", fl.tv_tau, B * sizeof(int));
        zeros("flow counters beside the scratch", fl.counters, static_cast<size_t>(fl.zero_words) * 4);
    });
}
cudaError_t fake_launch_cluster(const Params& prm, int, int, int, int, cudaStream_t st) {
    ++g_launches;
    return enqueue(st, [=] { inside("status word", prm.status, 4); });
}
cudaError_t fake_launch_stream(const Params& prm, int, int, bool, int, int, cudaStream_t st) {
    ++g_launches;
    return enqueue(st, [=] { inside("status word", prm.status, 4); });
}

}  // namespace bv

#define cudaGetDevice fake_cudaGetDevice
#define cudaDeviceGetAttribute fake_cudaDeviceGetAttribute
#define cudaMalloc fake_cudaMalloc
#define cudaMallocAsync fake_cudaMallocAsync
#define cudaFree fake_cudaFree
#define cudaFreeAsync fake_cudaFreeAsync
#define cudaMemset fake_cudaMemset
#define cudaMemsetAsync fake_cudaMemsetAsync
#define cudaMemcpyAsync fake_cudaMemcpyAsync
#define cudaThreadExchangeStreamCaptureMode fake_cudaThreadExchangeStreamCaptureMode
#define cudaStreamIsCapturing fake_cudaStreamIsCapturing
#define cudaGetLastError fake_cudaGetLastError
#define cudaStreamSynchronize fake_cudaStreamSynchronize
#define cudaHostAlloc fake_cudaHostAlloc
#define cudaFreeHost fake_cudaFreeHost
#define cudaDeviceSynchronize fake_cudaDeviceSynchronize
#define cudaStreamCreateWithFlags fake_cudaStreamCreateWithFlags
#define cudaStreamDestroy fake_cudaStreamDestroy
#define phase_max_ctas fake_phase_max_ctas
#define small_max_ctas fake_small_max_ctas
#define flow_max_ctas_per_sm fake_flow_max_ctas_per_sm
#define cluster_max_clusters fake_cluster_max_clusters
#define stream_max_clusters fake_stream_max_clusters
#define launch_phase fake_launch_phase
#define launch_small fake_launch_small
#define launch_flow fake_launch_flow
#define launch_cluster fake_launch_cluster
#define launch_stream fake_launch_stream
#include "bv_api.cu"

extern "C" {
void host_begin_capture(void* stream) { g_graphs.emplace_back(); g_capturing = true; g_captured = static_cast<cudaStream_t>(stream); }
int host_end_capture() { g_capturing = false; return static_cast<int>(g_graphs.size()) - 1; }
void host_replay(int graph) { for (const auto& f : g_graphs[graph]) f(); }
void host_set_device(int device) { t_device = device; }
// from now on: how many threads wait for a stream together, at most
void host_meet(int want) { g_meet_want = want; g_meet_most = 0; }
int host_met() { return g_meet_most; }
void host_refuse_cooperative(int on) { g_refuse_cooperative = on; }
// a verification of the decoding loop
int host_tables(int algo, int B, int gamma, int V, int dtype, int lse, int probe) {
    void* x = reinterpret_cast<void*>(1ull << 41);
    return bv::run_tables(algo, x, x, static_cast<int32_t*>(x), static_cast<int32_t*>(x), static_cast<float*>(x), lse ? static_cast<float*>(x) : nullptr,
                          B, gamma, V, dtype, 1.f, static_cast<int32_t*>(x), static_cast<int32_t*>(x), probe != 0, nullptr);
}
int host_launches() { return g_launches; }
int host_loop_pays(int V, int dtype, int B, int gamma, int token) { return bv::loop_pays(V, dtype, B, gamma, token != 0, 148); }
// which of the elements of `esz` bytes at p lie in [lo, hi)
void host_elements_inside(unsigned long long p, unsigned long long lo, unsigned long long hi, int esz, int* first, int* n) {
    const char *a = reinterpret_cast<const char*>(p), *b = reinterpret_cast<const char*>(lo), *c = reinterpret_cast<const char*>(hi);
    if (esz == 4) bv::elements_inside<4>(a, b, c, *first, *n); else bv::elements_inside<8>(a, b, c, *first, *n);
}
// what has gone wrong since the last question
const char* host_errors() { static std::string out; out = g_errors; g_errors.clear(); return out.c_str(); }
size_t host_live_bytes() { size_t n = 0; for (const auto& b : g_blocks) if (b.second.live) n += b.second.bytes; return n; }
}
