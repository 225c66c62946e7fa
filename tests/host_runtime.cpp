// The library's host runtime (vans_api.cu) on a CUDA runtime that runs nothing: every
// call and launch is written to a log, calls fail when told to, and a captured graph's
// entries are logged again when it is launched.  Built by test_host_runtime.py.
#include <map>
#include <string>
#include <vector>

#include "vans_internal.h"

namespace {

std::vector<std::string> g_log, *g_into = &g_log;   // the capture's list while one is open
std::map<std::string, int> g_fail;                  // calls until this one fails (1: the next)
cudaError_t g_last = cudaSuccess;                   // as cudaGetLastError has it
std::vector<std::vector<std::string>> g_graphs;
std::string g_text;
bool g_user_capture = false, g_quiet = false;       // quiet: steps are counted, not logged
long long g_steps = 0;
std::vector<long long> g_graph_steps;

void put(const std::string &s) {
    const size_t at = s.find_first_of("0123456789");
    const bool steps = s.compare(0, 4, "step") == 0 || s.compare(0, 5, "multi") == 0 ||
                       s.compare(0, 7, "cluster") == 0 || s.compare(0, 7, "monitor") == 0;
    if (steps) (g_into == &g_log ? g_steps : g_graph_steps.back()) += atoi(s.c_str() + at);
    if (!g_quiet || g_into != &g_log) g_into->push_back(s);
}
cudaError_t call(const char *name) {
    auto f = g_fail.find(name);
    if (f != g_fail.end() && f->second > 0 && --f->second == 0) return g_last = cudaErrorUnknown;
    return cudaSuccess;
}
cudaError_t logged(const std::string &s) {          // as a launch: an earlier call's error too
    put(s);
    call(s.substr(0, s.find(' ')).c_str());
    return cudaGetLastError();
}
std::string num(long long v) { return std::to_string(v); }

}  // namespace

extern "C" {

void fake_reset() {
    g_log.clear();
    g_fail.clear();
    g_into = &g_log;
    g_user_capture = g_quiet = false;
    g_last = cudaSuccess;
    g_steps = 0;
}
void fake_quiet() { g_quiet = true; }
long long fake_steps() { return g_steps; }
void fake_fail(const char *name, int after) { g_fail[name] = after; }
void fake_user_capture(int on) { g_user_capture = on != 0; }
const char *fake_log() {
    g_text.clear();
    for (const auto &s : g_log) g_text += s + "\n";
    return g_text.c_str();
}

cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)8; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)8; return call("event"); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *t, cudaEvent_t, cudaEvent_t) { *t = 1.f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return call("record"); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return g_user_capture ? cudaErrorCapturedEvent : cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = calloc(1, n); return call("hostalloc"); }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)16; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) {
    return g_user_capture ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    *s = g_user_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
    if (call("capture") != cudaSuccess) return cudaErrorUnknown;
    g_graphs.emplace_back();
    g_graph_steps.push_back(0);
    g_into = &g_graphs.back();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    g_into = &g_log;
    *g = (cudaGraph_t)g_graphs.size();
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long) {
    *e = (cudaGraphExec_t)g;
    return call("instantiate");
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
    if (g_user_capture) return cudaErrorStreamCaptureUnsupported;
    g_steps += g_graph_steps[(size_t)e - 1];
    if (!g_quiet)
        for (const auto &s : g_graphs[(size_t)e - 1]) g_log.push_back(s);
    return call("graph");
}
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return logged("memset"); }
cudaError_t cudaMemcpyAsync(void *to, const void *, size_t n, cudaMemcpyKind kind, cudaStream_t) {
    if (kind == cudaMemcpyDeviceToHost) memset(to, 0, n);       // status words: nothing wrong
    return logged("copy");
}

}  // extern "C"

namespace vans {

cudaError_t launch_step(int, const VDom &, const float *, float *, Launch L, cudaStream_t) {
    return logged("step 1 kind " + num(L.kind) + " warps " + num(L.warps) + " rows " + num(L.rows));
}
cudaError_t launch_multi(const VDom &, const float *, float *, int steps, int strips, cudaStream_t) {
    return logged("multi " + num(steps) + " strips " + num(strips));
}
cudaError_t multi_strips(const VDom &, int steps, int, int *strips) {
    *strips = 10 * steps;
    return logged("strips " + num(steps));
}
cudaError_t launch_step_cluster(int, const VDom &, const float *, float *, int n, Launch, bool pairs, cudaStream_t) {
    return logged("cluster " + num(n) + (pairs ? " pairs" : ""));
}
cudaError_t launch_step_monitor(int, const VDom &, const float *, float *, float *, float *, float *, float *, cudaStream_t) {
    return logged("monitor 1");
}
cudaError_t launch_monitor_finalize(const float *, float *, cudaStream_t) { return logged("maxima"); }
cudaError_t launch_moments(int, const VDom &, const float *, float *, float *, cudaStream_t) { return logged("moments"); }
cudaError_t launch_moments_rows(const VDom &, const float *, float *, float *, float *, float *, cudaStream_t) {
    return logged("moments");
}
cudaError_t launch_export(int, const VDom &, const float *, float *, cudaStream_t) { return logged("export"); }
cudaError_t launch_import(int, const VDom &, const float *, float *, cudaStream_t) { return logged("import"); }
cudaError_t launch_pad_eps(const VDom &, const float *, float *, int *, cudaStream_t, const int *) { return logged("pad"); }
cudaError_t launch_check_eps(const VDom &, const float *, int *, cudaStream_t) { return logged("check_eps"); }
cudaError_t launch_rebase_eps(int, const VDom &, const float *, float *, const int *, cudaStream_t) { return logged("rebase"); }
cudaError_t launch_init_moving(int, const VDom &, float *, cudaStream_t) { return logged("init"); }
cudaError_t launch_check(int, const VDom &, const float *, int *, cudaStream_t) { return logged("check"); }
cudaError_t launch_flux(int, const VDom &, const float *, int, float *, cudaStream_t) { return logged("flux"); }
cudaError_t launch_flux_seed(int, const VDom &, const float *, int, float *, float *, int, cudaStream_t) { return logged("seed"); }
cudaError_t launch_step_adjoint(int, const VDom &, const float *, const float *, float *, float *, int, Launch, cudaStream_t) {
    return logged("reverse 1");
}
cudaError_t launch_grad_finalize(int, const VDom &, const float *, const float *, float *, int, cudaStream_t) {
    return logged("stencil");
}
cudaError_t launch_ring_batched(const VDom *, const Tile *, int, int, Launch L, int *, cudaStream_t, unsigned long long *) {
    return logged("step 1 kind " + num(L.kind));
}
cudaError_t launch_step_batched(const VDom *, const Tile *, int, int, Launch, int, cudaStream_t) { return logged("step 1 kind 0"); }
cudaError_t launch_multi_batched(const VDom *, const Tile *, int, int, int, int steps, cudaStream_t) {
    return logged("multi " + num(steps));
}
cudaError_t launch_halo_pack(int, const VDom &, const float *, float *, float *, cudaStream_t) { return logged("pack"); }
cudaError_t launch_halo_unpack(int, const VDom &, float *, const float *, const float *, cudaStream_t) { return logged("unpack"); }
cudaError_t launch_eps_halo(const VDom &, const float *, const float *, float *, int *, cudaStream_t) { return logged("eps_halo"); }
int halo_floats(int, const VDom &) { return 1; }
int batched_blocks_per_sm(Launch) { return 1; }
int multi_out_cols(int) { return 56; }
bool launch_has_plates(int, Launch L) { return L.kind == 0; }
bool multi_fits(int q, const VDom &d) { return q == 9 && !d.nee && d.xwrap; }
bool cluster_fits(int, const VDom &d, int, int) { return d.cells <= 8192; }

}  // namespace vans
