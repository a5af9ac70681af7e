// The library's host sources (sfoc_api.cu, batch.cu) over a fake CUDA runtime
// and fake kernel launchers, compiled by the host compiler: allocations are
// counted, limited and given addresses first in, first out by size; launches
// are counted by name and advance a clock by a table of times per form, which
// is what the events measure.  Nothing here touches a device.
// (HOST_SHIM: force-included before the host sources, only what they need.)
#include <cuda_runtime.h>
#include <math.h>
static const uint3 blockIdx = {0, 0, 0};
inline int __float2int_rn(float v) { return (int)rintf(v); }

#ifndef HOST_SHIM
#include <stdlib.h>
#include <string.h>

#include <deque>
#include <map>
#include <string>

#include "host.h"

namespace {

constexpr int kSms = 152;
std::map<size_t, std::deque<void*>> g_free;
std::map<void*, size_t> g_live;
size_t g_bytes = 0, g_limit = ~(size_t)0;
bool g_capturing = false;
std::map<std::string, int> g_count;
int g_last_form = 0;
double g_clock = 0.0;
std::map<int, std::map<int, double>> g_cost;  // form -> full waves of one point per SM -> ms

cudaError_t count(const char* name) {
    ++g_count[name];
    return cudaSuccess;
}

int points(const sfoc::MatchJob& one, const sfoc::ItemSet& is) { return is.items ? is.n : one.n; }

// a correlation launch: form = 1000 path + side, its time by the number of waves
cudaError_t corr(int form, int n) {
    ++g_count["corr"];
    g_last_form = form;
    auto it = g_cost.find(form);
    if (it != g_cost.end() && !it->second.empty()) {
        const int period = it->second.rbegin()->first, k = (n + kSms - 1) / kSms;
        g_clock += (k / period) * it->second[period] + (k % period ? it->second[k % period] : 0.0);
    }
    return cudaSuccess;
}

}  // namespace

#define FAKE extern "C" __attribute__((visibility("default")))

FAKE size_t fk_live() { return g_live.size(); }
FAKE size_t fk_bytes() { return g_bytes; }
FAKE void fk_limit(size_t b) { g_limit = b; }
FAKE void fk_capturing(int on) { g_capturing = on != 0; }
FAKE int fk_count(const char* name) { return g_count.count(name) ? g_count[name] : 0; }
FAKE void fk_reset() { g_count.clear(); }
FAKE int fk_last_form() { return g_last_form; }
FAKE void fk_no_costs() { g_cost.clear(); }
FAKE void fk_cost(int form, int waves, double ms) { g_cost[form][waves] = ms; }

// ---- the runtime ------------------------------------------------------------

FAKE cudaError_t cudaMalloc(void** p, size_t n) {
    *p = nullptr;
    if (n == 0) return cudaSuccess;
    if (g_bytes + n > g_limit) return cudaErrorMemoryAllocation;
    auto& f = g_free[n];
    if (f.empty()) {
        *p = malloc(n);
    } else {
        *p = f.front();
        f.pop_front();
    }
    g_live[*p] = n;
    g_bytes += n;
    return cudaSuccess;
}
FAKE cudaError_t cudaFree(void* p) {
    if (!p) return cudaSuccess;
    auto it = g_live.find(p);
    if (it == g_live.end()) abort();  // freed twice
    g_bytes -= it->second;
    g_free[it->second].push_back(p);
    g_live.erase(it);
    return cudaSuccess;
}
FAKE cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
FAKE cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
FAKE cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
FAKE cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
FAKE cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
FAKE cudaError_t cudaSetDevice(int) { return cudaSuccess; }
FAKE cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
FAKE cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = kSms, count("attribute"); }
FAKE cudaError_t cudaGetLastError() { return cudaSuccess; }
FAKE const char* cudaGetErrorString(cudaError_t) { return "fake"; }
FAKE cudaError_t cudaGetSymbolAddress(void** p, const void*) { return *p = nullptr, cudaErrorUnknown; }
FAKE cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    return *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone, cudaSuccess;
}
FAKE cudaError_t cudaStreamSynchronize(cudaStream_t) { return count("sync"); }
FAKE cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    return *s = reinterpret_cast<cudaStream_t>(1), cudaSuccess;
}
FAKE cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
FAKE cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
FAKE cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
FAKE cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return *g = nullptr, cudaSuccess; }
FAKE cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    return *e = reinterpret_cast<cudaGraphExec_t>(1), cudaSuccess;
}
FAKE cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
FAKE cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
FAKE cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return count("graph"); }
FAKE cudaError_t cudaEventCreate(cudaEvent_t* e) {
    return *e = reinterpret_cast<cudaEvent_t>(new double(0.0)), cudaSuccess;
}
FAKE cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
FAKE cudaError_t cudaEventDestroy(cudaEvent_t e) {
    delete reinterpret_cast<double*>(e);
    return cudaSuccess;
}
FAKE cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
    return *reinterpret_cast<double*>(e) = g_clock, cudaSuccess;
}
FAKE cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
FAKE cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
    return *ms = (float)(*reinterpret_cast<double*>(b) - *reinterpret_cast<double*>(a)), cudaSuccess;
}

// ---- the launchers ----------------------------------------------------------

namespace sfoc {
cudaError_t launch_sfoc_steer(const float*, int, int, size_t, float*, size_t, const SteerTaps&, cudaStream_t) {
    return count("steer");
}
cudaError_t launch_sfoc_steer(const uint16_t*, int, int, size_t, float*, size_t, const SteerTaps&, cudaStream_t) {
    return count("steer");
}
cudaError_t launch_sfoc_smooth(const float*, size_t, int, int, const SmoothTaps&, Cube&, cudaStream_t) {
    return count("smooth");
}
int smooth_launch_count(const SmoothTaps&) { return 2; }
bool sfoc_batch_supported(const SteerTaps&, const SmoothTaps&) { return true; }
void sfoc_batch_tiles(int, int, int* a, int* b) { *a = *b = 1; }
cudaError_t launch_sfoc_batch(const ImgJob*, int, const int*, int, const int*, int, const SteerTaps&, const SmoothTaps&,
                              cudaStream_t) {
    return count("build_batch");
}
cudaError_t launch_steer_two(const ImgJob*, const SteerTaps&, cudaStream_t) { return count("steer_two"); }
cudaError_t launch_smooth_two(const ImgJob*, const SmoothTaps&, cudaStream_t) { return count("smooth_two"); }
size_t integral_scratch_bytes(int, int) { return 256; }
size_t integral_export_scratch_bytes(int, int) { return 256; }
size_t integral_batch_scratch_bytes(const Cube* const*, int) { return 256; }
size_t integral_batch_blob_bytes(int) { return 256; }
void integral_batch_blob(const Cube* const*, int, char*, void*, int*) {}
cudaError_t launch_integral(const Cube&, void*, cudaStream_t, int*) { return count("integral"); }
cudaError_t launch_integral_batch(const void*, int, const int*, cudaStream_t) { return count("integral"); }
cudaError_t launch_template_stats(const MatchJob&, const ItemSet&, cudaStream_t) { return count("stats"); }
cudaError_t launch_ncc_argmax(const MatchJob&, const ItemSet&, cudaStream_t) { return count("ncc"); }
MatchJob make_job(const Cube& ref, const Cube& sen, const int32_t* pts, int n, int m, int R, PointStat* stats,
                  float* maps, float* out_maps, fastncc_result* out) {
    MatchJob j;
    memset(&j, 0, sizeof(j));
    j.rf32 = ref.f32;
    j.rrm = ref.rm;
    j.sf32 = sen.f32;
    j.z = ref.z;
    j.m = m;
    j.R = R;
    j.n = n;
    j.pts = pts;
    j.stats = stats;
    j.maps = maps;
    j.out_maps = out_maps;
    j.out = out;
    return j;
}
size_t ransac_workspace_bytes(int) { return 256; }
cudaError_t launch_ransac(const double*, const double*, const uint8_t*, int, int, const int32_t*, int n_hyp, double, int,
                          double*, uint8_t*, int32_t*, int32_t*, void*, cudaStream_t, int* launches) {
    *launches = n_hyp > 0 ? 4 : 2;
    return cudaSuccess;
}
int corr_f32_class(int R) { return R <= 63 ? 1 : 0; }
bool corr_f32_supported(int m, int R) { return m + R <= 160; }
cudaError_t launch_corr_f32(const MatchJob& one, const ItemSet& is, int, cudaStream_t) {
    return corr(1000 * SFOC_CORR_DIRECT_F32, points(one, is));
}
bool corr_fft_supported(int m, int R) { return m + 2 * R <= 128; }
int corr_fft_side(int m, int R) { return m + 2 * R <= 64 ? 64 : 128; }
int corr_fft2_side(int m, int R) {
    const int lw = m + 2 * R;
    return lw <= 64 || (lw > 96 && lw <= 128) || lw > 224 ? 0 : (lw + 31) / 32 * 32;
}
cudaError_t launch_corr_fft(const MatchJob& one, const ItemSet& is, int L, bool, cudaStream_t) {
    return corr(1000 * SFOC_CORR_FFT + L, points(one, is));
}
cudaError_t launch_corr_fft2(const MatchJob& one, const ItemSet& is, int L, bool, cudaStream_t) {
    return corr(1000 * SFOC_CORR_FFT + L, points(one, is));
}
int corr_tc_class(int form, int, int) { return form == 3 ? 1 : 0; }
int corr_tc_auto_form(int, int) { return 3; }
bool corr_tc_maps(int, MatchJob&) { return true; }
cudaError_t launch_corr_tc(int, int, const MatchJob& one, const ItemSet& is, const int*, const int*, int, int*,
                           cudaStream_t) {
    return corr(1000 * SFOC_CORR_TC_BAND, points(one, is));
}
}  // namespace sfoc
#endif
