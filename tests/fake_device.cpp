// A CUDA runtime and kernels that run on the host, for tests of the host side
// (aaqaoa_host.cu compiled as C++): "device" memory is host memory, all streams
// are one queue, and nothing in the queue runs before a synchronisation, the
// latest that CUDA allows. The kernels below do what the host code may rely on,
// not the simulation: an energy is sum gamma + 2 sum beta + 1000 |E(cost)|.
#include <cuda_runtime.h>

#include <alloca.h>
#include <cmath>
#include <cstring>
#include <functional>
#include <utility>
#include <vector>

#include "aaqaoa_internal.h"

using namespace aaq;

namespace {

std::vector<std::function<void()>> g_queue;
int g_changed = 0;    // sources of queued copies that changed before the copy ran
int g_expire = 0;     // the next launch with a bounded wait finds it expired
int g_circuits = 0;   // whole-circuit launches
int g_lose = 0;       // the next whole-circuit launch writes nothing
int g_no_pinned = 0;  // cudaHostAlloc fails
cudaStreamCaptureMode g_mode = cudaStreamCaptureModeGlobal;  // this thread's
int g_unsafe = 0;     // allocations that would invalidate another thread's global capture

__attribute__((noinline)) void clobber_stack()
{
    volatile unsigned char *p = static_cast<unsigned char *>(alloca(1 << 16));
    for (int i = 0; i < (1 << 16); i++)
        p[i] = 0xA5;
}

void run_queue()
{
    clobber_stack();
    std::vector<std::function<void()>> q;
    q.swap(g_queue);
    for (auto &f : q)
        f();
}

template <typename F>
int edges_of(const F &f, int n)
{
    int e = 0;
    for (int k = 0; k < f.K; k++)
        for (int u = 0; u < n; u++)
            e += __builtin_popcountll(f.nbr[k][u]);
    return e / 2;
}

}  // namespace

extern "C" {

int fake_changed_sources() { return g_changed; }
void fake_expire_next_wait() { g_expire = 1; }
int fake_circuit_launches() { return g_circuits; }
void fake_lose_next_launch() { g_lose = 1; }
void fake_no_pinned_memory(int on) { g_no_pinned = on; }
int fake_unsafe_allocations() { return g_unsafe; }
int fake_capture_mode() { return (int)g_mode; }

cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorName(cudaError_t) { return "fake"; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) { memset(p, 0, sizeof *p); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { *p = const_cast<void *>(s); return cudaSuccess; }

CUresult fake_encode(...) { return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q)
{
    *p = reinterpret_cast<void *>(&fake_encode);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind kind, cudaStream_t)
{
    std::vector<unsigned char> was;
    if (kind == cudaMemcpyHostToDevice)
        was.assign(static_cast<const unsigned char *>(src), static_cast<const unsigned char *>(src) + n);
    g_queue.push_back([=] {
        if (!was.empty() && memcmp(was.data(), src, n))
            g_changed++;
        memcpy(dst, src, n);
    });
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *dst, const void *src, size_t n, cudaMemcpyKind)
{
    run_queue();
    memcpy(dst, src, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *dst, size_t dp, const void *src, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t)
{
    g_queue.push_back([=] {
        for (size_t i = 0; i < h; i++)
            memcpy(static_cast<char *>(dst) + i * dp, static_cast<const char *>(src) + i * sp, w);
    });
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *dst, int v, size_t n, cudaStream_t)
{
    g_queue.push_back([=] { memset(dst, v, n); });
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { run_queue(); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned)
{
    if (g_mode != cudaStreamCaptureModeRelaxed)
        g_unsafe++;
    if (g_no_pinned)
        return cudaErrorMemoryAllocation;
    *p = calloc(1, n);
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *m)
{
    std::swap(*m, g_mode);
    return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) { *d = h; return cudaSuccess; }

cudaError_t cudaEventCreate(cudaEvent_t *) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { run_queue(); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }

}  // extern "C"

namespace aaq {

int device_sms() { return 152; }
int agg_grid(bool) { return 608; }
int pass_grid(long long t) { return t < 152 ? (int)t : 152; }
int tile_bits(bool c128) { return c128 ? 12 : 13; }
int low_two_stage_bits(bool c128, int nv) { return (c128 ? 8 : 9) - (nv == 2 ? 1 : 0); }
void pass_geometry(bool c128, int nv, int *T, int *CB, int *HB)
{
    *T = (c128 ? 12 : 13) - (nv == 2 ? 1 : 0);
    *CB = c128 ? 3 : 4;
    *HB = nv == 2 ? 8 : 9;
}
size_t sample_chunk_count(int n) { return (size_t)1 << (n < 12 ? 0 : n - 7); }

// one CTA up to n = 10, a cluster up to 16, a team (its CTAs wait for one another) up to 20
bool circuit_plan(bool, bool, int n, int p, int, int B, CircuitPlan *q)
{
    if (n < CIRCUIT_MIN_QUBITS || n > CIRCUIT_MAX_QUBITS || p > 64 || (n > 16 && B > 1))
        return false;
    memset(q, 0, sizeof *q);
    q->c = n <= 10 ? 0 : n <= 16 ? 3 : 7;
    q->cluster = q->c == 3;
    q->Tl = n - 1 - q->c;
    return true;
}

int launch_circuit(bool, bool grad, const CircuitArgs &a, const CircuitPlan &q, cudaStream_t)
{
    g_circuits++;
    g_queue.push_back([=] {
        if (g_lose) {
            g_lose = 0;
            return;
        }
        const bool team = q.c && !q.cluster;
        if (team && (g_expire || a.drop_arrival))
            *a.err = 1;
        if (team)
            g_expire = 0;
        if (a.err_out)
            *a.err_out = *a.err;
        for (int b = 0; b < a.B; b++) {
            if (team && *a.err) {
                for (int r = 0; r < (grad ? 1 + 2 * a.p : 1); r++)
                    a.out[(size_t)b * a.out_stride + r] = NAN;
                continue;
            }
            const double *g = a.gamma ? a.gamma + (size_t)b * a.p : a.ang;
            const double *be = a.gamma ? a.beta + (size_t)b * a.p : a.ang + a.p;
            double *row = a.out + (size_t)b * a.out_stride;
            row[0] = 1000.0 * (a.fns ? edges_of(a.fns[b].cost, a.n) : edges_of(a.fn[0], a.n));
            for (int l = 0; l < a.p; l++) {
                row[0] += g[l] + 2.0 * be[l];
                if (grad) {
                    row[1 + l] = g[l];
                    row[1 + a.p + l] = be[l];
                }
            }
        }
    });
    return 0;
}

int launch_params(bool, int B, int p, int, int, const double *d_gamma, const double *d_beta, void *, MixRow *d_cs, int,
                  bool, double *d_out, long long out_count, cudaStream_t)
{
    g_queue.push_back([=] {
        for (int i = 0; i < B * p; i++) {
            d_cs[i].c = d_gamma[i];
            d_cs[i].s = d_beta[i];
        }
        for (long long i = 0; i < out_count; i++)
            d_out[i] = 0.0;
    });
    return 0;
}

int launch_pass(bool, int, const CUtensorMap &, const CUtensorMap &, const PassArgs &a, int, cudaStream_t)
{
    g_queue.push_back([=] {
        if (g_expire)
            *a.err = 1;
        g_expire = 0;
        if (a.slot_idx[0] != 0)
            return;
        for (int b = 0; b < a.B; b++) {
            double e = 1000.0 * edges_of(a.pt ? a.pt[b].cost : a.cost, a.n);
            for (int l = 0; l < a.p; l++)
                e += a.cs[(size_t)b * a.p + l].c + 2.0 * a.cs[(size_t)b * a.p + l].s;
            a.out[(size_t)b * a.out_stride] = e;
        }
    });
    return 0;
}

int launch_small(bool, const SmallArgs &, int, cudaStream_t) { return 0; }
int launch_maxcut(const CostFn &, int, unsigned long long *, cudaStream_t) { return 0; }
int launch_sample(bool, const void *, int, int, double *, double *, int, const double *, unsigned long long *, int *,
                  const CostFn &, cudaStream_t)
{
    return 0;
}
int launch_untwist(bool, void *, int, int, const MixRow *, int, int, cudaStream_t) { return 0; }
int launch_agg_fused(bool, const AggArgs &, cudaStream_t, int) { return 0; }
int launch_agg_terms(bool, const AggArgs &, cudaStream_t, int) { return 0; }
int launch_small_multi(bool, const SmallGraph *, int, int, int, int, int, const double *, const double *, double *,
                       cudaStream_t)
{
    return 0;
}
int launch_cluster_pass(const CUtensorMap *, const PassArgs &, cudaStream_t) { return 0; }

}  // namespace aaq
