// Host probe of the C API (capi.cpp), built by tests/test_capi_host.py with the host
// compiler: the CUDA runtime and the kernels' launches are fakes, so no device is
// involved.  Launches on streams and events are recorded with the set of launches that
// come before each, so that a captured batch's order can be checked.  Commands on stdin:
//   batch W H n host shift   a process_batch whose predictors are pair (i + shift) mod n's
//                            outputs (shift -1: other memory), run twice;
//                            prints "status parts unordered beside": the parts of the captured
//                            sequence, the (read, write) pairs it leaves unordered and the
//                            uploads that are launched as running beside other parts' passes
//   adjoint                  score calls of which the first one's initialisation of the
//                            workspace fails; prints per call "status initialised launched"
#include <bitset>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

#include <cuda_runtime.h>

template <class T>
cudaError_t cudaGetSymbolAddress(void **p, const T &s)
{
    *p = const_cast<T *>(&s);
    return cudaSuccess;
}
template <class T>
cudaError_t cudaMemcpyFromSymbolAsync(void *d, const T &s, size_t n, size_t, cudaMemcpyKind, cudaStream_t)
{
    std::memcpy(d, &s, n);
    return cudaSuccess;
}
template <class T>
cudaError_t cudaMemcpyToSymbolAsync(T &d, const void *s, size_t n, size_t, cudaMemcpyKind, cudaStream_t)
{
    std::memcpy(&d, s, n);
    return cudaSuccess;
}

#include "capi.cpp"

namespace {

using Set = std::bitset<4096>;
struct Op {
    bool reads, writes;  // the caller's predictors / the call's fields
    int first, count;
    Set before;
};
std::vector<Op> ops;
std::map<cudaStream_t, Set> at;
std::map<cudaEvent_t, Set> ev;
const PairIO *io_base = nullptr;
size_t handles = 0;
int inits = 0, fail_inits = 0, adjoints = 0, beside = 0;

int pair_of(const PtrRef &r) { return (int)((r.base - reinterpret_cast<const char *>(io_base)) / (long long)sizeof(PairIO)); }

cudaError_t op(cudaStream_t st, bool reads, bool writes, int first, int count)
{
    ops.push_back({reads, writes, first, count, at[st]});
    at[st].set(ops.size() - 1);
    return cudaSuccess;
}

template <class T>
cudaError_t make(T *p)
{
    *p = reinterpret_cast<T>(++handles);
    return cudaSuccess;
}

}  // namespace

namespace rpiv {
cudaError_t launch_deform(const DeformArgs &a, int n, cudaStream_t st)
{
    for (int i = 0; i < a.n_src; ++i)
        if (a.src[i].u.indirect) return op(st, true, false, pair_of(a.src[i].u), n);
    return op(st, false, false, 0, 0);
}
cudaError_t launch_uod(const UodArgs &a, int n, cudaStream_t st)
{
    return a.u_out.indirect ? op(st, false, true, pair_of(a.u_out), n) : op(st, false, false, 0, 0);
}
cudaError_t launch_vort(const VortArgs &a, int n, cudaStream_t st) { return op(st, false, true, pair_of(a.u), n); }
cudaError_t launch_frames(const FramesArgs &, int, cudaStream_t st) { return op(st, false, false, 0, 0); }
cudaError_t launch_upload(const UploadArgs &a, int, cudaStream_t st)
{
    beside += a.beside;
    return op(st, false, false, 0, 0);
}
cudaError_t launch_interp(const InterpArgs &, int, cudaStream_t st) { return op(st, false, false, 0, 0); }
cudaError_t launch_preprocess(const PreArgs &, void *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_ema(const float *, float *, size_t, float, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_pass_fp32(const PassArgs &, dim3, int, cudaStream_t st) { return op(st, false, false, 0, 0); }
cudaError_t launch_pass_bf16(const PassArgs &, dim3, int, cudaStream_t st) { return op(st, false, false, 0, 0); }
cudaError_t launch_pass_fp16(const PassArgs &, dim3, int, cudaStream_t st) { return op(st, false, false, 0, 0); }
void prepare_pass_fp32() {}
void prepare_pass_bf16() {}
void prepare_pass_fp16() {}
bool pass_supported_bf16(int R) { return R >= 0 && R <= 16; }
bool pass_supported_fp16(int R) { return R >= 0 && R <= 16; }
void attach_region_maps(PassArgs &a, int) { a.tma = 0; }
bool deform_nodes_fit(int, int s, int, int) { return s >= 3; }
size_t preprocess_scratch_bytes(int, int, int, int) { return 256; }
size_t adjoint_workspace_bytes(int W, int H, int, int, int, int) { return (size_t)W * H * 4; }
cudaError_t init_adjoint_workspace(void *, cudaStream_t)
{
    if (fail_inits > 0) {
        --fail_inits;
        return cudaErrorUnknown;
    }
    ++inits;
    return cudaSuccess;
}
void prepare_adjoint() {}
cudaError_t launch_adjoint(const AdjArgs &, cudaStream_t)
{
    ++adjoints;
    return cudaSuccess;
}
cudaError_t launch_refine_axpy(const float *, const float *, const float *, const float *, float, float *, float *, int,
                               cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_refine_absmax(const float *, const float *, int, float *, cudaStream_t) { return cudaSuccess; }
}  // namespace rpiv

extern "C" {
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { return *n = 1, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorName(cudaError_t) { return "error"; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaMalloc(void **p, size_t n) { return (*p = std::calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) { return *d = h, cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) { return a->type = cudaMemoryTypeHost, cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return make(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return at[s] |= ev[e], cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return make(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return make(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return ev[e] = at[s], cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *t, cudaEvent_t, cudaEvent_t) { return *t = 0.f, cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode)
{
    beside = 0;
    ops.clear();
    at.clear();
    ev.clear();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return make(g); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *g, cudaGraph_t, unsigned long long) { return make(g); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
}

static void batch(int W, int H, int n, int host, int shift)
{
    rpiv_config c;
    rpiv_config_default(&c);
    c.width = W;
    c.height = H;
    c.max_batch = n;
    c.host_frames = host;
    rpiv_handle *h = nullptr;
    if (rpiv_create(&c, 0, &h) != RPIV_OK) {
        std::printf("create: %s\n", rpiv_last_error());
        return;
    }
    io_base = h->io_dev;
    int nx = 0, ny = 0;
    rpiv_grid_shape(h, &nx, &ny);
    const size_t count = (size_t)nx * ny;
    std::vector<float> field(5 * n * count);  // per pair: u, v, and predictors of their own
    std::vector<const void *> img(n, field.data());
    std::vector<float *> u(n), v(n);
    std::vector<const float *> pu(n), pv(n);
    for (int i = 0; i < n; ++i) u[i] = &field[5 * i * count], v[i] = u[i] + count;
    for (int i = 0; i < n; ++i) {
        const int j = shift < 0 ? i : (i + shift) % n;
        pu[i] = u[j] + (shift < 0 ? 2 * count : 0);
        pv[i] = v[j] + (shift < 0 ? 2 * count : 0);
    }
    rpiv_status st = RPIV_OK;
    for (int k = 0; k < 2 && st == RPIV_OK; ++k)
        st = rpiv_process_batch(h, n, img.data(), img.data(), W, pu.data(), pv.data(), u.data(), v.data(), nullptr, nullptr, nullptr);
    std::set<int> parts;
    int unordered = 0;
    for (size_t w = 0; w < ops.size(); ++w) {
        if (!ops[w].writes) continue;
        parts.insert(ops[w].first);
        for (size_t r = 0; r < ops.size(); ++r) {
            if (!ops[r].reads || ops[w].before.test(r)) continue;
            bool shared = false;
            for (int i = ops[r].first; shift >= 0 && i < ops[r].first + ops[r].count; ++i) {
                const int j = (i + shift) % n;
                shared |= j >= ops[w].first && j < ops[w].first + ops[w].count;
            }
            unordered += shared;
        }
    }
    std::printf("%d %d %d %d\n", (int)st, (int)parts.size(), unordered, beside);
    rpiv_destroy(h);
}

static void adjoint()
{
    rpiv_config c;
    rpiv_config_default(&c);
    c.width = c.height = 64;
    rpiv_handle *h = nullptr;
    rpiv_create(&c, 0, &h);
    std::vector<float> f(64 * 64);
    float score = 0.f;
    fail_inits = 1;
    for (int k = 0; k < 3; ++k) {
        const rpiv_status st = rpiv_backward(h, f.data(), f.data(), 64, f.data(), f.data(), 1.f, nullptr, nullptr, &score, nullptr);
        std::printf("%d %d %d ", (int)st, inits, adjoints);
    }
    std::printf("\n");
    rpiv_destroy(h);
}

int main()
{
    char cmd[32];
    while (std::scanf("%31s", cmd) == 1) {
        int W, H, n, host, shift;
        if (std::string(cmd) == "batch" && std::scanf("%d %d %d %d %d", &W, &H, &n, &host, &shift) == 5) batch(W, H, n, host, shift);
        else if (std::string(cmd) == "adjoint") adjoint();
    }
    return 0;
}
