// fcm_run_noalloc: a whole FCM run that allocates no memory.
//
// Who needs this: code that may not allocate device memory when it runs —
// for example a host application whose device memory is reserved up front
// by a pool it does not control, a plugin inside a framework that owns the
// allocator, or a latency-critical service where a cudaMalloc (which can
// synchronise the device and can fail under memory pressure) is not
// acceptable. fcm_run keeps its scratch in a handle that allocates on first
// use; this entry point instead keeps it in one fixed array of device memory
// that is part of the library image and exists on every GPU that loads the
// library until the process exits.
//
// The scratch holds the device-side run state and the blocks' exchange slots
// of the cooperative whole-run kernel (the kernel fcm_run launches). Its size is
// fixed: slots for at most FCM_NOALLOC_MAX_BLOCKS thread blocks. Every call shares it, so calls whose
// work overlaps on the GPU (from several host threads, or on several streams
// without ordering between them) race and give wrong results.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "fcm.h"
#include "fcm_device.cuh"
#include "fcm_internal.h"
#include "fcm_run.h"

using namespace fcm;

namespace {

constexpr size_t kStateBytes = (sizeof(RunState) + 255) / 256 * 256;
constexpr size_t kSlotBytes = run_scratch_bytes(FCM_NOALLOC_MAX_BLOCKS);

// The scratch: run state, then the blocks' exchange scratch (zero at load).
// In host code this name is only a stand-in for the device array; its device
// address comes from cudaGetSymbolAddress, once per device.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kStateBytes + kSlotBytes];

constexpr int kMaxDevices = 64;

struct DeviceSetup {
    bool done = false;
    int status = FCM_OK;
    unsigned char* scratch = nullptr;  // device address of g_noalloc_scratch
    int num_sms = 0;
    unsigned nonce = 0;  // number of the last run on this device (the tag of its exchanges)
    bool fits[FCM_MAX_CLUSTERS + 1][4] = {};  // the whole-run kernel of [C][m kind] can be launched
};

std::mutex g_mu;
DeviceSetup g_dev[kMaxDevices];

// First call on a device: resolve the scratch address and the launch limits
// of every whole-run kernel, with that device current.
int setup_device(int dev) {
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceSetup& d = g_dev[dev];
    if (d.done) return d.status;
    d.done = true;
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) {
        cudaGetLastError();
        return d.status = FCM_ERR_CUDA;
    }
    d.scratch = static_cast<unsigned char*>(ptr);
    int coop = 0;
    if (cudaDeviceGetAttribute(&d.num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
        cudaGetLastError();
        return d.status = FCM_ERR_CUDA;
    }
    const RunTable& t = run_table();
    for (int C = 1; C <= FCM_MAX_CLUSTERS; ++C)
        for (int mk = 0; mk < 4; ++mk) d.fits[C][mk] = run_kernel_fits((const void*)t.run[C][mk], C);
    return d.status = FCM_OK;
}

bool on_device(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" int fcm_run_noalloc(const float* x, int64_t n, int C, float m, float eps, int max_iter,
                               int init_mode, const float* U0, float* U, float* V, void* cuda_stream,
                               fcm_report* rep) {
    if (!x || !U || !V) return FCM_ERR_INVALID_ARG;
    if (n < 1 || n > ((int64_t)1 << 40) || n % 4 != 0) return FCM_ERR_INVALID_ARG;
    if (C < 1 || C > FCM_MAX_CLUSTERS) return FCM_ERR_INVALID_ARG;
    if (!(m > 1.0f) || !std::isfinite(m) || !(eps >= 0.0f) || !std::isfinite(eps) || max_iter < 1)
        return FCM_ERR_INVALID_ARG;
    if (init_mode != FCM_INIT_U && init_mode != FCM_INIT_V) return FCM_ERR_INVALID_ARG;
    // the call copies through host memory and synchronises its stream, which a
    // stream under capture cannot do: refuse such a stream before any other
    // runtime call
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing((cudaStream_t)cuda_stream, &cap) != cudaSuccess) {
        cudaGetLastError();
        return FCM_ERR_INVALID_ARG;
    }
    if (cap != cudaStreamCaptureStatusNone) return FCM_ERR_INVALID_ARG;
    if (init_mode == FCM_INIT_U && !U0) U0 = U;
    const float* Uin = init_mode == FCM_INIT_U ? U0 : U;
    if (!on_device(x) || !on_device(U) || !on_device(Uin)) return FCM_ERR_INVALID_ARG;
    if ((uintptr_t)x % 16 || (uintptr_t)U % 16 || (uintptr_t)Uin % 16) return FCM_ERR_INVALID_ARG;

    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return FCM_ERR_CUDA;
    }
    int rc = setup_device(dev);
    if (rc) return rc;
    const DeviceSetup& d = g_dev[dev];
    cudaStream_t stream = (cudaStream_t)cuda_stream;

    const int mk = mkind_of(m);
    if (!d.fits[C][mk]) return FCM_ERR_CUDA;
    const RunShape shape = run_shape(n, C, std::min(d.num_sms, RUN_MAX_BLOCKS));
    if (shape.blocks > FCM_NOALLOC_MAX_BLOCKS) return FCM_ERR_TOO_LARGE;

    RunState* st = reinterpret_cast<RunState*>(d.scratch);
    char* slots = reinterpret_cast<char*>(d.scratch + kStateBytes);

    RunArgs ra;
    std::memset(&ra, 0, sizeof(ra));
    ra.x = x;
    ra.U0 = Uin;
    ra.U = U;
    ra.out = st;
    ra.scratch = slots;
    ra.n = n;
    ra.m = m;
    ra.inv_m1 = (float)(1.0 / ((double)m - 1.0));
    ra.eps = eps;
    ra.max_iter = max_iter;
    ra.from_u = init_mode == FCM_INIT_U;
    ra.resident = shape.resident;
    ra.max_blocks = std::min<int>(FCM_NOALLOC_MAX_BLOCKS, RUN_MAX_BLOCKS);
    ra.guard_n = run_guard_n(n);
    ra.lim = WaitLimits{DEFAULT_GRID_SPINS, DEFAULT_TMA_POLLS, 0u, 0u};
    const bool V_dev = on_device(V);
    if (init_mode == FCM_INIT_V && V_dev) ra.Vin = V;
    else if (init_mode == FCM_INIT_V) std::memcpy(ra.V0, V, sizeof(float) * C);
    if (V_dev) ra.Vout = V;

    // the status starts at running
    RunState hs;
    std::memset(&hs, 0, sizeof(hs));
    hs.status = STATUS_RUNNING;
    cudaError_t e = cudaMemcpyAsync(st, &hs, sizeof(RunState), cudaMemcpyHostToDevice, stream);
    // the run's number, and zeroed slots when the numbers start over (no slot
    // then shows a tag of an earlier run of the same number)
    unsigned& nonce = ra.nonce;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        nonce = ++g_dev[dev].nonce;
        if (nonce == 0) nonce = g_dev[dev].nonce = 1;
    }
    if (e == cudaSuccess && nonce == 1) e = cudaMemsetAsync(slots, 0, kSlotBytes, stream);
    if (e == cudaSuccess) {
        void* args[1] = {&ra};
        e = cudaLaunchCooperativeKernel((const void*)run_table().run[C][mk], dim3(shape.blocks), dim3(shape.threads), args, shape.smem,
                                        stream);
    }
    if (e != cudaSuccess) {
        std::lock_guard<std::mutex> lock(g_mu);
        g_dev[dev].nonce = 0;  // the number was not used: the next run zeroes the scratch
    }
    RunState out;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&out, st, sizeof(RunState), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e == cudaSuccess && !V_dev) std::memcpy(V, out.V, sizeof(float) * C);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return FCM_ERR_CUDA;
    }
    if (rep) {
        std::memset(rep, 0, sizeof(*rep));
        rep->iters = out.iters;
        rep->status = out.status;
        rep->flags = out.flags | (int)out.bounds;
        rep->C = C;
        rep->delta = out.delta;
        rep->J = out.J;
        for (int j = 0; j < C; ++j) rep->V64[j] = out.V64[j];
        rep->launches = 1;
    }
    return out.status == STATUS_RUNNING ? FCM_ERR_CUDA : out.status;
}
