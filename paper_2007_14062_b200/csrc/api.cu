// C-ABI entry points that touch the GPU: argument checks, device copies of the layout, library-owned
// scratch, kernel dispatch.  See include/bigbird.h for the contract of each function.
#include <cuda_runtime.h>

#include <cstring>
#include <memory>
#include <mutex>
#include <new>

#include "kernels.h"
#include "../../include/bigbird.h"

namespace bigbird {
namespace {

thread_local int t_last_cuda_error = 0;
thread_local int t_last_launches = 0;

constexpr int kMaxDevices = 64;
std::mutex g_mu;
DeviceScratch g_scratch[kMaxDevices];

int cuda_fail(cudaError_t e) {
    t_last_cuda_error = (int)e;
    return BIGBIRD_ECUDA;
}

// Library scratch of the current device, created on first use.
int get_scratch(int device, DeviceScratch** out) {
    if (device < 0 || device >= kMaxDevices) return BIGBIRD_EUNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceScratch& s = g_scratch[device];
    if (!s.status) {
        int* p = nullptr;
        cudaError_t e = cudaMalloc(&p, sizeof(int) * (2 + 2 * kCounterSlots));
        if (e != cudaSuccess) return cuda_fail(e);
        e = cudaMemset(p, 0, sizeof(int) * (2 + 2 * kCounterSlots));
        if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);        // see upload_layout
        if (e != cudaSuccess) { cudaFree(p); return cuda_fail(e); }
        s.status = p;
        s.counters = p + 2;
    }
    *out = &s;
    return BIGBIRD_OK;
}

// Memory pool of a device: workspaces of calls come from it in stream order, so calls on different streams or threads never
// share one.  It keeps up to 64 MB between calls; it is made with the first use and destroyed with the last layout that has a
// copy on the device (what a call still in flight holds goes when that call is done).
struct DevicePool {
    cudaMemPool_t pool = nullptr;
    int layouts = 0;
};
DevicePool g_pools[kMaxDevices];

int hold_pool(int device) {
    if (device < 0 || device >= kMaxDevices) return BIGBIRD_EUNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_mu);
    ++g_pools[device].layouts;
    return BIGBIRD_OK;
}
void release_pool(int device) {
    std::lock_guard<std::mutex> lock(g_mu);
    DevicePool& d = g_pools[device];
    if (--d.layouts == 0 && d.pool) {
        cudaMemPoolDestroy(d.pool);
        d.pool = nullptr;
    }
}
int get_pool(int device, cudaMemPool_t* out) {
    std::lock_guard<std::mutex> lock(g_mu);
    DevicePool& d = g_pools[device];
    if (!d.pool) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = device;
        cudaError_t e = cudaMemPoolCreate(&d.pool, &props);
        if (e != cudaSuccess) { d.pool = nullptr; return cuda_fail(e); }
        uint64_t keep = 64ull << 20;
        e = cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    *out = d.pool;
    return BIGBIRD_OK;
}

void free_device_layout(DeviceLayout& d) {
    cudaFree(d.block);
    if (d.device >= 0) release_pool(d.device);
    d = DeviceLayout{};
}

// Device copy of the layout: one allocation, one copy.  (Nothing here throws: the callers are C entry points.)
int upload_layout(const bigbird_layout* L, DeviceLayout& d) {
    struct Array {
        void** dst;            // where its device address goes
        const void* src;
        size_t bytes;
    };
    auto array = [](auto** dst, const auto& v) { return Array{(void**)dst, v.data(), v.size() * sizeof(v[0])}; };
    const Array arrays[] = {array(&d.row_ptr, L->row_ptr), array(&d.col_idx, L->col_idx), array(&d.col_ptr, L->col_ptr), array(&d.row_idx, L->row_idx),
                            array(&d.items, L->items_abs), array(&d.steps, L->steps), array(&d.items_t, L->items_t), array(&d.steps_t, L->steps_t),
                            array(&d.global_pairs, L->global_pairs), array(&d.block_order, L->block_order)};
    auto align256 = [](size_t x) { return (x + 255) / 256 * 256; };
    size_t total = 256;
    for (const Array& a : arrays) total += align256(a.bytes);
    std::unique_ptr<unsigned char[]> host(new (std::nothrow) unsigned char[total]);
    if (!host) return BIGBIRD_ENOMEM;
    cudaError_t e = cudaMalloc(&d.block, total);
    if (e != cudaSuccess) return cuda_fail(e);
    size_t at = 0;
    for (const Array& a : arrays) {
        if (a.bytes) std::memcpy(host.get() + at, a.src, a.bytes);
        *a.dst = (unsigned char*)d.block + at;
        at += align256(a.bytes);
    }
    // Waited for: a copy's call may return while it is on its way from the driver's staging memory, and a stream that does not
    // synchronise with the legacy one (torch's streams do not) would not wait for it.
    e = cudaMemcpyAsync(d.block, host.get(), at, cudaMemcpyHostToDevice, cudaStreamLegacy);
    if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);
    return e == cudaSuccess ? BIGBIRD_OK : cuda_fail(e);
}

// Device copy of the layout on the current device (made on first use, remade if the device changes).
int get_device_layout(const bigbird_layout* L, int device, DeviceLayout* out) {
    std::lock_guard<std::mutex> lock(L->mu);
    DeviceLayout& d = L->dev;
    if (d.device != device) {
        if (d.device >= 0) {
            int cur = device;
            cudaSetDevice(d.device);
            free_device_layout(d);
            cudaSetDevice(cur);
        }
        int rc = upload_layout(L, d);
        if (rc != BIGBIRD_OK) { free_device_layout(d); return rc; }
        rc = hold_pool(device);
        if (rc != BIGBIRD_OK) { free_device_layout(d); return rc; }
        d.device = device;
    }
    *out = d;
    return BIGBIRD_OK;
}

int get_sms(int device, int* sms) {
    static int counts[kMaxDevices];
    if (device < 0 || device >= kMaxDevices) return BIGBIRD_EUNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_mu);
    if (!counts[device]) {
        const cudaError_t e = cudaDeviceGetAttribute(&counts[device], cudaDevAttrMultiProcessorCount, device);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    *sms = counts[device];
    return BIGBIRD_OK;
}

int check_common(const void* q, const void* k, const void* v, const bigbird_layout* L, void* out,
                 int B, int H, int64_t N, int D, int b, int dtype) {
    if (!q || !k || !v || !L || !out) return BIGBIRD_EINVAL;
    if (B < 1 || H < 1 || N < 1 || D < 1 || b < 1) return BIGBIRD_EINVAL;
    if (L->N != N || L->b != b || L->H != H) return BIGBIRD_EINVAL;
    if (dtype != BIGBIRD_FP32 && dtype != BIGBIRD_BF16) return BIGBIRD_EUNSUPPORTED;
    if ((((uintptr_t)q) | ((uintptr_t)k) | ((uintptr_t)v) | ((uintptr_t)out)) & 15) return BIGBIRD_EINVAL;
    return BIGBIRD_OK;
}

int fwd(bool force_simt, const void* q, const void* k, const void* v, const bigbird_layout* L,
        const uint8_t* kpm, void* out, float* lse, int B, int H, int64_t N, int D, int b, float scale,
        int dtype, void* stream) {
    t_last_launches = 0;
    int rc = check_common(q, k, v, L, out, B, H, N, D, b, dtype);
    if (rc != BIGBIRD_OK) return rc;
    const bool simt = force_simt || dtype == BIGBIRD_FP32;
    if (simt) {
        if (D != 32 && D != 64 && D != 128) return BIGBIRD_EUNSUPPORTED;
        if ((int64_t)B * H > 65535) return BIGBIRD_EUNSUPPORTED;
    } else {
        if (D != 64 || b != 64) return BIGBIRD_EUNSUPPORTED;
    }
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return cuda_fail(e);
    DeviceLayout dl;
    rc = get_device_layout(L, device, &dl);
    if (rc != BIGBIRD_OK) return rc;
    FwdArgs a{q, k, v, kpm, out, lse, B, H, D, b, L->nb, N, scale, dtype, (cudaStream_t)stream};
    if (simt) {
        int sms = 0;
        rc = get_sms(device, &sms);
        if (rc != BIGBIRD_OK) return rc;
        e = launch_attn_fwd_simt(a, *L, dl, sms, &t_last_launches);
        return e == cudaSuccess ? BIGBIRD_OK : cuda_fail(e);
    }
    DeviceScratch* sc = nullptr;
    rc = get_scratch(device, &sc);
    if (rc != BIGBIRD_OK) return rc;
    cudaError_t ce = cudaSuccess;
    cudaMemPool_t pool = nullptr;
    rc = get_pool(device, &pool);
    if (rc != BIGBIRD_OK) return rc;
    rc = launch_attn_fwd_sm100(a, *L, dl, *sc, pool, &t_last_launches, &ce);
    if (rc == BIGBIRD_ECUDA) t_last_cuda_error = (int)ce;
    return rc;
}

}  // namespace
}  // namespace bigbird

extern "C" {

int bigbird_attn_fwd(const void* q, const void* k, const void* v, const bigbird_layout* layout,
                     const uint8_t* key_padding_mask, void* out, float* lse, int B, int H, int64_t N, int D,
                     int b, float scale, int dtype, void* stream) {
    return bigbird::fwd(false, q, k, v, layout, key_padding_mask, out, lse, B, H, N, D, b, scale, dtype, stream);
}

int bigbird_attn_fwd_simt(const void* q, const void* k, const void* v, const bigbird_layout* layout,
                          const uint8_t* key_padding_mask, void* out, float* lse, int B, int H, int64_t N,
                          int D, int b, float scale, int dtype, void* stream) {
    return bigbird::fwd(true, q, k, v, layout, key_padding_mask, out, lse, B, H, N, D, b, scale, dtype, stream);
}

int bigbird_attn_bwd(const void* q, const void* k, const void* v, const void* out, const float* lse, const void* dout,
                     const bigbird_layout* layout, const uint8_t* key_padding_mask, void* dq, void* dk, void* dv,
                     int B, int H, int64_t N, int D, int b, float scale, int dtype, void* stream) {
    using namespace bigbird;
    t_last_launches = 0;
    int rc = check_common(q, k, v, layout, dq, B, H, N, D, b, dtype);
    if (rc != BIGBIRD_OK) return rc;
    if (!out || !lse || !dout || !dk || !dv) return BIGBIRD_EINVAL;
    if ((((uintptr_t)out) | ((uintptr_t)dout) | ((uintptr_t)dk) | ((uintptr_t)dv)) & 15) return BIGBIRD_EINVAL;
    if (D != 32 && D != 64 && D != 128) return BIGBIRD_EUNSUPPORTED;
    if ((int64_t)B * H > 65535) return BIGBIRD_EUNSUPPORTED;
    if (!(scale > 0.f) || !(scale < INFINITY)) return BIGBIRD_EINVAL;
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return cuda_fail(e);
    DeviceLayout dl;
    rc = get_device_layout(layout, device, &dl);
    if (rc != BIGBIRD_OK) return rc;
    BwdArgs a{q, k, v, out, lse, dout, key_padding_mask, dq, dk, dv, B, H, D, b, layout->nb, N, scale, dtype, (cudaStream_t)stream};
    cudaMemPool_t pool = nullptr;
    rc = get_pool(device, &pool);
    if (rc != BIGBIRD_OK) return rc;
    if (attn_bwd_sm100_takes(a)) {
        DeviceScratch* sc = nullptr;
        rc = get_scratch(device, &sc);
        if (rc != BIGBIRD_OK) return rc;
        rc = launch_attn_bwd_sm100(a, *layout, dl, pool, sc->status, &t_last_launches, &e);
        if (rc == BIGBIRD_ECUDA) t_last_cuda_error = (int)e;
        return rc;
    }
    int sms = 0;
    rc = get_sms(device, &sms);
    if (rc != BIGBIRD_OK) return rc;
    e = launch_attn_bwd_simt(a, *layout, dl, pool, sms, &t_last_launches);
    return e == cudaSuccess ? BIGBIRD_OK : cuda_fail(e);
}

int bigbird_layout_destroy(bigbird_layout* L) {
    if (!L) return BIGBIRD_EINVAL;
    if (L->dev.device >= 0) {
        int cur = 0;
        const bool have = cudaGetDevice(&cur) == cudaSuccess;
        if (cudaSetDevice(L->dev.device) == cudaSuccess) bigbird::free_device_layout(L->dev);
        if (have) cudaSetDevice(cur);
    }
    delete L;
    return BIGBIRD_OK;
}

int bigbird_last_status(void* stream, int* status, int* detail) {
    if (!status) return BIGBIRD_EINVAL;
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return bigbird::cuda_fail(e);
    bigbird::DeviceScratch* sc = nullptr;
    int rc = bigbird::get_scratch(device, &sc);
    if (rc != BIGBIRD_OK) return rc;
    e = cudaStreamSynchronize((cudaStream_t)stream);
    if (e != cudaSuccess) return bigbird::cuda_fail(e);
    int host[2] = {0, 0};
    e = cudaMemcpy(host, sc->status, sizeof(host), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return bigbird::cuda_fail(e);
    if (host[0] != 0) {
        // a kernel gave up: its work counters may be left non-zero, so clear the whole block
        e = cudaMemset(sc->status, 0, sizeof(int) * (2 + 2 * bigbird::kCounterSlots));
        if (e != cudaSuccess) return bigbird::cuda_fail(e);
    }
    *status = host[0];
    if (detail) *detail = host[1];
    return BIGBIRD_OK;
}

int bigbird_selftest_wait_expiry(void* stream) {
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return bigbird::cuda_fail(e);
    bigbird::DeviceScratch* sc = nullptr;
    int rc = bigbird::get_scratch(device, &sc);
    if (rc != BIGBIRD_OK) return rc;
    e = bigbird::launch_wait_expiry_selftest(*sc, (cudaStream_t)stream);
    return e == cudaSuccess ? BIGBIRD_OK : bigbird::cuda_fail(e);
}

int bigbird_last_cuda_error(void) { return bigbird::t_last_cuda_error; }
int bigbird_last_launch_count(void) { return bigbird::t_last_launches; }

}  // extern "C"
