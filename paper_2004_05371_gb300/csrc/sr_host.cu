// sr_reduce_sum_host: the sum of an array in HOST memory, result to host.
//
// The input streams to the device in chunks through two staging buffers, on
// two copy streams (both copy engines), while the caller's stream reduces the
// chunk that already arrived: each chunk's units write their partials into
// their own range of the workspace slots (the first kernel of the two-kernel
// form), and one final kernel reduces all slots in order.  Copy of chunk k+1
// overlaps the reduction of chunk k.
//
// A page-locked array of at most two chunks, within one allocation or registration, is
// read in place by one kernel instead: with so little to overlap, the copy, its events and the launches after it
// cost more than they hide (link 210 GB/s either way; pipeline / in place, us:
// 4 KiB 23 / 16, 1 MiB 31 / 21, 16 MiB 112 / 97, 64 MiB 353 / 335, 128 MiB 676 / 653).  Above, the
// pipeline stays within 2 % and leaves the SMs to other streams.
//
// The result is written by the kernel into page-locked memory of the library's
// (a copy back to the device's caller took another 8 us).
#include <algorithm>
#include <condition_variable>
#include <cstring>
#include <map>
#include <mutex>
#include <utility>

#include <cuda.h>  // types of the driver's pointer query (fetched at run time)

#include "sr_hostrange.h"
#include "sr_internal.h"

namespace sr {
namespace {

constexpr size_t kChunkBytes = 64u << 20;
constexpr size_t kInPlaceBytes = 2 * kChunkBytes;  // page-locked arrays up to here are read in place
constexpr int kResultSlots = 64;  // 64 bytes apart; a call holds one until its value is copied out

struct HostPipe {
    unsigned char* stage[2] = {nullptr, nullptr};
    cudaStream_t copy[2] = {nullptr, nullptr};
    cudaEvent_t copied[2] = {nullptr, nullptr};
    cudaEvent_t consumed[2] = {nullptr, nullptr};
    size_t chunk = 0;
    unsigned char* result = nullptr;  // kResultSlots page-locked slots, host and device address alike
    uint64_t busy = 0;                // slots held (under g_hp_mu)
    std::condition_variable freed;
    std::mutex copying;               // held by the call that uses the staging buffers and events
};

std::mutex g_hp_mu;
std::map<std::pair<int, cudaStream_t>, HostPipe> g_pipes;

// The pair's pipe with its result slots, and (chunk > 0) staging for chunks of that size.
int get_pipe(cudaStream_t s, size_t chunk, HostPipe** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return status_from_cuda(e);
    std::lock_guard<std::mutex> lk(g_hp_mu);
    HostPipe& p = g_pipes[std::make_pair(dev, s)];
    *out = &p;
    if (!p.result) {
        void* h = nullptr;
        e = cudaHostAlloc(&h, kResultSlots * 64, cudaHostAllocMapped);
        if (e != cudaSuccess) return status_from_cuda(e);
        p.result = static_cast<unsigned char*>(h);
    }
    if (chunk == 0) return SR_OK;  // in place: nothing to stage
    if (p.chunk < chunk) {
        for (int b = 0; b < 2; ++b) {
            if (p.stage[b]) cudaFree(p.stage[b]);
            p.stage[b] = nullptr;
        }
        for (int b = 0; b < 2; ++b) {
            e = cudaMalloc(&p.stage[b], chunk);
            if (e != cudaSuccess) {
                p.chunk = 0;
                return status_from_cuda(e);
            }
        }
        p.chunk = chunk;
    }
    for (int b = 0; b < 2; ++b) {
        if (!p.copy[b]) {
            e = cudaStreamCreateWithFlags(&p.copy[b], cudaStreamNonBlocking);
            if (e != cudaSuccess) return status_from_cuda(e);
        }
        if (!p.copied[b]) {
            e = cudaEventCreateWithFlags(&p.copied[b], cudaEventDisableTiming);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p.consumed[b], cudaEventDisableTiming);
            if (e != cudaSuccess) return status_from_cuda(e);
        }
    }
    return SR_OK;
}

}  // namespace

void release_host_pipe(cudaStream_t s) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    std::lock_guard<std::mutex> lk(g_hp_mu);
    auto it = g_pipes.find(std::make_pair(dev, s));
    if (it == g_pipes.end()) return;
    HostPipe& p = it->second;
    for (int b = 0; b < 2; ++b) {
        if (p.copy[b]) cudaStreamSynchronize(p.copy[b]);
        if (p.stage[b]) cudaFree(p.stage[b]);
        if (p.copy[b]) cudaStreamDestroy(p.copy[b]);
        if (p.copied[b]) cudaEventDestroy(p.copied[b]);
        if (p.consumed[b]) cudaEventDestroy(p.consumed[b]);
    }
    if (p.result) cudaFreeHost(p.result);
    g_pipes.erase(it);
}

}  // namespace sr

using namespace sr;

namespace {

// A result slot of the pipe, this call's alone until it returns: with more calls than slots
// blocked on one stream, the others wait for one (before, they took the slots in turn, and
// an earlier call could find a later one's sum in its own).
class ResultSlot {
public:
    explicit ResultSlot(HostPipe* hp) : hp_(hp) {
        std::unique_lock<std::mutex> lk(g_hp_mu);
        hp_->freed.wait(lk, [&] { return ~hp_->busy != 0; });
        for (k_ = 0; (hp_->busy >> k_) & 1; ++k_) {
        }
        hp_->busy |= uint64_t(1) << k_;
        host = hp_->result + 64 * (size_t)k_;
        const cudaError_t e = cudaHostGetDevicePointer(&dev, host, 0);
        status = e == cudaSuccess ? SR_OK : status_from_cuda(e);
    }
    ~ResultSlot() {
        {
            std::lock_guard<std::mutex> lk(g_hp_mu);
            hp_->busy &= ~(uint64_t(1) << k_);
        }
        hp_->freed.notify_one();
    }
    ResultSlot(const ResultSlot&) = delete;
    ResultSlot& operator=(const ResultSlot&) = delete;

    unsigned char* host = nullptr;
    void* dev = nullptr;
    int status = SR_OK;

private:
    HostPipe* hp_;
    int k_ = 0;
};
static_assert(kResultSlots == 64, "one bit per slot");

// A driver function by name (nullptr where there is none).
template <class Fn> Fn driver_function(const char* name) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult r;
    if (cudaGetDriverEntryPointByVersion(name, &f, 12000, cudaEnableDefault, &r) != cudaSuccess ||
        r != cudaDriverEntryPointSuccess) {
        cudaGetLastError();
        f = nullptr;
    }
    return reinterpret_cast<Fn>(f);
}

// The driver's view of one host address (no page-locked memory where it has none to give).
HostRange query_host(uintptr_t at) {
    static const auto get =
        driver_function<CUresult (*)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr)>("cuPointerGetAttributes");
    static const auto current = driver_function<CUresult (*)(CUcontext*)>("cuCtxGetCurrent");
    HostRange h;
    if (!get || !current) return h;
    // The driver answers only with a context current: a thread's first calls of the runtime
    // need not have made one so (with one, it stays the caller's).
    CUcontext ctx = nullptr;
    int dev = 0;
    if (current(&ctx) != CUDA_SUCCESS) return h;
    cudaPointerAttributes a;
    if ((!ctx && (cudaGetDevice(&dev) != cudaSuccess || cudaSetDevice(dev) != cudaSuccess)) ||
        cudaPointerGetAttributes(&a, reinterpret_cast<const void*>(at)) != cudaSuccess) {
        cudaGetLastError();
        return h;
    }
    if (a.type != cudaMemoryTypeHost || !a.devicePointer) return h;
    CUdeviceptr start = 0;
    size_t size = 0;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* data[] = {&start, &size};
    if (get(2, what, data, (CUdeviceptr)at) != CUDA_SUCCESS) return h;
    h.page_locked = true;
    h.start = (uintptr_t)start;
    h.size = size;
    h.device = reinterpret_cast<uintptr_t>(a.devicePointer);
    return h;
}

// The reduction reads the host array in place (no staging copies).
int host_direct(const void* host_x, int64_t n, int dtype, void* host_out, sr_config c, sr_stream_t stream) {
    const int stage = c.variant & SR_STAGE_MASK;
    if ((stage != SR_AUTO && stage != SR_LAST_BLOCK) || (c.variant & SR_F_BULK)) return SR_ERR_UNSUPPORTED;
    c.variant = (c.variant & ~(SR_STAGE_MASK | SR_F_HOST_DIRECT)) | SR_LAST_BLOCK;
    const void* fake_out = reinterpret_cast<const void*>(uintptr_t(1) << 20);
    int st = reduce_validate(host_x, n, dtype, fake_out, c);
    if (st != SR_OK) return st;
    const DeviceInfo* d = current_device(&st);
    if (!d) return st;
    const void* dx = host_x;
    if (n > 0) {
        cudaPointerAttributes a;
        cudaError_t e = cudaPointerGetAttributes(&a, host_x);
        if (e != cudaSuccess) return status_from_cuda(e);
        if (a.type == cudaMemoryTypeHost) {
            void* mapped = nullptr;
            e = cudaHostGetDevicePointer(&mapped, const_cast<void*>(host_x), 0);
            if (e != cudaSuccess) return status_from_cuda(e);
            dx = mapped;
        } else if (a.type == cudaMemoryTypeUnregistered) {
            int pageable = 0;
            e = cudaDeviceGetAttribute(&pageable, cudaDevAttrPageableMemoryAccess, d->dev);
            if (e != cudaSuccess) return status_from_cuda(e);
            if (!pageable) return SR_ERR_UNSUPPORTED;
        } else {
            return SR_ERR_ARG;  // device or managed memory: use sr_reduce_sum_ex
        }
    }
    Plan p;
    cudaStream_t s = (cudaStream_t)stream;
    st = reduce_plan(dx, n, dtype, c, *d, &p);
    if (st != SR_OK) return st;
    Workspace ws;
    st = get_workspace(s, &ws);
    if (st != SR_OK) return st;
    HostPipe* hp = nullptr;
    st = get_pipe(s, 0, &hp);
    if (st != SR_OK) return st;
    ResultSlot slot(hp);
    if (slot.status != SR_OK) return slot.status;
    st = reduce_launch(dx, slot.dev, p, *d, ws, s);
    if (st != SR_OK) return st;
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return status_from_cuda(e);
    std::memcpy(host_out, slot.host, (dtype == SR_I32 || p.fp64) ? 8 : 4);
    return SR_OK;
}

}  // namespace

extern "C" int sr_reduce_sum_host(const void* host_x, int64_t n, int dtype, void* host_out, const sr_config* cfg,
                                  sr_stream_t stream) {
    sr_config c;
    std::memset(&c, 0, sizeof c);
    if (cfg) c = *cfg;
    if (host_out == nullptr) return SR_ERR_ARG;
    if (c.variant & SR_F_HOST_DIRECT) return host_direct(host_x, n, dtype, host_out, c, stream);
    const int stage = c.variant & SR_STAGE_MASK;
    if (stage != SR_AUTO && stage != SR_TWO_KERNEL) return SR_ERR_UNSUPPORTED;
    if (c.variant & SR_F_BULK) return SR_ERR_UNSUPPORTED;
    c.variant = (c.variant & ~SR_STAGE_MASK) | SR_TWO_KERNEL;
    // validate with a device-style stand-in for out (the host result is copied)
    const void* fake_out = reinterpret_cast<const void*>(uintptr_t(1) << 20);
    int st = reduce_validate(host_x, n, dtype, fake_out, c);
    if (st != SR_OK) return st;
    const DeviceInfo* d = current_device(&st);
    if (!d) return st;
    cudaStream_t s = (cudaStream_t)stream;
    Workspace ws;
    st = get_workspace(s, &ws);
    if (st != SR_OK) return st;
    const int es = elem_size(dtype);
    const size_t bytes = (size_t)n * es;
    if (stage == SR_AUTO && bytes > 0 && bytes <= kInPlaceBytes &&
        one_page_locked_range(reinterpret_cast<uintptr_t>(host_x), bytes, query_host)) {
        c.variant &= ~SR_STAGE_MASK;
        return host_direct(host_x, n, dtype, host_out, c, stream);
    }
    size_t chunk = kChunkBytes;
    // at most kMaxUnits partial slots in total: bigger chunks for huge inputs
    const int64_t max_chunks = kMaxUnits / (8 * d->sms);
    if ((int64_t)((bytes + chunk - 1) / chunk) > max_chunks) {
        chunk = (bytes + max_chunks - 1) / max_chunks;
        chunk = (chunk + (1u << 20) - 1) & ~((size_t)(1u << 20) - 1);
    }
    // One call at a time copies through a stream's staging buffers: with two, the second
    // one's copies, which its own stream orders behind nothing, overwrote the first one's.
    HostPipe* hp = nullptr;
    st = get_pipe(s, 0, &hp);
    if (st != SR_OK) return st;
    std::lock_guard<std::mutex> copying(hp->copying);
    st = get_pipe(s, chunk, &hp);
    if (st != SR_OK) return st;

    const bool fp64 = (c.variant & SR_F_FP64_COMBINE) && dtype != SR_I32;
    ResultSlot result(hp);
    if (result.status != SR_OK) return result.status;
    int slot = 0;
    Plan last;
    bool have_plan = false;
    const unsigned char* hx = static_cast<const unsigned char*>(host_x);
    const size_t per_chunk = chunk / es;  // elements per chunk (chunk is a multiple of 16 B)
    for (size_t k = 0, off = 0; off < bytes || k == 0; ++k, off += chunk) {
        const int b = (int)(k & 1);
        const size_t len = std::min(chunk, bytes - off);
        const int64_t nk = (int64_t)(len / es);
        cudaError_t e;
        if (k >= 2) {
            e = cudaStreamWaitEvent(hp->copy[b], hp->consumed[b], 0);
            if (e != cudaSuccess) return status_from_cuda(e);
        }
        if (len) {
            e = cudaMemcpyAsync(hp->stage[b], hx + off, len, cudaMemcpyHostToDevice, hp->copy[b]);
            if (e != cudaSuccess) return status_from_cuda(e);
        }
        e = cudaEventRecord(hp->copied[b], hp->copy[b]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, hp->copied[b], 0);
        if (e != cudaSuccess) return status_from_cuda(e);
        Plan p;
        st = reduce_plan(hp->stage[b], nk, dtype, c, *d, &p);
        if (st != SR_OK) return st;
        if (slot + p.units > kMaxUnits) return SR_ERR_ARG;
        Workspace wk = ws;
        wk.partials = ws.partials + (size_t)slot * kSlotBytes;
        st = reduce_launch(hp->stage[b], result.dev, p, *d, wk, s, /*skip_final=*/true);
        if (st != SR_OK) return st;
        slot += p.units;
        last = p;
        have_plan = true;
        e = cudaEventRecord(hp->consumed[b], s);
        if (e != cudaSuccess) return status_from_cuda(e);
        (void)per_chunk;
        if (len == 0) break;
    }
    if (!have_plan) return SR_ERR_ARG;
    st = reduce_launch_final(last, slot, result.dev, ws, s);
    if (st != SR_OK) return st;
    const cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return status_from_cuda(e);
    std::memcpy(host_out, result.host, (dtype == SR_I32 || fp64) ? 8 : 4);
    return SR_OK;
}
