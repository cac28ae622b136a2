// Device memory of the library.  cudaMalloc and cudaFree map and unmap memory through the kernel driver:
// a fraction of a millisecond each on a quiet machine, tens to hundreds when other processes of the host
// do the same, and a Compressor that hands over a new policy every few seconds pays for a dozen of them
// each time (building and calibrating the residual network: 9 ms at best, 20 to 300 on a busy host).
// So blocks that policies give back are kept for the next one: at most kKept bytes per process, none for
// longer than kIdle without use, and all of them are returned to the driver when an allocation fails or the
// caller asks (accerl_trim).  A thread that exists only while something is kept returns what has lain idle:
// a process that builds a policy and then only steps it makes no call that could.  Blocks are handed back
// only when nothing on the device uses them any more, so any thread and any stream may have them next.
//
// Running out of host memory for the bookkeeping is an allocation that fails, or a block that is not kept:
// nothing here throws.
//
// Pinned host memory for parameters on their way to the device and quantised ones on their way back is
// kept in the same manner (at most kKeptHost bytes): pageable blocks of that size are fresh pages for
// every policy, 0.4 ms of faults each, and copies from and to them are staged by the driver.
#include <cuda.h>

#include <algorithm>
#include <chrono>
#include <list>
#include <mutex>
#include <new>
#include <thread>
#include <unordered_map>

#include "internal.h"

namespace accerl {

namespace {

constexpr size_t kKept = (size_t)512 << 20;
constexpr size_t kKeptHost = (size_t)64 << 20;
#ifndef ACCERL_KEEP_IDLE_MS
#define ACCERL_KEEP_IDLE_MS 30000
#endif
constexpr std::chrono::milliseconds kIdle(ACCERL_KEEP_IDLE_MS);
constexpr int kHost = -1;  // in place of a device

struct Piece {
    size_t bytes;
    int device;  // or kHost
    int current; // the device that was current when it was allocated
};
struct Block : Piece {
    void *ptr;
    std::chrono::steady_clock::time_point since;
};

struct Memory {
    std::mutex mu;
    std::list<Block> kept;  // oldest first
    size_t kept_bytes = 0, kept_host_bytes = 0;
    std::unordered_map<void *, Piece> live;  // every block handed out
    bool watched = false;                    // the thread that ends what is idle runs

    size_t &bytes_of(int device) { return device == kHost ? kept_host_bytes : kept_bytes; }
    Block pop(std::list<Block>::iterator it)
    {
        const Block b = *it;
        bytes_of(b.device) -= b.bytes;
        kept.erase(it);
        return b;
    }
    static void release(void *ptr, int device)
    {
        if ((device == kHost ? cudaFreeHost(ptr) : cudaFree(ptr)) != cudaSuccess) cudaGetLastError();
    }
    static cudaError_t fresh(void **out, size_t bytes, int device)
    {
        return device == kHost ? cudaHostAlloc(out, bytes, cudaHostAllocPortable) : cudaMalloc(out, bytes);
    }
    cudaError_t take(void **out, size_t bytes, int device, int current);
    void give(void *ptr, bool idle);
    void release_all();
    bool watch();
    void end_idle();
};

Memory &memory()
{
    alignas(Memory) static char room[sizeof(Memory)];
    static Memory *m = new (room) Memory;  // (never destroyed: the driver may be gone before static objects are)
    return *m;
}

// side streams not in use (creating one, with its events, takes a tenth of a millisecond)
constexpr size_t kKeptStreams = 8;
std::mutex g_stream_mu;
SideStream g_streams[kKeptStreams];
size_t g_n_streams = 0;
void destroy(SideStream &s)
{
    for (cudaEvent_t ev : s.events) cudaEventDestroy(ev);
    cudaStreamDestroy(s.stream);
    s = SideStream();
}

}  // namespace

cudaError_t take_side_stream(SideStream *out)
{
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lock(g_stream_mu);
        for (size_t i = 0; i < g_n_streams; ++i)
            if (g_streams[i].device == device) {
                *out = g_streams[i];
                g_streams[i] = g_streams[--g_n_streams];
                return cudaSuccess;
            }
    }
    SideStream s;
    s.device = device;
    for (cudaEvent_t &ev : s.events)
        if ((e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess) break;
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&s.stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) {
        *out = s;
        return e;
    }
    for (cudaEvent_t ev : s.events)
        if (ev) cudaEventDestroy(ev);
    return e;
}

void give_side_stream(SideStream &s, bool idle)
{
    if (!s.stream) return;
    if (idle) {
        std::lock_guard<std::mutex> lock(g_stream_mu);
        if (g_n_streams < kKeptStreams) {
            g_streams[g_n_streams++] = s;
            s = SideStream();
            return;
        }
    }
    destroy(s);
}

cudaError_t Memory::take(void **out, size_t bytes, int device, int current)
{
    *out = nullptr;
    bytes = std::max<size_t>(bytes, 1);
    const size_t grain = bytes < ((size_t)1 << 20) ? (size_t)64 << 10 : (size_t)2 << 20;
    const size_t want = (bytes + grain - 1) / grain * grain;
    std::lock_guard<std::mutex> lock(mu);
    auto best = kept.end();  // the smallest kept block that is not much too large
    for (auto it = kept.begin(); it != kept.end(); ++it)
        if (it->device == device && it->bytes >= want && it->bytes <= want + want / 2 + grain &&
            (best == kept.end() || it->bytes < best->bytes))
            best = it;
    auto handed_out = [&](void *ptr, const Piece &piece) {
        try {
            live[ptr] = piece;
            return true;
        } catch (const std::bad_alloc &) {
            return false;
        }
    };
    if (best != kept.end()) {
        if (!handed_out(best->ptr, *best)) return cudaErrorMemoryAllocation;
        *out = pop(best).ptr;
        return cudaSuccess;
    }
    cudaError_t e = fresh(out, want, device);
    if (e == cudaErrorMemoryAllocation && !kept.empty()) {
        cudaGetLastError();
        release_all();
        e = fresh(out, want, device);
    }
    if (e == cudaSuccess && !handed_out(*out, Piece{want, device, current})) {
        release(*out, device);
        *out = nullptr;
        e = cudaErrorMemoryAllocation;
    }
    return e;
}

void Memory::give(void *ptr, bool idle)
{
    if (!ptr) return;
    std::lock_guard<std::mutex> lock(mu);
    const auto it = live.find(ptr);
    if (it == live.end()) return;
    const Piece piece = it->second;
    live.erase(it);
    const size_t limit = piece.device == kHost ? kKeptHost : kKept;
    if (!idle || piece.bytes > limit || !watch()) {
        release(ptr, piece.device);
        return;
    }
    try {
        kept.push_back(Block{piece, ptr, std::chrono::steady_clock::now()});
    } catch (const std::bad_alloc &) {
        release(ptr, piece.device);
        return;
    }
    bytes_of(piece.device) += piece.bytes;
    for (auto at = kept.begin(); bytes_of(piece.device) > limit; ) {  // the oldest of its kind
        const auto next = std::next(at);
        if ((at->device == kHost) == (piece.device == kHost)) {
            const Block b = pop(at);
            release(b.ptr, b.device);
        }
        at = next;
    }
}

void Memory::release_all()
{
    int before = 0;
    const bool back = cudaGetDevice(&before) == cudaSuccess;
    while (!kept.empty()) {
        const Block b = pop(kept.begin());
        if (cudaSetDevice(b.current) == cudaSuccess) release(b.ptr, b.device);
    }
    if (back) cudaSetDevice(before);
}

// the thread for end_idle, if it is not there; false: there can be none
bool Memory::watch()
{
    if (watched) return true;
    try {
        std::thread([this] { end_idle(); }).detach();
        watched = true;
    } catch (const std::exception &) {
    }
    return watched;
}

void Memory::end_idle()
{
    // (a free on this thread is none of a capture's business: nothing that is kept is used by any)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    std::unique_lock<std::mutex> lock(mu);
    while (!kept.empty()) {
        const auto due = kept.front().since + kIdle;
        if (std::chrono::steady_clock::now() < due) {
            lock.unlock();
            std::this_thread::sleep_until(due);
            lock.lock();
            continue;
        }
        const Block b = pop(kept.begin());
        lock.unlock();
        if (cudaSetDevice(b.current) == cudaSuccess) release(b.ptr, b.device);  // (else the process ends)
        lock.lock();
    }
    watched = false;
}

cudaError_t device_alloc(void **out, size_t bytes)
{
    *out = nullptr;
    int device = 0;
    const cudaError_t e = cudaGetDevice(&device);
    return e == cudaSuccess ? memory().take(out, bytes, device, device) : e;
}

void release_kept()
{
    {
        std::lock_guard<std::mutex> lock(memory().mu);
        memory().release_all();
    }
    std::lock_guard<std::mutex> lock(g_stream_mu);
    while (g_n_streams) destroy(g_streams[--g_n_streams]);
}

void device_free(void *ptr, bool idle) { memory().give(ptr, idle); }

cudaError_t pinned_alloc(std::shared_ptr<char[]> *out, size_t bytes)
{
    void *ptr = nullptr;
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = memory().take(&ptr, bytes, kHost, device);
    try {
        if (e == cudaSuccess) {  // (where the shared pointer cannot be made, it gives the block back itself)
            *out = std::shared_ptr<char[]>((char *)ptr, [](char *at) { memory().give(at, true); });
            return e;
        }
        // pageable memory serves as well: the driver stages its copies
        cudaGetLastError();
        *out = std::shared_ptr<char[]>(new char[std::max<size_t>(bytes, 1)]);
        return cudaSuccess;
    } catch (const std::bad_alloc &) {
        return cudaErrorMemoryAllocation;
    }
}

// Pinned and mapped, 4-byte aligned, and all of it inside one allocation or registration: with its two ends in
// different ones there may be pageable memory between them.
bool device_reaches(const void *host, size_t bytes)
{
    if ((uintptr_t)host & 3) return false;
    typedef CUresult (*Query)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);
    static const Query query = [] {
        void *sym = nullptr;
        cudaDriverEntryPointQueryResult found;
        const bool ok = cudaGetDriverEntryPoint("cuPointerGetAttributes", &sym, cudaEnableDefault, &found) == cudaSuccess &&
                        found == cudaDriverEntryPointSuccess;
        return ok ? (Query)sym : (Query) nullptr;
    }();
    if (!query) return false;
    unsigned type = 0, managed = 0;  // (stays 0 for memory the driver does not know)
    CUdeviceptr device = 0, start = 0;
    size_t size = 0;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                  CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void *to[] = {&type, &managed, &device, &start, &size};
    if (query(5, what, to, (CUdeviceptr)host) != CUDA_SUCCESS) return false;
    const CUdeviceptr at = (CUdeviceptr)host;
    return type == CU_MEMORYTYPE_HOST && !managed && device == at && start && start <= at && at - start <= size &&
           bytes <= size - (at - start);
}

}  // namespace accerl
