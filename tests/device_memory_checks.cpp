// csrc/device_memory.cu and the side streams of csrc/internal.h on the host, against a fake of the CUDA calls they make.  One check per run, named on
// the command line; exits 0 when it holds, else says what does not.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <chrono>
#include <map>
#include <mutex>
#include <new>
#include <string>
#include <thread>

// the allocations that are still granted
static std::atomic<long> grants{1L << 40};
void *operator new(size_t bytes)
{
    void *p = grants-- > 0 ? malloc(bytes ? bytes : 1) : nullptr;
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }

namespace fake {
struct Range {  // host memory the driver knows
    size_t bytes;
    unsigned type;
    bool mapped;
};
std::map<uintptr_t, Range> ranges;

CUresult pointer_attributes(unsigned n, CUpointer_attribute *what, void **to, CUdeviceptr at)
{
    auto it = ranges.upper_bound((uintptr_t)at);
    const bool known = it != ranges.begin() && (uintptr_t)at < (--it)->first + it->second.bytes;
    for (unsigned i = 0; i < n; ++i) {
        switch (what[i]) {
        case CU_POINTER_ATTRIBUTE_MEMORY_TYPE: *(unsigned *)to[i] = known ? it->second.type : 0; break;
        case CU_POINTER_ATTRIBUTE_IS_MANAGED: *(unsigned *)to[i] = 0; break;
        case CU_POINTER_ATTRIBUTE_DEVICE_POINTER: *(CUdeviceptr *)to[i] = known && it->second.mapped ? at : 0; break;
        case CU_POINTER_ATTRIBUTE_RANGE_START_ADDR: *(CUdeviceptr *)to[i] = known ? (CUdeviceptr)it->first : 0; break;
        case CU_POINTER_ATTRIBUTE_RANGE_SIZE: *(size_t *)to[i] = known ? it->second.bytes : 0; break;
        default: return CUDA_ERROR_INVALID_VALUE;
        }
    }
    return CUDA_SUCCESS;
}
}  // namespace fake

namespace fake {
std::string steps;  // calls that order streams
int failing = -1;   // which of them fails
cudaError_t step(const char *name)
{
    steps += std::string(steps.empty() ? "" : " ") + name;
    return failing-- == 0 ? cudaErrorUnknown : cudaSuccess;
}
std::atomic<int> allocations{0}, frees{0}, host_frees{0};  // frees: of device memory
int streams = 0;                 // alive
bool refuse_pinned = false;
thread_local int device = 0;
thread_local bool relaxed = false;
std::atomic<int> freed_on{-1};
std::atomic<bool> freed_relaxed{false};
}  // namespace fake

extern "C" {
cudaError_t cudaGetDevice(int *d) { return *d = fake::device, cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return fake::device = d, cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *mode)
{
    fake::relaxed = *mode == cudaStreamCaptureModeRelaxed;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void **out, size_t bytes) { return ++fake::allocations, *out = malloc(bytes), cudaSuccess; }
cudaError_t cudaFree(void *p)
{
    fake::freed_on = fake::device;
    fake::freed_relaxed = fake::relaxed;
    return ++fake::frees, free(p), cudaSuccess;
}
cudaError_t cudaHostAlloc(void **out, size_t bytes, unsigned)
{
    return fake::refuse_pinned ? cudaErrorMemoryAllocation : (*out = malloc(bytes), cudaSuccess);
}
cudaError_t cudaFreeHost(void *p) { return ++fake::host_frees, free(p), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return *e = (cudaEvent_t)malloc(1), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return free(e), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return ++fake::streams, *s = (cudaStream_t)malloc(1), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return --fake::streams, free(s), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return fake::step("record"); }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return fake::step("wait"); }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return fake::step("synchronize"); }
cudaError_t cudaGetDriverEntryPoint(const char *name, void **out, unsigned long long, cudaDriverEntryPointQueryResult *found)
{
    const bool known = !strcmp(name, "cuPointerGetAttributes");
    *out = known ? (void *)fake::pointer_attributes : nullptr;
    *found = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
}

#include "device_memory.cu"

#define CHECK(x)                                              \
    do {                                                      \
        if (!(x)) {                                           \
            printf("line %d: %s does not hold\n", __LINE__, #x); \
            return 1;                                         \
        }                                                     \
    } while (0)

using namespace accerl;

// a range counts as the device's only when all of it lies in one known, mapped piece of host memory
static int reach()
{
    alignas(4096) static char memory[16384];
    const uintptr_t m = (uintptr_t)memory;
    CHECK(!device_reaches(memory, 64));
    fake::ranges[m] = {4096, CU_MEMORYTYPE_HOST, true};
    fake::ranges[m + 8192] = {4096, CU_MEMORYTYPE_HOST, true};
    CHECK(device_reaches(memory, 4096) && device_reaches(memory + 4092, 4) && device_reaches(memory + 8192, 64));
    CHECK(!device_reaches(memory + 4092, 8));
    CHECK(!device_reaches(memory, 8192 + 64));  // both ends known, pageable memory between them
    CHECK(!device_reaches(memory + 64, 8192));
    CHECK(!device_reaches(memory + 2, 4));
    fake::ranges[m + 8192].mapped = false;
    CHECK(!device_reaches(memory + 8192, 64));
    fake::ranges[m].type = CU_MEMORYTYPE_DEVICE;
    CHECK(!device_reaches(memory, 64));
    return 0;
}

// what is given back idle serves the next allocation; what may still be in use goes back to the driver
static int busy()
{
    void *a = nullptr, *b = nullptr;
    CHECK(device_alloc(&a, 100000) == cudaSuccess && fake::allocations == 1);
    device_free(a, true);
    CHECK(fake::frees == 0);
    CHECK(device_alloc(&b, 100000) == cudaSuccess && b == a && fake::allocations == 1);
    device_free(b, false);
    CHECK(fake::frees == 1);
    CHECK(device_alloc(&a, 100000) == cudaSuccess && fake::allocations == 2);
    device_free(a, true);
    device_free(nullptr, false);
    SideStream s;
    CHECK(take_side_stream(&s) == cudaSuccess && fake::streams == 1);
    give_side_stream(s, false);
    CHECK(fake::streams == 0 && !s.stream);
    CHECK(take_side_stream(&s) == cudaSuccess);
    give_side_stream(s, true);
    CHECK(fake::streams == 1 && take_side_stream(&s) == cudaSuccess && fake::streams == 1);
    return 0;
}

// where the driver grants no pinned memory, parameters travel in ordinary memory
static int pageable()
{
    std::shared_ptr<char[]> a, b;
    fake::refuse_pinned = true;
    CHECK(pinned_alloc(&a, 5000) == cudaSuccess && a);
    memset(a.get(), 1, 5000);
    CHECK(pinned_alloc(&b, 0) == cudaSuccess && b);
    a.reset();
    fake::refuse_pinned = false;
    CHECK(pinned_alloc(&a, 5000) == cudaSuccess && a);
    return 0;
}

// host memory that runs out anywhere on the way fails the call or drops the block, and throws nothing
static int hungry()
{
    void *first = nullptr;
    for (long n = 0; n < 12; ++n) {
        void *a = nullptr, *b = nullptr;
        std::shared_ptr<char[]> h;
        SideStream s;
        grants = n;
        const cudaError_t ea = device_alloc(&a, 1000), eb = device_alloc(&b, 5 << 20), eh = pinned_alloc(&h, 1000);
        CHECK((ea == cudaSuccess) == (a != nullptr) && (eb == cudaSuccess) == (b != nullptr) && (eh == cudaSuccess) == !!h);
        CHECK(ea == cudaSuccess || ea == cudaErrorMemoryAllocation);
        CHECK(take_side_stream(&s) == cudaSuccess);
        device_free(a, true);
        device_free(b, true);
        h.reset();
        give_side_stream(s, true);
        grants = 1L << 40;
    }
    CHECK(device_alloc(&first, 1000) == cudaSuccess);
    return 0;
}

static bool soon(const std::atomic<int> &count, int value)
{
    for (int i = 0; i < 100 && count != value; ++i) std::this_thread::sleep_for(std::chrono::milliseconds(20));
    return count == value;
}

// what lies idle goes back without another call of the library, on its own device and outside any capture's
// rules; twice, since the thread that does it ends in between
static int idle()
{
    using std::chrono::milliseconds;
    for (int round = 1; round <= 2; ++round) {
        void *a = nullptr, *b = nullptr;
        std::shared_ptr<char[]> h;
        fake::device = 3;
        CHECK(device_alloc(&a, 100000) == cudaSuccess && device_alloc(&b, 9 << 20) == cudaSuccess && pinned_alloc(&h, 1000) == cudaSuccess);
        device_free(a, true);
        h.reset();
        fake::device = 0;
        CHECK(fake::frees == 2 * (round - 1) && fake::host_frees == round - 1);
        CHECK(soon(fake::frees, 2 * round - 1) && soon(fake::host_frees, round));
        CHECK(fake::freed_on == 3 && fake::freed_relaxed && fake::device == 0);
        std::this_thread::sleep_for(milliseconds(3 * ACCERL_KEEP_IDLE_MS));
        CHECK(fake::frees == 2 * round - 1);  // (b is in use)
        device_free(b, false);
    }
    return 0;
}

// used blocks do not age: what is given back again and again stays
static int in_use()
{
    for (int i = 0; i < 30; ++i) {
        void *a = nullptr;
        CHECK(device_alloc(&a, 100000) == cudaSuccess);
        std::this_thread::sleep_for(std::chrono::milliseconds(ACCERL_KEEP_IDLE_MS / 10));
        device_free(a, true);
    }
    CHECK(fake::allocations == 1 && fake::frees == 0);
    return 0;
}

// accerl_trim
static int trim()
{
    void *a = nullptr, *b = nullptr, *c = nullptr;
    std::shared_ptr<char[]> h;
    SideStream s;
    CHECK(device_alloc(&a, 100000) == cudaSuccess && device_alloc(&b, 9 << 20) == cudaSuccess && pinned_alloc(&h, 1000) == cudaSuccess);
    CHECK(take_side_stream(&s) == cudaSuccess && device_alloc(&c, 5000) == cudaSuccess);
    device_free(a, true);
    device_free(b, true);
    h.reset();
    give_side_stream(s, true);
    CHECK(fake::frees == 0 && fake::streams == 1);
    release_kept();
    CHECK(fake::frees == 2 && fake::host_frees == 1 && fake::streams == 0);
    release_kept();
    CHECK(fake::frees == 2);
    device_free(c, true);
    CHECK(device_alloc(&a, 5000) == cudaSuccess && a == c);
    return 0;
}

// a side stream that work was launched on is always waited for, whichever call fails
static int side()
{
    SideStream s;
    CHECK(take_side_stream(&s) == cudaSuccess);
    const char *want[5] = {"record", "record wait", "record wait record synchronize", "record wait record wait synchronize",
                           "record wait record wait"};
    for (int returns_early = 0; returns_early < 2; ++returns_early)
        for (int i = 0; i < 5; ++i) {
            fake::steps.clear();
            fake::failing = i;
            {
                SideWork work(nullptr, s);
                const cudaError_t e = work.begin();
                CHECK((e == cudaSuccess) == (i >= 2));
                if (e == cudaSuccess && !returns_early) CHECK((work.join() == cudaSuccess) == (i >= 4));
            }
            CHECK(fake::steps == want[i]);
        }
    return 0;
}

int main(int argc, char **argv)
{
    const std::string name = argc > 1 ? argv[1] : "";
    if (name == "reach") return reach();
    if (name == "busy") return busy();
    if (name == "pageable") return pageable();
    if (name == "hungry") return hungry();
    if (name == "idle") return idle();
    if (name == "in_use") return in_use();
    if (name == "trim") return trim();
    if (name == "side") return side();
    printf("no check %s\n", name.c_str());
    return 2;
}
