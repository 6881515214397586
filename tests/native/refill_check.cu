// Host-only driver of plans that are refilled: includes the library's batch.cu
// with the CUDA runtime calls it makes replaced by stand-ins ("device" memory
// is host memory), makes a plan, captures its launch, refills it and looks at
// what a replay of the captured launch would run.
// Input: "before rows n_items", then the items' stream counts; before = 1: the
// plan is refilled once, with the same items, before the launch is captured.
// before = 2 "rows n_items fewer rows_then" then the counts: no launch is captured
// and the plan is refilled with the first `fewer` items at rows_then rows each;
// the records are left out.
// Output: "shape" and "tiles" of the plan when captured and after the refill,
// "allocs" of device memory by the refill, then per record that the replay
// takes "item mode s0 streams new" (streams: how many a CTA of the captured
// size covers; new: whether the record writes to the new outputs).
#include <cinttypes>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include <cuda_runtime.h>

namespace fake {
int allocs = 0;
bool capturing = false;
template <class T>
cudaError_t alloc(T **p, size_t bytes)
{
    *p = static_cast<T *>(std::calloc(bytes, 1));
    ++allocs;
    return cudaSuccess;
}
template <class T>
cudaError_t host_alloc(T **p, size_t bytes, unsigned)
{
    *p = static_cast<T *>(std::calloc(bytes, 1));
    return cudaSuccess;
}
cudaError_t release(void *) { return cudaSuccess; }  // a replay may still read it
cudaError_t copy(void *to, const void *from, size_t bytes)
{
    std::memcpy(to, from, bytes);
    return cudaSuccess;
}
cudaError_t ok() { return cudaSuccess; }
cudaError_t device(int *d) { return *d = 0, cudaSuccess; }
cudaError_t attribute(int *v) { return *v = 152, cudaSuccess; }
template <class Kernel>
cudaError_t occupancy(int *fit, Kernel, int, size_t)
{
    return *fit = 4, cudaSuccess;
}
cudaError_t capture_status(cudaStreamCaptureStatus *s)
{
    *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t event(cudaEvent_t *e)
{
    static int any;
    *e = reinterpret_cast<cudaEvent_t>(&any);
    return cudaSuccess;
}
}  // namespace fake

#define cudaMalloc fake::alloc
#define cudaHostAlloc fake::host_alloc
#define cudaFree fake::release
#define cudaFreeHost fake::release
#define cudaMemcpy(to, from, bytes, kind) fake::copy(to, from, bytes)
#define cudaMemcpyAsync(to, from, bytes, kind, stream) fake::copy(to, from, bytes)
#define cudaMemsetAsync(to, value, bytes, stream) fake::ok()
#define cudaGetDevice fake::device
#define cudaSetDevice(d) fake::ok()
#define cudaDeviceGetAttribute(v, what, d) fake::attribute(v)
#define cudaStreamIsCapturing(stream, status) fake::capture_status(status)
#define cudaEventCreateWithFlags(e, flags) fake::event(e)
#define cudaEventSynchronize(e) fake::ok()
#define cudaEventRecord(e, stream) fake::ok()
#define cudaStreamSynchronize(stream) fake::ok()
#define cudaGetLastError() fake::ok()
#define cudaOccupancyMaxActiveBlocksPerMultiprocessor fake::occupancy

#include "batch.cu"

namespace gbrng {
int set_error(int status) { return status; }
int cuda_status(cudaError_t e) { return e == cudaSuccess ? 0 : RNG_ERR_CUDA; }
int one_cta_smem(const void *, int) { return 0; }
}  // namespace gbrng
extern "C" int rng_last_error(void) { return 0; }

int main()
{
    using namespace gbrng;
    // the launches name host memory: they must not find a GPU
    setenv("CUDA_VISIBLE_DEVICES", "", 1);
    int before = 0;
    uint64_t rows = 0;
    size_t n_items = 0;
    size_t fewer = 0;
    uint64_t rows_then = 0;
    if (std::scanf("%d %" SCNu64 " %zu", &before, &rows, &n_items) != 3 ||
        (before == 2 && std::scanf("%zu %" SCNu64, &fewer, &rows_then) != 2))
        return 2;
    std::vector<Gen> gens(n_items);
    // stand-in addresses: a place for every item's output, the new ones above
    uint32_t *const base = reinterpret_cast<uint32_t *>(uintptr_t{1} << 48);
    const uint64_t step = uint64_t{1} << 32, fresh = uint64_t{1} << 44;
    auto items_at = [&](uint64_t offset) {
        std::vector<rng_batch_item> items(n_items);
        for (size_t i = 0; i < n_items; ++i)
            items[i] = rng_batch_item{reinterpret_cast<rng_handle>(&gens[i]), rows,
                                      base + offset + i * step, 0, 0, 0, 0};
        return items;
    };
    for (size_t i = 0; i < n_items; ++i) {
        if (std::scanf("%" SCNu64, &gens[i].n) != 1)
            return 2;
        gens[i].kind = RNG_KISS;
        gens[i].d_state = reinterpret_cast<uint32_t *>((uintptr_t)(i + 1) << 32);
    }
    const auto old_items = items_at(0), new_items = items_at(fresh);
    rng_plan_handle plan = rng_plan_create(old_items.data(), n_items, 0, 0);
    if (!plan || (before == 1 && rng_plan_refill(plan, old_items.data(), n_items, nullptr)))
        return 1;
    auto report = [&](const Plan &p) {
        std::printf("shape %d %d tiles %" PRIu64 "\n", p.threads, p.grid, p.n_units);
    };
    if (before == 2) {
        report(*reinterpret_cast<Plan *>(plan));
        auto items = new_items;
        items.resize(fewer);
        for (rng_batch_item &it : items)
            it.n_per_stream = rows_then;
        fake::allocs = 0;
        if (rng_plan_refill(plan, items.data(), items.size(), nullptr))
            return 1;
        report(*reinterpret_cast<Plan *>(plan));
        std::printf("allocs %d\n", fake::allocs);
        return 0;
    }
    fake::capturing = true;
    if (rng_plan_launch(plan, nullptr))
        return 1;
    fake::capturing = false;
    const Plan taken = *reinterpret_cast<Plan *>(plan);  // what the capture holds
    report(taken);
    fake::allocs = 0;
    if (rng_plan_refill(plan, new_items.data(), n_items, nullptr))
        return 1;
    report(*reinterpret_cast<Plan *>(plan));
    std::printf("allocs %d\n", fake::allocs);
    for (uint64_t u = 0; u < taken.n_units; ++u) {
        const Unit &U = taken.d_units[u];
        const uint32_t mode = U.code >> 3, threads = (uint32_t)taken.threads;
        const uint32_t most = mode == kTail      ? threads
                              : mode == kShifted ? 4 * (31 * (threads / 32) + 1)
                                                 : 4 * threads;
        std::printf("%" PRIu64 " %u %u %u %d\n", (uint64_t)((uintptr_t)U.state >> 32) - 1, mode,
                    U.s0, std::min(U.count, most) + U.tail, U.out >= base + fresh);
    }
    return 0;
}
