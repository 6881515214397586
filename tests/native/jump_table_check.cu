// Host-only driver of the handle's MWC jump table: includes the library's jump.cu
// with the CUDA runtime calls it makes replaced by stand-ins, and takes the table
// for calls on streams with given handles and ids.
// Input: per call "handle id rows segs ready" (ready = 1: ready_jump_table, else
// mwc_jump_table).  Output: per call "table events syncs": whether it got a table, and
// the waits for the build's event and for the device that it made.
#include <cinttypes>
#include <cstdio>
#include <cstdlib>

#include <cuda_runtime.h>

namespace fake {
unsigned long long id = 0;
int events = 0, syncs = 0;
cudaError_t ok() { return cudaSuccess; }
template <class T>
cudaError_t alloc(T **p, size_t bytes)
{
    *p = static_cast<T *>(std::malloc(bytes));
    return cudaSuccess;
}
cudaError_t release(void *p)
{
    std::free(p);
    return cudaSuccess;
}
cudaError_t event(cudaEvent_t *e)
{
    static int any;
    *e = reinterpret_cast<cudaEvent_t>(&any);
    return cudaSuccess;
}
cudaError_t stream_id(unsigned long long *v)
{
    *v = id;
    return cudaSuccess;
}
cudaError_t wait()
{
    ++events;
    return cudaSuccess;
}
cudaError_t sync()
{
    ++syncs;
    return cudaSuccess;
}
}  // namespace fake

#define cudaMalloc fake::alloc
#define cudaFree fake::release
#define cudaEventCreateWithFlags(e, flags) fake::event(e)
#define cudaEventRecord(e, stream) fake::ok()
#define cudaGetLastError() fake::ok()
#define cudaStreamGetId(stream, v) fake::stream_id(v)
#define cudaStreamWaitEvent(stream, e, flags) fake::wait()
#define cudaDeviceSynchronize() fake::sync()

#include "jump.cu"

namespace gbrng {
int set_error(int status) { return status; }
int cuda_status(cudaError_t e) { return e == cudaSuccess ? 0 : RNG_ERR_CUDA; }
}  // namespace gbrng

int main()
{
    using namespace gbrng;
    // the launches name host memory: they must not find a GPU
    setenv("CUDA_VISIBLE_DEVICES", "", 1);
    Gen g;
    uint32_t a = 0;
    g.n = 64;
    g.kind = RNG_MWC32;
    g.d_a = &a;
    g.jmul_segs = 1024;
    uintptr_t handle;
    uint64_t rows, segs;
    int ready;
    while (std::scanf("%" SCNuPTR " %llu %" SCNu64 " %" SCNu64 " %d", &handle, &fake::id, &rows,
                      &segs, &ready) == 5) {
        const uint64_t *table = nullptr;
        fake::events = fake::syncs = 0;
        const cudaStream_t st = reinterpret_cast<cudaStream_t>(handle);
        if (ready ? ready_jump_table(&g, rows, segs, st, &table)
                  : mwc_jump_table(&g, rows, segs, st, &table))
            return 1;
        std::printf("%d %d %d\n", table ? 1 : 0, fake::events, fake::syncs);
    }
    return 0;
}
