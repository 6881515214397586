// A small statistical battery on the device (rng_battery): counts of four
// tests of the DIEHARD / TestU01 families over stream-interleaved outputs,
// for the randomness checks the paper runs with those suites (Sec.
// "Performance evaluation").  The host forms the statistics from the counts.
//
//   monobit    one bits in all outputs
//   frequency  top 8 bits, 256 bins
//   serial     non-overlapping pairs (u_{2k}, u_{2k+1}) of a stream, top 4
//              bits of each, 16 x 16 cells
//   birthday   512 consecutive outputs of a stream, days = top 24 bits;
//              sorted, spacings (first day, then neighbour differences),
//              sorted; repeats = spacings equal to the one before; at most
//              RNG_BATTERY_BIRTHDAY_MAX samples
//
// sample_kernel: everything the whole samples hold.  A CTA takes 16 samples at
// a time (the same 512 rows of 16 neighbouring streams, so its reads are row
// segments), counts bits and pairs on the way into shared memory, and each of
// its warps then sorts and examines one sample.  count_kernel: the same three
// histograms of the outputs that belong to no sample (rows past the last
// multiple of 512, and streams past the cap).
#include <algorithm>
#include <atomic>

#include "gbrng.cuh"

namespace gbrng {
namespace {

constexpr int kCountThreads = 256;
constexpr uint64_t kPairsPerTile = 64;
constexpr int kDays = 512;
constexpr unsigned kAllLanes = 0xFFFFFFFFu;

struct DeviceCounts {
    unsigned long long ones;
    unsigned long long bytes[256];
    unsigned long long serial[256];
    unsigned long long birthday[16];
};

// Rows [row0, row1) of streams [s_begin, n); row0 even.  Read-bound: the
// loads of four row pairs are in flight at a time.
__global__ void __launch_bounds__(kCountThreads)
count_kernel(const uint32_t *__restrict__ u, uint64_t n, uint64_t s_begin, uint64_t row0,
             uint64_t row1, uint64_t tile_pairs, DeviceCounts *out)
{
    __shared__ uint32_t bytes[256], serial[256];
    __shared__ unsigned long long ones_sum;
    const int t = threadIdx.x;
    bytes[t] = 0;
    serial[t] = 0;
    if (t == 0)
        ones_sum = 0;
    __syncthreads();
    const uint64_t s = s_begin + (uint64_t)blockIdx.x * kCountThreads + t;
    uint64_t r = row0 + (uint64_t)blockIdx.y * 2 * tile_pairs;
    uint64_t ones = 0;
    if (s < n) {
        const uint64_t r1 = min(row1, r + 2 * tile_pairs);
#pragma unroll 4
        for (; r + 1 < r1; r += 2) {
            const uint32_t a = __ldg(u + r * n + s), b = __ldg(u + (r + 1) * n + s);
            ones += __popc(a) + __popc(b);
            atomicAdd(&bytes[a >> 24], 1u);
            atomicAdd(&bytes[b >> 24], 1u);
            atomicAdd(&serial[(a >> 28) * 16 + (b >> 28)], 1u);
        }
        if (r < r1) {  // the last row of an odd count: no pair
            const uint32_t a = __ldg(u + r * n + s);
            ones += __popc(a);
            atomicAdd(&bytes[a >> 24], 1u);
        }
    }
    atomicAdd(&ones_sum, (unsigned long long)ones);
    __syncthreads();
    if (bytes[t])
        atomicAdd(&out->bytes[t], (unsigned long long)bytes[t]);
    if (serial[t])
        atomicAdd(&out->serial[t], (unsigned long long)serial[t]);
    if (t == 0)
        atomicAdd(&out->ones, ones_sum);
}

// A sample's repeated spacings are 512 less the number of distinct ones, so
// only the days are sorted, and by counting: days are spread over 2^24, so
// 1024 buckets of their top 10 bits hold at most a few each.  One warp per
// sample, 16 days per lane.
//   1. a shared atomic on the bucket's counter (four 8-bit counters per word)
//      gives each day its rank in the bucket; the words' sums are the 256
//      top-byte bins, which the frequency test needs anyway
//   2. a warp scan of the counters gives the buckets' first places, each day
//      goes to place + rank, and lane l reads back places 16 l .. 16 l + 15:
//      sorted but for the order inside buckets, which as many odd-even
//      transposition passes as the fullest bucket holds put right
//   3. the spacings set bits of a 2^15-bit map (their low 15 bits); a spacing
//      whose bit was set already is a candidate, about 6 per sample of which
//      2 are repeats, and the occurrences of each candidate are counted over
//      all 512 spacings
// What it costs is shared-memory wavefronts (about 450 per sample, against
// some 6000 cycles of two bitonic sorts with a barrier per stage, one day per
// thread); the ranks packed four bits each and the byte counts in shared memory
// keep it within 64 registers (spilled words went to L2 past the shared memory:
// 1.24 ms).  At 65536 x 4096 on GB300 the whole battery call took 12.0 ms with
// those sorts and takes 1.16 ms with this kernel.
// Inputs that are not spread (a bucket of 16 days or more, more than 32
// candidates) take repeats_by_sorting, so no input costs more than before.
constexpr int kSampleWarps = 16;
constexpr int kSampleThreads = 32 * kSampleWarps;
constexpr int kSampleCtas = 2;       // per SM: one loads while the other sorts
constexpr int kScratch = 1024;       // words per warp: counters and places, then the bit map
constexpr int kFirstPlaces = 256;    // word of the scratch where the places start
constexpr uint32_t kMostInBucket = 15;
constexpr uint32_t kMostCandidates = 32;
// A sample's column: 512 days, first rotated by the column's index (so that
// a row's 16 words fall into different banks), then as 16 places and 4 words
// of padding per lane (so that a lane's four 16-byte reads do not collide).
constexpr int kColumn = 640;

struct SampleShared {
    uint32_t scratch[kSampleWarps][kScratch];
    uint32_t column[kSampleWarps][kColumn];
    uint32_t bytes[256], serial[256];
    uint32_t birthday[16];
    unsigned long long ones;
};

// Ascending bitonic sort of kDays values by one warp.
__device__ void bitonic512(uint32_t *v, int lane)
{
    for (int k = 2; k <= kDays; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = lane; t < kDays / 2; t += 32) {
                const int i = 2 * t - (t & (j - 1)), p = i + j;
                const uint32_t a = v[i], b = v[p];
                if ((a > b) == ((i & k) == 0)) {
                    v[i] = b;
                    v[p] = a;
                }
            }
            __syncwarp();
        }
    }
}

// Repeated spacings of the sample at src (stride n), for any input: v holds
// kDays words.
__device__ __noinline__ int repeats_by_sorting(uint32_t *v, const uint32_t *src, uint64_t n,
                                               int lane)
{
    for (int i = lane; i < kDays; i += 32)
        v[i] = __ldg(src + (uint64_t)i * n) >> 8;
    __syncwarp();
    bitonic512(v, lane);
    uint32_t gap[kDays / 32];
    for (int i = 0; i < kDays / 32; ++i) {
        const int e = lane + 32 * i;
        gap[i] = e ? v[e] - v[e - 1] : v[0];
    }
    __syncwarp();
    for (int i = 0; i < kDays / 32; ++i)
        v[lane + 32 * i] = gap[i];
    __syncwarp();
    bitonic512(v, lane);
    int r = 0;
    for (int i = 0; i < kDays / 32; ++i) {
        const int e = lane + 32 * i;
        r += e > 0 && v[e] == v[e - 1];
    }
    return __reduce_add_sync(kAllLanes, r);
}

// Where byte value b's count is kept: lane l adds those of bytes 4 l + i and
// 128 + 4 l + i, and its neighbours' lie beside them.
__device__ __forceinline__ int byte_at(int b)
{
    return 32 * (4 * (b >> 7) + (b & 3)) + (b >> 2 & 31);
}

// Repeated spacings of the sample whose words are col[shift .. shift + 512)
// (col is overwritten), or -1 when the days are not spread.  scratch: its
// first 256 words zero on entry, and on exit unless -1 is returned.  Adds the
// sample's top-byte counts to `bytes` (byte_at).
__device__ __forceinline__ int repeats(uint32_t *scratch, uint32_t *col, int shift, int lane,
                                       uint32_t *bytes)
{
    constexpr int P = kDays / 32;
    const uint32_t below = (1u << lane) - 1;
    uint4 *const quad = reinterpret_cast<uint4 *>(scratch);
    uint32_t u[P];
#pragma unroll
    for (int i = 0; i < P; ++i)
        u[i] = col[shift + lane + 32 * i];
    // bucket u >> 22: counter word u >> 24, bits 8 * (bucket % 4) up; the ranks
    // are kept four bits each
    uint32_t rank[2] = {0, 0}, most = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t old[P / 2];
#pragma unroll
        for (int i = 0; i < P / 2; ++i) {
            const uint32_t v = u[h * (P / 2) + i];
            old[i] = atomicAdd(&scratch[v >> 24], 1u << ((v >> 22 << 3) & 31));
        }
#pragma unroll
        for (int i = 0; i < P / 2; ++i) {
            const uint32_t r = (old[i] >> ((u[h * (P / 2) + i] >> 22 << 3) & 31)) & 255u;
            most = max(most, r);
            rank[h] |= r << (4 * i);  // spilt over only when `most` is 15 or more
        }
    }
    most = __reduce_max_sync(kAllLanes, most);
    __syncwarp();
    if (most >= kMostInBucket) {  // the counters may have overflowed
#pragma unroll
        for (int i = 0; i < P; ++i)
            atomicAdd(&bytes[byte_at(u[i] >> 24)], 1u);
        return -1;
    }
    {
        const uint4 lo = quad[lane], hi = quad[32 + lane];
        const uint32_t c[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        constexpr uint32_t kSums = 0x01010101u;  // byte k of c * kSums: counters 0 .. k
        uint32_t both = 0;  // both halves' totals: counts stay below 2^16
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t sum = c[i] * kSums >> 24;
            atomicAdd(&bytes[32 * i + lane], sum);
            both += sum << (i < 4 ? 0 : 16);
        }
        uint32_t s = both;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kAllLanes, s, o);
            if (lane >= o)
                s += y;
        }
        const uint32_t low_half = __shfl_sync(kAllLanes, s, 31) & 0xFFFFu;
        s -= both;
        uint4 *const first_of = reinterpret_cast<uint4 *>(scratch + kFirstPlaces);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t before = h == 0 ? s & 0xFFFFu : (s >> 16) + low_half;
#pragma unroll
            for (int i = 0; i < 4; i += 2) {
                uint32_t w[4];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const uint32_t incl = c[4 * h + i + j] * kSums;
                    const uint32_t excl = incl - c[4 * h + i + j], base = before * 0x10001u;
                    w[2 * j] = __byte_perm(excl, 0, 0x4140) + base;  // 16-bit places
                    w[2 * j + 1] = __byte_perm(excl, 0, 0x4342) + base;
                    before += incl >> 24;
                }
                first_of[64 * h + 2 * lane + i / 2] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    }
    __syncwarp();
    const uint16_t *const first_of = reinterpret_cast<const uint16_t *>(scratch + kFirstPlaces);
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const uint32_t place = first_of[u[i] >> 22] + (rank[i / (P / 2)] >> (4 * (i % (P / 2))) & 15u);
        col[place + ((place & ~15u) >> 2)] = u[i] >> 8;
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kScratch / 128; ++i)  // the bit map
        quad[lane + 32 * i] = make_uint4(0, 0, 0, 0);
    uint32_t d[P];
#pragma unroll
    for (int i = 0; i < P / 4; ++i) {
        const uint4 q = reinterpret_cast<const uint4 *>(col)[5 * lane + i];
        d[4 * i] = q.x;
        d[4 * i + 1] = q.y;
        d[4 * i + 2] = q.z;
        d[4 * i + 3] = q.w;
    }
    // odd-even transposition: `most` + 1 days share the fullest bucket
    for (uint32_t pass = 0; pass <= most; pass += 2) {
#pragma unroll
        for (int i = 0; i < P; i += 2) {
            const uint32_t a = min(d[i], d[i + 1]), b = max(d[i], d[i + 1]);
            d[i] = a;
            d[i + 1] = b;
        }
        const uint32_t next = __shfl_down_sync(kAllLanes, d[0], 1);
        const uint32_t prev = __shfl_up_sync(kAllLanes, d[P - 1], 1);
#pragma unroll
        for (int i = 1; i < P - 1; i += 2) {
            const uint32_t a = min(d[i], d[i + 1]), b = max(d[i], d[i + 1]);
            d[i] = a;
            d[i + 1] = b;
        }
        if (lane < 31)
            d[P - 1] = min(d[P - 1], next);
        if (lane > 0)
            d[0] = max(d[0], prev);
    }
    const uint32_t prev = __shfl_up_sync(kAllLanes, d[P - 1], 1);
#pragma unroll
    for (int i = P - 1; i > 0; --i)
        d[i] -= d[i - 1];
    if (lane > 0)
        d[0] -= prev;  // the first spacing is the first day itself
    __syncwarp();  // the map is clear, the places are read
    uint32_t seen[P];
#pragma unroll
    for (int i = 0; i < P; ++i)
        seen[i] = atomicOr(&scratch[(d[i] >> 5) & (kScratch - 1)], 1u << (d[i] & 31));
    uint32_t found = 0;  // candidates, listed in col
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const bool hit = (seen[i] >> (d[i] & 31)) & 1u;
        const uint32_t m = __ballot_sync(kAllLanes, hit);
        if (m) {
            const uint32_t at = found + __popc(m & below);
            if (hit && at < kMostCandidates)
                col[at] = d[i];
            found += __popc(m);
        }
    }
    __syncwarp();
    quad[lane] = make_uint4(0, 0, 0, 0);  // the next sample's counters
    quad[32 + lane] = make_uint4(0, 0, 0, 0);
    if (found > kMostCandidates)
        return -1;
    // a value that occurs k times is k - 1 repeats; every value that occurs
    // twice or more is among the candidates
    const uint32_t cand = col[lane];
    uint32_t left = found == 32 ? kAllLanes : (1u << found) - 1;
    int r = 0;
    while (left) {
        const uint32_t v = __shfl_sync(kAllLanes, cand, __ffs(left) - 1);
        int k = 0;
#pragma unroll
        for (int i = 0; i < P; ++i)
            k += d[i] == v;
        r += __reduce_add_sync(kAllLanes, k) - 1;
        left &= ~__ballot_sync(kAllLanes, cand == v);
    }
    __syncwarp();
    return r;
}

// Samples 0 .. samples - 1 (sample i = block i / n of stream i % n: rows
// 512 b .. 512 b + 511), 16 consecutive ones per CTA and pass: lane c % 16
// loads column c, one of 16 consecutive rows after the other, both halves of
// the warp 16 rows apart.
__global__ void __launch_bounds__(kSampleThreads, kSampleCtas)
sample_kernel(const uint32_t *__restrict__ u, uint64_t n, uint32_t samples, DeviceCounts *out)
{
    extern __shared__ __align__(16) unsigned char shared_bytes[];
    SampleShared &S = *reinterpret_cast<SampleShared *>(shared_bytes);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    constexpr int R = 16;  // rows per thread
    for (int i = t; i < kSampleWarps * kScratch; i += kSampleThreads)
        (&S.scratch[0][0])[i] = 0;
    if (t < 256) {
        S.bytes[t] = 0;
        S.serial[t] = 0;
    }
    if (t < 16)
        S.birthday[t] = 0;
    if (t == 0)
        S.ones = 0;
    uint32_t ones = 0;  // at most 512 per pass, below 2^21 / 16 passes
    const int c = lane & (kSampleWarps - 1);
    const int row = 32 * warp + R * (lane >> 4);
    auto sample_at = [&](uint32_t q) {  // its first word
        const uint64_t b = n > q ? 0 : q / (uint32_t)n, s = n > q ? q : q % (uint32_t)n;
        return u + b * kDays * n + s;
    };
    for (uint64_t q0 = (uint64_t)blockIdx.x * kSampleWarps; q0 < samples;
         q0 += (uint64_t)gridDim.x * kSampleWarps) {
        __syncthreads();  // the columns of the pass before are done with
        if (q0 + c < samples) {
            const uint32_t *src = sample_at((uint32_t)q0 + c) + (uint64_t)row * n;
            uint32_t x[R];
#pragma unroll
            for (int j = 0; j < R; ++j) {
                x[j] = __ldg(src);
                src += n;
            }
            uint32_t *const dst = &S.column[c][c + row];
#pragma unroll
            for (int j = 0; j < R; j += 2) {
                dst[j] = x[j];
                dst[j + 1] = x[j + 1];
                ones += __popc(x[j]) + __popc(x[j + 1]);
                atomicAdd(&S.serial[(x[j] >> 28) * 16 + (x[j + 1] >> 28)], 1u);
            }
        }
        __syncthreads();
        if (q0 + warp < samples) {
            int r = repeats(S.scratch[warp], S.column[warp], warp, lane, S.bytes);
            if (r < 0) {
                __syncwarp();
                r = repeats_by_sorting(S.scratch[warp], sample_at((uint32_t)q0 + warp), n, lane);
                __syncwarp();
                for (int i = lane; i < kFirstPlaces; i += 32)
                    S.scratch[warp][i] = 0;
                __syncwarp();
            }
            if (lane == 0)
                atomicAdd(&S.birthday[r < 15 ? r : 15], 1u);
        }
    }
    atomicAdd(&S.ones, (unsigned long long)ones);
    __syncthreads();
    if (t < 256) {
        atomicAdd(&out->bytes[t], (unsigned long long)S.bytes[byte_at(t)]);
        atomicAdd(&out->serial[t], (unsigned long long)S.serial[t]);
    }
    if (t < 16 && S.birthday[t])
        atomicAdd(&out->birthday[t], (unsigned long long)S.birthday[t]);
    if (t == 0)
        atomicAdd(&out->ones, S.ones);
}

// Device counts of the calls in progress: a few fixed ones per device, so that
// a call need not allocate and free (about 30 us, and the free waits for the
// device); further calls at once, from other host threads, allocate.
constexpr int kSlots = 8, kMaxDevices = 64;
__device__ DeviceCounts g_slots[kSlots];
std::atomic<bool> g_taken[kMaxDevices][kSlots];

// One call's counts, given back when the call returns (it has synchronised).
struct Scratch {
    DeviceCounts *counts = nullptr;
    std::atomic<bool> *taken = nullptr;  // nullptr: allocated

    DeviceCounts *take()
    {
        int dev = -1;
        void *base = nullptr;
        if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices &&
            cudaGetSymbolAddress(&base, g_slots) == cudaSuccess)
            for (int i = 0; i < kSlots; ++i)
                if (!g_taken[dev][i].exchange(true)) {
                    taken = &g_taken[dev][i];
                    return counts = static_cast<DeviceCounts *>(base) + i;
                }
        if (cudaMalloc(&counts, sizeof(DeviceCounts)) != cudaSuccess)
            counts = nullptr;
        return counts;
    }
    ~Scratch()
    {
        if (taken)
            taken->store(false);
        else
            cudaFree(counts);
    }
};

// Counts rows [row0, row1) of streams [s_begin, n).
int launch_count(const uint32_t *u, uint64_t n, uint64_t s_begin, uint64_t row0, uint64_t row1,
                 DeviceCounts *d, cudaStream_t st)
{
    if (row0 >= row1 || s_begin >= n)
        return RNG_OK;
    const uint64_t gx = (n - s_begin + kCountThreads - 1) / kCountThreads;
    if (gx > 0x7FFFFFFFull)
        return set_error(RNG_ERR_ARG);
    // row pairs per tile: at least kPairsPerTile, more when the grid's y
    // dimension (at most 65535) would not cover the rows
    const uint64_t pairs = (row1 - row0 + 1) / 2;
    const uint64_t tile = std::max<uint64_t>(kPairsPerTile, (pairs + 65534) / 65535);
    const uint64_t gy = (pairs + tile - 1) / tile;
    count_kernel<<<dim3((unsigned)gx, (unsigned)gy), kCountThreads, 0, st>>>(u, n, s_begin, row0,
                                                                             row1, tile, d);
    return cuda_status(cudaGetLastError());
}

int launch_samples(const uint32_t *u, uint64_t n, uint32_t samples, DeviceCounts *d,
                   cudaStream_t st)
{
    if (samples == 0)
        return RNG_OK;
    constexpr int kSMs = 152;
    const unsigned groups = (samples + kSampleWarps - 1) / kSampleWarps;
    int e = cuda_status(cudaFuncSetAttribute(sample_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(SampleShared)));
    if (e)
        return e;
    sample_kernel<<<std::min<unsigned>(groups, kSampleCtas * kSMs), kSampleThreads,
                    sizeof(SampleShared), st>>>(u, n, samples, d);
    return cuda_status(cudaGetLastError());
}

}  // namespace
}  // namespace gbrng

using namespace gbrng;

extern "C" int rng_battery(const void *dev_u, uint64_t n_streams, uint64_t n_per_stream,
                           rng_battery_counts *host_counts, void *cuda_stream)
{
    if (!dev_u || !host_counts || n_streams == 0 || (uintptr_t)dev_u % 4 != 0 ||
        n_per_stream > UINT64_MAX / 4 / n_streams)
        return set_error(RNG_ERR_ARG);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const uint32_t *u = static_cast<const uint32_t *>(dev_u);
    Scratch scratch;
    DeviceCounts *const d = scratch.take();
    if (!d)
        return set_error(RNG_ERR_OOM);
    int status = cuda_status(cudaMemsetAsync(d, 0, sizeof(DeviceCounts), st));
    const uint64_t blocks = n_per_stream / kDays;
    // sample i: block i / n_streams of stream i % n_streams, i < the cap
    const uint64_t samples = std::min<uint64_t>(blocks * n_streams, RNG_BATTERY_BIRTHDAY_MAX);
    // the outputs in no sample: the rest of the block the cap falls into, and
    // every row after the last block with samples
    const uint64_t done = samples / n_streams, cut = samples % n_streams;
    const uint64_t rest = kDays * (done + (cut ? 1 : 0));
    if (!status && n_per_stream && (n_streams + kCountThreads - 1) / kCountThreads > 0x7FFFFFFFull)
        status = set_error(RNG_ERR_ARG);
    if (!status)
        status = launch_samples(u, n_streams, (uint32_t)samples, d, st);
    if (!status && cut)
        status = launch_count(u, n_streams, cut, kDays * done, rest, d, st);
    if (!status)
        status = launch_count(u, n_streams, 0, rest, n_per_stream, d, st);
    DeviceCounts h{};
    if (!status)
        status = cuda_status(cudaMemcpyAsync(&h, d, sizeof(h), cudaMemcpyDeviceToHost, st));
    if (!status)
        status = cuda_status(cudaStreamSynchronize(st));
    if (status) {
        cudaStreamSynchronize(st);  // nothing writes the counts when they are given back
        return status;
    }
    host_counts->n_outputs = n_streams * n_per_stream;
    host_counts->ones = h.ones;
    for (int k = 0; k < 256; ++k) {
        host_counts->bytes[k] = h.bytes[k];
        host_counts->serial[k] = h.serial[k];
    }
    host_counts->birthday_samples = samples;
    for (int k = 0; k < 16; ++k)
        host_counts->birthday[k] = h.birthday[k];
    return RNG_OK;
}
