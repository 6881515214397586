// Jump-ahead tables and rng_jump (sequence splitting, Sec. "Parallelizing
// RNGs").  The tables hold, for m = 0..63, the GF(2) matrix of 2^m xor128
// steps (128 columns of 4 words), of 2^m XORSHIFT8 steps (256 columns of 8
// words), of 2^m xorshift32 steps (32 columns) and the affine map (A, C) of
// 2^m LCG steps.  One CTA builds them on the device by repeated squaring,
// once per device and process.
#include <algorithm>
#include <mutex>

#include "jump.cuh"

namespace gbrng {
namespace {

constexpr int kLevels = 64;
constexpr int kMaxDevices = 64;

struct DeviceTables {
    void *mem = nullptr;
    JumpTables t{};
};
DeviceTables g_tables[kMaxDevices];
std::mutex g_mutex;

// Column j of level m is level m-1 applied to its own column j.
__global__ void __launch_bounds__(256)
build_tables(uint4 *t128, uint32_t *t32, uint2 *tl, uint4 *t8)
{
    __shared__ uint4 cur[128];
    __shared__ uint4 cur8[512];  // column j: cur8[2j] (words 0-3), cur8[2j+1] (4-7)
    __shared__ uint32_t cur32[32];
    const int j = threadIdx.x;
    {
        uint32_t v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int q = 0; q < 8; ++q)
            v[q] = (j >> 5) == q ? 1u << (j & 31) : 0u;
        xorshift8_step(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);
        cur8[2 * j] = make_uint4(v[0], v[1], v[2], v[3]);
        cur8[2 * j + 1] = make_uint4(v[4], v[5], v[6], v[7]);
        t8[2 * j] = cur8[2 * j];
        t8[2 * j + 1] = cur8[2 * j + 1];
        if (j < 128) {
            uint32_t s[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                s[q] = (j >> 5) == q ? 1u << (j & 31) : 0u;
            xor128_step(s[0], s[1], s[2], s[3]);
            cur[j] = make_uint4(s[0], s[1], s[2], s[3]);
            t128[j] = cur[j];
        }
        if (j < 32) {
            uint32_t y = 1u << j;
            xorshift32_step(y);
            cur32[j] = y;
            t32[j] = y;
        }
    }
    for (int m = 1; m < kLevels; ++m) {
        __syncthreads();
        // XORSHIFT8: every thread one column
        const uint4 lo = cur8[2 * j], hi = cur8[2 * j + 1];
        const uint32_t vw8[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        uint4 r8lo = make_uint4(0, 0, 0, 0), r8hi = make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            for (int b = 0; b < 32; ++b) {
                if ((vw8[q] >> b) & 1u) {
                    const uint4 c0 = cur8[2 * (32 * q + b)], c1 = cur8[2 * (32 * q + b) + 1];
                    r8lo.x ^= c0.x;
                    r8lo.y ^= c0.y;
                    r8lo.z ^= c0.z;
                    r8lo.w ^= c0.w;
                    r8hi.x ^= c1.x;
                    r8hi.y ^= c1.y;
                    r8hi.z ^= c1.z;
                    r8hi.w ^= c1.w;
                }
            }
        }
        uint4 r = make_uint4(0, 0, 0, 0);
        if (j < 128) {
            const uint4 v = cur[j];
            const uint32_t vw[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                for (int b = 0; b < 32; ++b) {
                    if ((vw[q] >> b) & 1u) {
                        const uint4 c = cur[32 * q + b];
                        r.x ^= c.x;
                        r.y ^= c.y;
                        r.z ^= c.z;
                        r.w ^= c.w;
                    }
                }
            }
        }
        uint32_t r32 = 0;
        if (j < 32) {
            const uint32_t y = cur32[j];
            for (int b = 0; b < 32; ++b)
                if ((y >> b) & 1u)
                    r32 ^= cur32[b];
        }
        __syncthreads();
        cur8[2 * j] = r8lo;
        cur8[2 * j + 1] = r8hi;
        t8[m * 512 + 2 * j] = r8lo;
        t8[m * 512 + 2 * j + 1] = r8hi;
        if (j < 128) {
            cur[j] = r;
            t128[m * 128 + j] = r;
        }
        if (j < 32) {
            cur32[j] = r32;
            t32[m * 32 + j] = r32;
        }
    }
    if (j == 0) {
        uint32_t A = 69069u, C = 1234567u;  // one step of Eq. 7
        for (int m = 0; m < kLevels; ++m) {
            tl[m] = make_uint2(A, C);
            C = A * C + C;  // the map after itself
            A = A * A;
        }
    }
}

// Entry y*n + s: a_s^(y*rows) mod p_s in Montgomery form (0 for y = 0, the
// segment that needs no jump).
__global__ void __launch_bounds__(256)
mwc_table_kernel(const uint32_t *__restrict__ a, uint64_t n, uint64_t rows, uint32_t segs,
                 uint64_t *__restrict__ out)
{
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * segs)
        return;
    const uint64_t y = i / n, s = i - y * n;
    out[i] = y == 0 ? 0 : mwc_power(a[s], y * rows);
}

// rng_jump of the kinds without a big GF(2) part: one stream per thread.
// KISS and KISS_XOR: the xorshift32 and LCG parts are the same map for every
// stream.  For more than three set bits of k each CTA composes it first: a
// stream then takes four table reads in place of 32 columns per set bit (2^20
// KISS streams by 24 set bits on GB300: 236 -> 105 us, of which the MWC power
// is 67).  Composing takes a CTA about 2 us, the columns 0.6 us a bit at
// 76,636 streams (KISS_XOR: 8.7 against 10.1 us at three bits, 9.6 against
// 10.4 at four, 13.4 against 11.4 at eight).
template <int KIND>
__global__ void __launch_bounds__(256) jump_kernel(rng_device_view v, uint64_t k, JumpTables T)
{
    constexpr bool kKiss = KIND == RNG_KISS || KIND == RNG_KISS_XOR;
    __shared__ KissJump J;
    const bool compose = kKiss && __popcll(k) > 3;
    if constexpr (kKiss)
        if (compose)
            kiss_jump_fill(J, k, T);
    const uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= v.n_streams)
        return;
    Engine<KIND> e;
    e.load(v, s);
    if constexpr (KIND == RNG_MWC32 || KIND == RNG_KISS) {
        mwc_jump(e.a, e.x, e.c, k);
    } else {
        mwc16_jump(e.a & 0xFFFFu, e.z, k);
        mwc16_jump(e.a >> 16, e.w, k);
    }
    if constexpr (KIND == RNG_KISS) {
        if (compose)
            kiss_jump_apply(J, e.y, e.z);
        else
            kiss_jump_bits(e.y, e.z, k, T);
    } else if constexpr (KIND == RNG_KISS_XOR) {
        if (compose)
            kiss_jump_apply(J, e.y, e.l);
        else
            kiss_jump_bits(e.y, e.l, k, T);
    }
    e.store(v, s);
}

// The columns of M^k (W words each, 32 W of them) for the matrix whose powers
// M^(2^m) are `table`, one warp per column: out[W j ..] is column j.  The set
// bits' matrices are copied to shared memory a few at a time, so that a chain
// of them runs at the reductions' latency.
template <int W>
__global__ void __launch_bounds__(128)
compose_kernel(const uint32_t *__restrict__ table, uint64_t k, uint32_t *__restrict__ out)
{
    constexpr int kWords = 32 * W * W, kAtOnce = W == 4 ? 16 : 4;  // 32 KB
    __shared__ __align__(16) uint32_t level[kAtOnce][kWords];
    const int lane = threadIdx.x & 31;
    const int j = blockIdx.x * 4 + (threadIdx.x >> 5);
    uint32_t v[W];
#pragma unroll
    for (int q = 0; q < W; ++q)
        v[q] = (j >> 5) == q ? 1u << (j & 31) : 0u;
    for (uint64_t r = k; r;) {
        int levels = 0;
        for (; levels < kAtOnce && r; ++levels, r &= r - 1) {
            const uint32_t *src = table + (size_t)kWords * (__ffsll((long long)r) - 1);
            for (int i = 4 * threadIdx.x; i < kWords; i += 4 * 128)
                copy16_async(&level[levels][i], src + i);
        }
        copies_done();
        for (int m = 0; m < levels; ++m)
            gf2_apply_warp<W>(level[m], v, lane);
        __syncthreads();
    }
    uint32_t mine = 0;
#pragma unroll
    for (int q = 0; q < W; ++q)
        mine = lane == q ? v[q] : mine;
    if (lane < W)
        out[W * j + lane] = mine;
}

// Every stream's W words times the matrix of columns `cols`, by tables of the
// images of each group of BITS bits (32 W / BITS groups, 2^BITS entries of W
// words, in shared memory): one read and W xors per group in place of BITS
// masked columns.  The reads collide like any random 16-byte reads (about 9
// wavefronts a warp), which is what bounds it; eight-bit groups need 64 KB at
// W = 4, four-bit groups 32 KB at W = 8.  Measured in
// launch_jump.
constexpr int kApplyThreads = 512;

template <int W, int BITS>
__global__ void __launch_bounds__(kApplyThreads)
apply_kernel(uint32_t *__restrict__ state, uint64_t n, const uint32_t *__restrict__ cols)
{
    constexpr int G = 32 * W / BITS, H = W / 4;
    extern __shared__ __align__(16) uint4 images[];  // [(G << BITS) * H], then 32 W columns
    uint4 *const col = images + (G << BITS) * H;
    for (int i = threadIdx.x; i < 32 * W * H; i += kApplyThreads)
        col[i] = __ldg(reinterpret_cast<const uint4 *>(cols) + i);
    __syncthreads();
    for (int e = threadIdx.x; e < G << BITS; e += kApplyThreads) {
        uint4 x[H] = {};
#pragma unroll
        for (int b = 0; b < BITS; ++b) {
            const uint32_t mask = 0u - ((uint32_t)(e >> b) & 1u);
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const uint4 c = col[((e >> BITS) * BITS + b) * H + h];
                x[h].x ^= c.x & mask;
                x[h].y ^= c.y & mask;
                x[h].z ^= c.z & mask;
                x[h].w ^= c.w & mask;
            }
        }
#pragma unroll
        for (int h = 0; h < H; ++h)
            images[e * H + h] = x[h];
    }
    __syncthreads();
    for (uint64_t s = (uint64_t)blockIdx.x * kApplyThreads + threadIdx.x; s < n;
         s += (uint64_t)gridDim.x * kApplyThreads) {
        uint32_t v[W];
#pragma unroll
        for (int q = 0; q < W; ++q)
            v[q] = state[q * n + s];
        uint4 x[H] = {};
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const uint32_t e = (v[g * BITS / 32] >> (g * BITS % 32)) & ((1u << BITS) - 1);
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const uint4 c = images[((g << BITS) + e) * H + h];
                x[h].x ^= c.x;
                x[h].y ^= c.y;
                x[h].z ^= c.z;
                x[h].w ^= c.w;
            }
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {
            state[(4 * h) * n + s] = x[h].x;
            state[(4 * h + 1) * n + s] = x[h].y;
            state[(4 * h + 2) * n + s] = x[h].z;
            state[(4 * h + 3) * n + s] = x[h].w;
        }
    }
}

template <int W, int BITS>
int launch_composed(Gen *g, uint64_t k, const uint32_t *table, cudaStream_t st)
{
    constexpr int smem = ((32 * W / BITS << BITS) + 32 * W) * W * 4;
    int e = cuda_status(cudaFuncSetAttribute(
        apply_kernel<W, BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    if (e)
        return e;
    compose_kernel<W><<<8 * W, 128, 0, st>>>(table, k, g->d_jump_cols);
    e = cuda_status(cudaGetLastError());
    if (e)
        return e;
    // resident CTAs stay and walk the streams: each builds the tables once
    const uint64_t blocks =
        std::min<uint64_t>((g->n + kApplyThreads - 1) / kApplyThreads, 152 * (W == 4 ? 3 : 4));
    apply_kernel<W, BITS>
        <<<(unsigned)blocks, kApplyThreads, smem, st>>>(g->d_state, g->n, g->d_jump_cols);
    return cuda_status(cudaGetLastError());
}

}  // namespace

int jump_tables(JumpTables *out)
{
    int dev = 0;
    int st = cuda_status(cudaGetDevice(&dev));
    if (st)
        return st;
    if (dev < 0 || dev >= kMaxDevices)
        return set_error(RNG_ERR_NODEV);
    std::lock_guard<std::mutex> lock(g_mutex);
    DeviceTables &d = g_tables[dev];
    if (!d.mem) {
        const size_t b128 = sizeof(uint4) * 128 * kLevels;
        const size_t b8 = sizeof(uint4) * 512 * kLevels;
        const size_t b32 = sizeof(uint32_t) * 32 * kLevels;
        const size_t bl = sizeof(uint2) * kLevels;
        void *mem = nullptr;
        if (cudaMalloc(&mem, b128 + b8 + b32 + bl) != cudaSuccess)
            return set_error(RNG_ERR_OOM);
        char *base = static_cast<char *>(mem);
        uint4 *t128 = reinterpret_cast<uint4 *>(base);
        uint4 *t8 = reinterpret_cast<uint4 *>(base + b128);
        uint32_t *t32 = reinterpret_cast<uint32_t *>(base + b128 + b8);
        uint2 *tl = reinterpret_cast<uint2 *>(base + b128 + b8 + b32);
        build_tables<<<1, 256>>>(t128, t32, tl, t8);
        st = cuda_status(cudaGetLastError());
        if (!st)
            st = cuda_status(cudaStreamSynchronize(0));
        if (st) {
            cudaFree(mem);
            return st;
        }
        d.mem = mem;
        d.t = JumpTables{t128, t32, tl, t8};
    }
    *out = d.t;
    return RNG_OK;
}

namespace {

constexpr int kMostTableWaits = 4;

// Hands the table to a call on `st`, after its build.
int use_jump_table(Gen *g, cudaStream_t st, const uint64_t **table)
{
    unsigned long long id = 0;
    int e = cuda_status(cudaStreamGetId(st, &id));
    if (e)
        return e;
    if (id != g->jmul_stream) {
        e = cuda_status(cudaStreamWaitEvent(st, g->jmul_built, 0));
        if (e)
            return e;
        g->jmul_shared = true;
    }
    *table = g->d_jmul;
    return RNG_OK;
}

}  // namespace

int ready_jump_table(Gen *g, uint64_t rows, uint64_t segs, cudaStream_t st,
                     const uint64_t **table)
{
    *table = nullptr;
    if (!g->d_jmul || g->jmul_rows != rows || segs > g->jmul_cap)
        return RNG_OK;
    return use_jump_table(g, st, table);
}

int mwc_jump_table(Gen *g, uint64_t rows, uint64_t segs, cudaStream_t st,
                   const uint64_t **table)
{
    if (!g->d_a || segs == 0 || segs > g->jmul_segs)
        return set_error(RNG_ERR_ARG);
    const bool grow = segs > g->jmul_cap;
    if (!grow && g->jmul_rows == rows)
        return use_jump_table(g, st, table);
    // The old table may still be read by earlier calls: on this stream they come
    // before a rebuild, but on another (or before the table is freed) the
    // device has to finish them.  A handle that keeps changing streams and
    // lengths goes without the table in the end.
    unsigned long long id = 0;
    int e = cuda_status(cudaStreamGetId(st, &id));
    if (e)
        return e;
    const bool wait = g->d_jmul && (g->jmul_shared || id != g->jmul_stream);
    if (wait && !grow && g->jmul_waits == kMostTableWaits) {
        *table = nullptr;
        return RNG_OK;
    }
    if (grow || wait) {
        e = cuda_status(cudaDeviceSynchronize());
        if (e)
            return e;
        g->jmul_waits += wait && !grow ? 1 : 0;
    }
    if (grow) {
        cudaFree(g->d_jmul);
        g->d_jmul = nullptr;
        g->jmul_cap = 0;
        g->jmul_rows = 0;
        if (cudaMalloc(&g->d_jmul, (size_t)segs * g->n * 8) != cudaSuccess)
            return set_error(RNG_ERR_OOM);
        g->jmul_cap = (uint32_t)segs;
    }
    if (!g->jmul_built)
        e = cuda_status(cudaEventCreateWithFlags(&g->jmul_built, cudaEventDisableTiming));
    if (e)
        return e;
    const uint64_t total = g->n * g->jmul_cap;
    const uint64_t blocks = (total + 255) / 256;
    g->jmul_rows = 0;  // until the new one is on its way
    mwc_table_kernel<<<(unsigned)blocks, 256, 0, st>>>(g->d_a, g->n, rows, g->jmul_cap,
                                                       g->d_jmul);
    g->jmul_stream = id;
    g->jmul_shared = false;
    e = cuda_status(cudaGetLastError());
    if (!e)
        e = cuda_status(cudaEventRecord(g->jmul_built, st));
    if (e)
        return e;
    g->jmul_rows = rows;
    *table = g->d_jmul;
    return RNG_OK;
}

int launch_jump(Gen *g, uint64_t k, cudaStream_t stream)
{
    if (k == 0)
        return RNG_OK;
    JumpTables T{};
    if (needs_jump_tables(g->kind)) {
        int st = jump_tables(&T);
        if (st)
            return st;
    }
    // The kinds with a big GF(2) part multiply the set bits' matrices together
    // first, also for a single bit: 2^20 streams jumped by 24 set bits (GB300,
    // us a call, before -> after) xor128 1305 -> 29, XORSHIFT8 5627 -> 165; 256
    // streams by one set bit 8.4 -> 5.1 and 25.4 -> 9.2, by 24 bits 178 -> 7.5
    // and 577 -> 20.
    if (g->kind == RNG_XOR128)
        return launch_composed<4, 8>(g, k, reinterpret_cast<const uint32_t *>(T.xor128), stream);
    if (g->kind == RNG_XORSHIFT8)
        return launch_composed<8, 4>(g, k, reinterpret_cast<const uint32_t *>(T.xs8), stream);
    rng_device_view v{g->kind, g->device, g->words, g->n, g->d_state, g->d_a};
    const uint64_t blocks = (g->n + 255) / 256;
    if (blocks > 0x7FFFFFFFull)
        return set_error(RNG_ERR_ARG);
    const unsigned b = (unsigned)blocks;
    switch (g->kind) {
    case RNG_MWC32: jump_kernel<RNG_MWC32><<<b, 256, 0, stream>>>(v, k, T); break;
    case RNG_KISS: jump_kernel<RNG_KISS><<<b, 256, 0, stream>>>(v, k, T); break;
    case RNG_MWC16X2: jump_kernel<RNG_MWC16X2><<<b, 256, 0, stream>>>(v, k, T); break;
    default: jump_kernel<RNG_KISS_XOR><<<b, 256, 0, stream>>>(v, k, T); break;
    }
    return cuda_status(cudaGetLastError());
}

}  // namespace gbrng
