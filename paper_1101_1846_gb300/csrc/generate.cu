// Launch policy of the generation kernels (shapes, splitting) and the
// dispatch of a call to its kind's launcher (gen_kernels.cuh): the three
// target kinds are instantiated here, the paper's own generators in
// generate_paper.cu.
#include <mutex>
#include <vector>

#include "gen_kernels.cuh"
#include "rng_tune.h"

namespace gbrng {
namespace {

// Launch shape per (kind, fmt): groups of four streams per thread V, CTA
// size, store hint, and one = one CTA per SM (a shared-memory reservation
// keeps a second CTA off the SM).  Defaults are the best measured on GB300;
// gbrng_set_launch / gbrng_set_launch_class change the first three (the
// autotuner does), gbrng_set_launch_ctas the last.
struct Shape {
    int v;
    int block;
    int hint;
    int one;
};
// MWC uint32 writes its rows through TMA bulk copies (hint 2): 6 % faster
// per launch on GB300 than 16-byte stores from two CTAs per SM, level with
// them from one.  xor128 uint32 was 1.4 % faster through TMA until 16-byte
// stores from one CTA per SM overtook it (below); the FP32 forms measured
// the same, and KISS and XORSHIFT8, whose steps cost more, ran 4-40 %
// slower that way.  Per-warp bulk copies of 512 B (each warp
// staging its own rows, no block barrier) were slower than both.
//
// Two size classes: calls of fewer than kSmallStreams streams (class 0) and
// the rest (class 1).  At 2^20 streams x 1024 the kernels fill the GPU
// differently (medians of three sweeps of every shape on one GB300): xor128
// FP32 ran 1345 GS/s with its 2^22 shape (1, 128) and 1615 with (2, 128);
// KISS FP32 1580 with (2, 512), 1619 with (1, 256) and 1706 with (1, 128);
// xor128 uint32 1691 through TMA and 1728 with (1, 128) and plain stores.
//
// One CTA of 512 threads per SM, against the best shapes without it (two
// rounds on one GB300, GS/s): at 2^22 x 1024, MWC f32 1807 -> 1821, xor128
// u32 1790-1800 (TMA) -> 1804, xor128 f32 1771 -> 1805, KISS u32 1757 ->
// 1797, KISS f32 1716 -> 1813 (with plain stores; 1765 streaming); MWC u32
// stays with TMA (1823 against 1818).  At 2^20 x 1024 only xor128 f32 gains
// (1609-1614 -> 1717 with V = 2).  As for the barrier-synced kernels, fewer
// warps writing at once keep each SM's write stream denser.
constexpr Shape kShape[2][kKinds][2] = {
    {
        {{1, 256, 2, 0}, {2, 512, 1, 0}},  // MWC u32, f32
        {{1, 128, 0, 0}, {2, 512, 1, 1}},  // xor128
        {{2, 512, 1, 0}, {1, 128, 1, 0}},  // KISS
        {{2, 256, 1, 0}, {2, 256, 1, 0}},  // MWC16X2
        {{1, 256, 1, 0}, {1, 256, 1, 0}},  // XORSHIFT8 (eight state words per stream)
        {{2, 256, 1, 0}, {2, 256, 1, 0}},  // KISS_XOR
    },
    {
        {{1, 256, 2, 0}, {1, 512, 1, 1}},  // MWC u32, f32
        {{1, 512, 1, 1}, {1, 512, 1, 1}},  // xor128
        {{1, 512, 1, 1}, {1, 512, 0, 1}},  // KISS
        {{2, 256, 1, 0}, {2, 256, 1, 0}},  // MWC16X2
        {{1, 256, 1, 0}, {1, 256, 1, 0}},  // XORSHIFT8 (eight state words per stream)
        {{2, 256, 1, 0}, {2, 256, 1, 0}},  // KISS_XOR
    },
};
// The shapes in use: the ones above, and what callers set instead.
struct SetShape {
    Shape shape;
    bool set;
};
SetShape g_set_shape[2][kKinds][2];

Shape &shape_to_set(int size_class, int kind, int fmt)
{
    SetShape &s = g_set_shape[size_class][kind][fmt];
    if (!s.set)
        s = SetShape{kShape[size_class][kind][fmt], true};
    return s.shape;
}

const Shape &shape_in_use(int size_class, int kind, int fmt)
{
    const SetShape &s = g_set_shape[size_class][kind][fmt];
    return s.set ? s.shape : kShape[size_class][kind][fmt];
}
constexpr uint64_t kSmallStreams = (uint64_t)1 << 21;

// CTAs per SM of the barrier-synced kernels, [kind][fmt][realigned]: 1 =
// one CTA of 512 threads per SM, 0 = as many as fit (two at their register
// counts).  Measured on GB300 at (2^22 - 4) x 1024 (16-byte rows) and
// (2^22 - 2) x 1024 (realigned), GS/s with two CTAs -> with one:
//   MWC u32 1760 -> 1766 / 1686 -> 1756;  MWC f32 1717 -> 1783 / 1694 -> 1772
//   xor128 u32 1663 -> 1746 / 1689 -> 1753;  xor128 f32 1670 -> 1695 / 1710 -> 1685
//   KISS u32 1713 -> 1797 / 1683 -> 1744;  KISS f32 1720 -> 1617 / 1690 -> 1441
// Where the step is cheap, fewer warps writing at once keep the write
// stream denser; the FP32 forms of xor128 and KISS need the second CTA's
// warps to cover their arithmetic.  The paper's kinds keep 0 (not measured).
constexpr int kRowCtas[kKinds][2][2] = {
    {{1, 1}, {1, 1}},  // MWC u32 (16-byte rows, realigned), f32
    {{1, 1}, {1, 0}},  // xor128
    {{1, 1}, {0, 0}},  // KISS
    {{0, 0}, {0, 0}},  // MWC16X2
    {{0, 0}, {0, 0}},  // XORSHIFT8
    {{0, 0}, {0, 0}},  // KISS_XOR
};
int g_row_ctas[kKinds][2][2];  // a caller's: 1 + the value, 0 = the table's

// Fewest rows of a split segment, as log2, per kind (0: never split), and
// the rows it has when that gives threads enough.  The jump that starts a
// segment costs about as much as the fewest rows: MWC32 a Montgomery product
// or a power, the base-2^16 parts a 32-bit power each, the KISS kinds that and
// the CTA's composed maps, xor128 and XORSHIFT8 a composed matrix (SegmentJump).
// A call that has all the threads it wants takes segments of equal length,
// any multiple of eight rows (76,636 x 2400 MWC: 113 us with 16 of 152 rows, 121
// with ten of 256), but for xor128 and XORSHIFT8, whose jumps compose a matrix
// per set bit of the segment's first row (xor128 there: 124 us with 256 rows,
// 145 with 200), KISS f32, of which half as many CTAs are resident (us, equal
// lengths and powers of two: 116,332 x 1335 121, 113; 64,448 x 3137 134, 128;
// 193,744 x 1030 131, 123), and the consumers.  Its MWC powers are taken in the
// kernel: against rows that long they cost nothing (76,632 x 4096: MWC 184 us
// with the handle's table, 181 without; KISS u32 198 and 192), and calls of many
// lengths rebuild no table.  Shorter segments keep powers of two and the table (MWC
// 4096 x 4096: 15.0 us with it, 18.9 without).
// From a sweep on GB300 of 32 ... 300,001 streams by 150 ... 16384 rows, every
// kind, aligned and not, segments of 2^5 ... 2^11 rows and whole calls.
int g_split_log2[kKinds] = {5, 7, 5, 5, 8, 5};
constexpr int kSplitRowsLog2[kKinds] = {6, 8, 7, 7, 9, 8};
// Consumer calls, one stream per thread, pay the same jumps for a quarter of
// the work a row (XORSHIFT8 sums, whole -> split, us: 1000 x 8192 212 -> 60,
// 10,000 x 8192 213 -> 132; 1000 x 65,536 1671 -> 125).
constexpr int kReduceRowsLog2[kKinds] = {6, 8, 7, 8, 10, 8};
// Fewer threads than this in all, and fewer CTAs than SMs: shorter segments,
// down to the fewest rows.
// (4099 x 1024 KISS: 16.5 us with 64 rows, 20.6 with 128; 1001 x 16384, which
// reaches 32,000 threads with 128: 29.1 with 128, 32.0 with 64; 4096 x 4800
// KISS_XOR: 22.7 with 128, 33.3 with 256, which has 19,000 threads.)
constexpr uint64_t kSplitThreads[kKinds] = {16000, 16000, 16000, 16000, 16000, 40000};
// No table for calls this short: their exponents are as short.
constexpr uint64_t kNoTableSteps = 128;
// Calls of fewer threads than half of this are "few-stream" calls, which
// split.
constexpr uint64_t kFewStreamThreads = (uint64_t)kSMs * 1024;
// Threads a split generate call may have: 2048 per SM, the most that can be
// resident.  Against 1024 per SM this was measured on GB300 at
// 76,632 x 16,384: MWC32 1584 -> 1740 GS/s, KISS 1575 -> 1680, xor128
// 1575 -> 1670; at 76,636 x 16,384, MWC16X2 1449 -> 1500 and KISS_XOR
// 1541 -> 1680.  Consumer (reduce) calls, one stream per thread, keep 1024.
constexpr uint64_t kSplitFillThreads = (uint64_t)kSMs * 2048;

// KISS_XOR, whose steps cost most of those with cheap jumps, runs best as one
// wave of CTAs while its segments stay this short (u32, us in one wave and in
// more, by rows of the one wave's segments: 512 76,636 x 4096 193, 205; 683
// 20,004 x 12,288 162, 183; 768 76,636 x 6144 279, 290; 1024 76,636 x 8192 367,
// 375; 1536 76,636 x 12,288 592, 544.  Realigned rows: 30,001 x 8192, 683 rows,
// 187, 200, but 76,633 x 4096, 1024 rows, 264, 252).
constexpr uint64_t kOneWaveRows = 1024;
constexpr uint64_t kOneWaveRowsShifted = 512;

inline uint64_t round8(uint64_t rows) { return (rows + 7) / 8 * 8; }

inline uint64_t split_threads(SplitForm form, uint64_t streams)
{
    return form == SplitForm::kReduce ? streams : (streams + 3) / 4;
}

// Fewest rows of a call that is worth splitting.  More threads fill more of the
// device as they are, and the jumps of more segments cost more in all; rows of 16
// bytes, whose whole form pays for row barriers, and FP32, whose whole forms wait
// longest for their conversions, split sooner.  The lines come from 3400 calls
// timed whole and split; split over whole, GB300:
//   rows            200  300  400  500  650  800 1000 1300 1600 2000 2600
//   MWC u32
//     20,000        .86  .70  .64
//     50,000       1.01 1.00  .95 1.00  .87  .98 1.00  .87
//     76,632       1.17 1.13 1.02 1.03 1.04 1.00  .95 1.02  .96
//     202,048      1.10 1.08 1.08 1.01 1.00  .99
//   KISS u32
//     50,000       1.14  .90  .83  .96  .79  .81
//     76,632       1.14 1.11 1.09 1.03 1.06 1.07 1.02  .99  .97
//     202,048       .90  .91  .88  .85
//   MWC16X2 u32
//     20,000       1.25  .99 1.12  .95  .78
//     50,000       1.22 1.16 1.03 1.26 1.10 1.05 1.02  .96 1.00 1.00  .88
//     76,632       1.17 1.28 1.07 1.15 1.07 1.14 1.06 1.08 1.03  .98  .95
//     76,636 f32    .89 1.01  .94  .92  .89  .85
//   KISS_XOR u32
//     20,000        .97  .91  .75
//     50,000       1.28 1.20 1.05 1.14  .90  .84  .99  .80
//     76,632       1.29 1.39 1.20 1.14 1.21 1.13  .98 1.09 1.16  .97  .94
//     76,636       1.04 1.08  .94  .84  .92
//   xor128: 1000 x 700 1.0, x 927 .78, f32 x 513 .98, x 927 .57; 1004 x 600 1.0, f32
//     x 400 .80; 20,000 x 1024 1.10, f32 x 600 .88; 40,000 x 2000 1.16, f32 1.07;
//     60,004 f32 x 600 1.16, x 800 .97; 173,440 x 1813 f32 .75
//   XORSHIFT8: 4096 x 1024 1.14, x 1300 .87, f32 x 1024 .94; 40,000 x 6000 .90;
//     50,000 x 8000 1.06, x 16,000 .85, f32 x 8000 .90; 76,632 x 16,000 1.20, x
//     20,000 1.03
uint64_t aligned_min_steps(int kind, int fmt, bool sectors, uint64_t threads)
{
    // shorter calls take 4-8 us whole, one group per thread (kSmallCall), and as
    // long split
    constexpr uint64_t least = 129;
    const bool f32 = fmt == RNG_F32;
    const bool many = threads > (uint64_t)kSMs * 128;  // more than a warp a scheduler
    switch (kind) {
    case RNG_XOR128:
        if (many)
            return 1024;
        if (threads <= 64)
            return f32 ? 300 : 400;
        if (threads <= (f32 ? 5000 : 3700))
            return f32 ? (sectors ? 520 : 400) : sectors ? 760 : 600;
        if (f32 && !sectors)
            return threads <= 10000 ? 520 : 760;
        return std::max<uint64_t>(
            1024, std::min<uint64_t>(2048, f32 ? threads * 9 / 40 : threads * 3 / 10));
    case RNG_XORSHIFT8:
        if (!f32 && threads > 10000 && threads <= 26000)
            return threads <= 17000 ? 16000 : 24000;
        return std::max<uint64_t>(f32 || threads <= 64 ? 1024 : 1150, threads * 3 / 5);
    case RNG_MWC32:
        return many ? 250 : std::max(least, threads / (sectors ? 40 : f32 ? 80 : 64));
    case RNG_KISS: return many ? 160 : std::max(least, threads / (f32 && !sectors ? 80 : 42));
    case RNG_MWC16X2:
        if (f32 && !sectors)
            return threads <= 6000 ? least : std::max<uint64_t>(180, threads / 85);
        return std::max<uint64_t>(180, threads / (sectors ? 17 : 26));
    default:
        if (!sectors)
            return std::max(least, threads / 60);
        return std::max<uint64_t>(threads < 1000 ? least : 180,
                                  threads / (threads <= 14000 ? 28 : 13));
    }
}

// The same for rows that are not 16-byte aligned: fewer than four streams, which
// run one to a thread with no row to realign (three streams, whole and split, us:
// xor128 u32 x 4000 38, 40, f32 x 3000 38, 35; XORSHIFT8 x 6000 132, 143; KISS u32 x
// 500 12, 14, f32 x 400 14, 13; MWC x 400 4.6, 4.8; MWC16X2 x 400 5.5, 5.8; KISS_XOR
// u32 x 500 12.1, 12.7, f32 x 400 13.4, 12.3), one group of four (XORSHIFT8 x 1254
// 86, 91; KISS u32 x 256 12.5, 13.3; KISS_XOR u32 x 160 11.3, 12.0), or more (KISS
// 150,001 x 300: 29, 44; 1001 x 300: 17.6, 13.4; KISS_XOR, the slowest steps, 1001 x
// 129: 14.8, 9.4; XORSHIFT8 54,014 x 5838: 362, 431).
uint64_t shifted_min_steps(int kind, int fmt, uint64_t streams, uint64_t threads)
{
    constexpr uint64_t kTail[2][kKinds] = {{450, 4400, 600, 450, 7000, 560},
                                           {450, 2800, 380, 450, 7000, 360}};
    constexpr uint64_t kGroup[2][kKinds] = {{256, 1024, 288, 256, 1300, 200},
                                            {256, 1024, 256, 256, 1300, 150}};
    if (streams <= 4)
        return (streams < 4 ? kTail : kGroup)[fmt == RNG_F32 ? 1 : 0][kind];
    switch (kind) {
    case RNG_XOR128:
        return std::max<uint64_t>(1024, std::min<uint64_t>(2048, threads * 3 / 10));
    case RNG_XORSHIFT8: return std::max<uint64_t>(1024, threads * 3 / 5);
    case RNG_KISS_XOR: return std::max<uint64_t>(129, threads / 50);
    default: return std::max<uint64_t>(256, std::min<uint64_t>(1024, threads / 10));
    }
}

uint64_t split_min_steps(int kind, SplitForm form, int fmt, uint64_t streams)
{
    const uint64_t threads = split_threads(form, streams);
    if (form == SplitForm::kShifted)
        return shifted_min_steps(kind, fmt, streams, threads);
    if (form != SplitForm::kReduce)
        return aligned_min_steps(kind, fmt, form == SplitForm::kAligned, threads);
    switch (kind) {
    case RNG_XOR128:
        return std::max<uint64_t>(1024, std::min<uint64_t>(2048, threads * 3 / 10));
    case RNG_XORSHIFT8: return std::max<uint64_t>(1024, threads * 3 / 5);
    case RNG_MWC16X2: return std::max<uint64_t>(129, threads / 50);
    default: return 129;
    }
}

}  // namespace

LaunchShape launch_shape(int kind, int fmt, uint64_t streams)
{
    const int size_class = streams < kSmallStreams ? 0 : 1;
    const Shape s = shape_in_use(size_class, kind, fmt), d = kShape[size_class][kind][fmt];
    return LaunchShape{s.v, s.block, s.hint, s.one,
                       s.v != d.v || s.block != d.block || s.hint != d.hint || s.one != d.one};
}

int row_ctas(int kind, int fmt, bool realigned)
{
    const int set = g_row_ctas[kind][fmt][realigned ? 1 : 0];
    return set ? set - 1 : kRowCtas[kind][fmt][realigned ? 1 : 0];
}

bool row_ctas_set(int kind, int fmt, bool realigned)
{
    return row_ctas(kind, fmt, realigned) != kRowCtas[kind][fmt][realigned ? 1 : 0];
}

namespace {

// The smallest multiple of 1 KB of dynamic shared memory above half an SM's
// share (less the per-CTA reservation), if the kernel then fits one CTA.
int find_one_cta_smem(const void *kernel, int threads, int dev)
{
    int per_sm = 0, reserved = 0, optin = 0, fit = 0;
    if (cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
            cudaSuccess)
        return 0;
    // two CTAs would need 2 * (smem + reserved) > per_sm
    const int smem = ((per_sm / 2 - reserved + 1 + 1023) / 1024) * 1024;
    if (smem <= 0 || smem > optin ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kernel, threads, smem) !=
            cudaSuccess ||
        fit != 1) {
        cudaGetLastError();  // leave no sticky error from the probe behind
        return 0;
    }
    return smem;
}

}  // namespace

int one_cta_smem(const void *kernel, int threads)
{
    // answers per (kernel, threads, device), found once each
    struct Known {
        const void *kernel;
        int threads, dev, smem;
    };
    static std::mutex mu;
    static std::vector<Known> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess)
        return 0;
    std::lock_guard<std::mutex> lock(mu);
    for (const Known &k : known)
        if (k.kernel == kernel && k.threads == threads && k.dev == dev)
            return k.smem;
    const int smem = find_one_cta_smem(kernel, threads, dev);
    known.push_back(Known{kernel, threads, dev, smem});
    return smem;
}

int resident_ctas(const void *kernel, int threads, int smem)
{
    struct Known {
        const void *kernel;
        int threads, smem, dev, ctas;
    };
    static std::mutex mu;
    static std::vector<Known> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess)
        return 0;
    std::lock_guard<std::mutex> lock(mu);
    for (const Known &k : known)
        if (k.kernel == kernel && k.threads == threads && k.smem == smem && k.dev == dev)
            return k.ctas;
    int sms = 0, fit = 0;
    if ((smem && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      smem) != cudaSuccess) ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kernel, threads, smem) !=
            cudaSuccess) {
        cudaGetLastError();  // leave no sticky error from the probe behind
        fit = 0;
    }
    known.push_back(Known{kernel, threads, smem, dev, sms * fit});
    return sms * fit;
}

uint32_t split_max_segments(uint64_t n)
{
    const uint64_t threads = (n + 3) / 4;
    return (uint32_t)std::min<uint64_t>(kSplitFillThreads / std::max<uint64_t>(threads, 1), 65535);
}

bool split_wanted(int kind, SplitForm form, int fmt, uint64_t streams, uint64_t steps)
{
    if (g_split_log2[kind] == 0 || streams == 0 || streams > kSplitMaxStreams ||
        steps > (1ull << 31))
        return false;
    const uint64_t threads = split_threads(form, streams);
    return 2 * threads <= kFewStreamThreads &&  // else they fill the device already
           steps >= split_min_steps(kind, form, fmt, streams);
}

bool split_segments(int kind, SplitForm form, int fmt, uint64_t streams, uint64_t steps,
                    uint64_t tiles, uint64_t resident, uint64_t max_segments, Segments *out)
{
    const bool reduce = form == SplitForm::kReduce;
    const uint64_t threads = split_threads(form, streams);
    const int fewest = g_split_log2[kind];
    uint64_t want = std::min<uint64_t>(
        std::min<uint64_t>((reduce ? kFewStreamThreads : kSplitFillThreads) / threads, 65535),
        max_segments);
    if (kind == RNG_KISS_XOR && !reduce && resident >= 2 * tiles &&
        steps <= (form == SplitForm::kShifted ? kOneWaveRowsShifted : kOneWaveRows) *
                     (resident / tiles))
        want = std::min(want, resident / tiles);
    if (want < 2)
        return false;
    auto count = [&](uint64_t L) { return (steps + L - 1) / L; };
    uint64_t L = 1ull << std::max(fewest, (reduce ? kReduceRowsLog2 : kSplitRowsLog2)[kind]);
    while (!reduce && L > 1ull << fewest && threads * count(L) < kSplitThreads[kind] &&
           tiles * count(L) < kSMs)
        L >>= 1;
    // as many segments as threads allow, each longer than L: of one length
    const bool full = count(L) > want;
    const bool pow2 = kind == RNG_XOR128 || kind == RNG_XORSHIFT8 ||
                      (kind == RNG_KISS && fmt == RNG_F32);
    if (full && !reduce && !pow2) {
        L = round8(count(want));
        L = round8(count(count(L)));
    }
    while (L < steps && count(L) > want)
        L <<= 1;
    if (count(L) < 2)
        return false;
    *out = Segments{L, count(L), reduce || (!full && steps > kNoTableSteps)};
    return true;
}

int launch_generate(int kind, int fmt, const GenLaunch &p, cudaStream_t st)
{
    switch (kind) {
    case RNG_MWC32: return launch_kind<RNG_MWC32>(fmt, p, st);
    case RNG_XOR128: return launch_kind<RNG_XOR128>(fmt, p, st);
    case RNG_KISS: return launch_kind<RNG_KISS>(fmt, p, st);
    default: return launch_generate_paper(kind, fmt, p, st);
    }
}

}  // namespace gbrng

extern "C" int gbrng_set_row_ctas(int kind, int fmt, int realigned, int ctas_per_sm)
{
    using namespace gbrng;
    if (kind < 0 || kind >= kKinds || fmt < 0 || fmt > 1 || realigned < 0 || realigned > 1 ||
        ctas_per_sm < 0 || ctas_per_sm > 1)
        return set_error(RNG_ERR_ARG);
    g_row_ctas[kind][fmt][realigned] = 1 + ctas_per_sm;
    return RNG_OK;
}

extern "C" int gbrng_get_row_ctas(int kind, int fmt, int realigned, int *ctas_per_sm)
{
    using namespace gbrng;
    if (kind < 0 || kind >= kKinds || fmt < 0 || fmt > 1 || realigned < 0 || realigned > 1 ||
        !ctas_per_sm)
        return set_error(RNG_ERR_ARG);
    *ctas_per_sm = row_ctas(kind, fmt, realigned != 0);
    return RNG_OK;
}

extern "C" int gbrng_set_launch_class(int kind, int fmt, int size_class, int v, int block,
                                      int hint)
{
    using namespace gbrng;
    if (kind < 0 || kind >= kKinds || fmt < 0 || fmt > 1 || size_class < 0 || size_class > 1 ||
        (v != 1 && v != 2) || block < 32 || block > 512 || (block & (block - 1)) || hint < 0 ||
        hint > 2)
        return set_error(RNG_ERR_ARG);
    Shape &s = shape_to_set(size_class, kind, fmt);
    s.v = v;
    s.block = block;
    s.hint = hint;
    return RNG_OK;
}

extern "C" int gbrng_set_launch_ctas(int kind, int fmt, int size_class, int ctas_per_sm)
{
    using namespace gbrng;
    if (kind < 0 || kind >= kKinds || fmt < 0 || fmt > 1 || size_class < 0 || size_class > 1 ||
        ctas_per_sm < 0 || ctas_per_sm > 1)
        return set_error(RNG_ERR_ARG);
    shape_to_set(size_class, kind, fmt).one = ctas_per_sm;
    return RNG_OK;
}

extern "C" int gbrng_get_launch_ctas(int kind, int fmt, int size_class, int *ctas_per_sm)
{
    using namespace gbrng;
    if (kind < 0 || kind >= kKinds || fmt < 0 || fmt > 1 || size_class < 0 || size_class > 1 ||
        !ctas_per_sm)
        return set_error(RNG_ERR_ARG);
    *ctas_per_sm = shape_in_use(size_class, kind, fmt).one;
    return RNG_OK;
}

extern "C" int gbrng_get_launch_class(int kind, int fmt, int size_class, int *v, int *block,
                                      int *hint)
{
    using namespace gbrng;
    if (kind < 0 || kind >= kKinds || fmt < 0 || fmt > 1 || size_class < 0 || size_class > 1 ||
        !v || !block || !hint)
        return set_error(RNG_ERR_ARG);
    *v = shape_in_use(size_class, kind, fmt).v;
    *block = shape_in_use(size_class, kind, fmt).block;
    *hint = shape_in_use(size_class, kind, fmt).hint;
    return RNG_OK;
}

extern "C" int gbrng_set_launch(int kind, int fmt, int v, int block, int hint)
{
    return gbrng_set_launch_class(kind, fmt, 1, v, block, hint);
}

extern "C" int gbrng_set_split(int kind, int log2_rows)
{
    using namespace gbrng;
    if (kind < 0 || kind >= kKinds || log2_rows < 0 || log2_rows > 30)
        return set_error(RNG_ERR_ARG);
    g_split_log2[kind] = log2_rows;
    return RNG_OK;
}

extern "C" int gbrng_get_split(int kind, int *log2_rows)
{
    using namespace gbrng;
    if (kind < 0 || kind >= kKinds || !log2_rows)
        return set_error(RNG_ERR_ARG);
    *log2_rows = g_split_log2[kind];
    return RNG_OK;
}

extern "C" int gbrng_get_launch(int kind, int fmt, int *v, int *block, int *hint)
{
    return gbrng_get_launch_class(kind, fmt, 1, v, block, hint);
}
