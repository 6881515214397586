// The generation kernels, templated on the generator kind, and
// launch_kind<KIND>, which picks the kernel for a call.  Included by the
// translation units that instantiate them (generate.cu: the three target
// kinds; generate_paper.cu: the paper's own generators), so that each one
// compiles only its kinds.
//
// Every thread keeps the state of its streams in
// registers for the whole call, steps them n times and writes each step's
// outputs with one 16-byte store per group of four adjacent streams, so a
// warp writes 512 contiguous bytes of one output row per store instruction.
// The paper's kernels (Sec. "GPU implementations": MWC, XorShift in
// registers, KISS) keep one stream per thread with 4-byte stores; four
// streams per thread give the 16-byte stores and four independent
// dependency chains per thread.
//
// Layout: output j of stream s at out[j*ld + s] (ld = n_streams for a plain
// call); state word w of stream s at state[w*n + s].
//
// Paths (chosen per call by launch_kind):
//   aligned  n % 4 == 0 and out 16-byte aligned: gen_vec when every row is
//            32-byte aligned (a CTA of B threads covers 4*V*B consecutive
//            streams, thread t owns the groups starting at base + 4t + 4Bv,
//            v < V), else gen_vec_sync (one group per thread, barriers);
//   shifted  otherwise, for the first n & ~3 streams: gen_shift, rows written
//            with 16-byte stores after a warp-shuffle realignment;
//   tail     the last n % 4 streams, taken by one extra CTA of gen_shift with
//            4-byte stores.
// Calls of few streams split into jumped segments: gen_split (aligned rows)
// or gen_split_shift (the others).
#pragma once

#include <algorithm>

#include "gen_body.cuh"
#include "jump.cuh"

namespace gbrng {
namespace {

// Streams [s_begin, s_begin + count) of the generator; out points at the
// output element of stream s_begin in row 0.
template <int KIND, int FMT, int V, int HINT>
__global__ void __launch_bounds__(512)
gen_vec(uint32_t *__restrict__ state, const uint32_t *__restrict__ mult, uint64_t n,
        uint32_t steps, uint32_t *__restrict__ out, uint64_t ld, uint64_t s_begin,
        uint64_t count)
{
    const uint64_t B = blockDim.x;
    const uint64_t c_first = (uint64_t)blockIdx.x * (4 * V) * B + 4 * (uint64_t)threadIdx.x;
    if (V == 2 && c_first + 4 * B < count)
        body_vec<KIND, FMT, V, HINT>(state, mult, n, steps, out + c_first, ld,
                                     s_begin + c_first, 4 * B);
    else if (c_first < count)
        body_vec<KIND, FMT, 1, HINT>(state, mult, n, steps, out + c_first, ld,
                                     s_begin + c_first, 4 * B);
}

// Rows 16-byte but not 32-byte aligned: one group per thread, barriers every
// SYNC_ROWS rows; every thread runs the rows (idle groups store nothing).
template <int KIND, int FMT, int HINT>
__global__ void __launch_bounds__(512)
gen_vec_sync(uint32_t *__restrict__ state, const uint32_t *__restrict__ mult, uint64_t n,
             uint32_t steps, uint32_t *__restrict__ out, uint64_t ld, uint64_t s_begin,
             uint64_t count)
{
    const uint64_t c_first = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    body_vec_sync<KIND, FMT, HINT>(state, mult, n, steps, out + c_first, ld, s_begin + c_first,
                                   c_first < count);
}

// The first count & ~3 streams in realigned groups of four, 31K + 1 groups
// per CTA of K warps (see body_shift); the last CTA of the grid takes the
// count % 4 tail streams (one per thread), alongside the CTAs of the last wave
// where these leave it a place (even_threads sees to that).
template <int KIND, int FMT, int HINT>
__global__ void __launch_bounds__(512)
gen_shift(uint32_t *__restrict__ state, const uint32_t *__restrict__ mult, uint64_t n,
          uint32_t steps, uint32_t *__restrict__ out, uint64_t ld, uint64_t s_begin,
          uint64_t count)
{
    const uint64_t main = count & ~(uint64_t)3;
    if (main < count && blockIdx.x == gridDim.x - 1) {
        uint64_t c = main + threadIdx.x;
        if (c < count)
            body_scalar<KIND, FMT, HINT>(state, mult, n, steps, out + c, ld, s_begin + c);
        return;
    }
    const uint64_t per_cta = 31 * (blockDim.x / 32) + 1;
    const uint64_t g0 = (uint64_t)blockIdx.x * per_cta;
    const uint64_t left = main / 4 - g0;
    body_shift<KIND, FMT, HINT>(state, mult, n, steps, out + 4 * g0, ld, s_begin + 4 * g0,
                                (uint32_t)(left < per_cta ? left : per_cta));
}

// Dynamic shared memory (nothing is stored there) that keeps gen_split of 16-
// but not 32-byte rows to three CTAs of 256 threads per SM: as in the
// barrier-synced kernels, fewer warps writing at once keep the write stream
// denser.  GB300, us a call without it and with it (two per SM: 397, 378 and 395
// at 76,636 x 8192, against 377, 382 and 379 with three and 447, 415 and 417
// without, MWC, KISS and MWC16X2):
//                    MWC u32   f32       KISS u32  MWC16X2 u32  xor128 u32
//   20,004 x 4096     59  56    58  59    64  62    69  59       84  84
//   40,004 x 4096    109 105   111 102   110 112   110 103      118 120
//   60,004 x 8192    323 303   328 299   317 298   325 302      337 329
//   76,636 x 8192    403 380   417 379   410 386   410 378      397 405
// KISS f32 is within 2 % either way.  KISS_XOR and XORSHIFT8, bound by their
// arithmetic, keep as many as fit (XORSHIFT8, of whose CTAs with their 24 KB
// matrix only two would: f32 40,004 x 16,384 823 797, 10,004 x 8192 224 217).
constexpr int kSyncSplitSmem = 60 * 1024;

// Warps of groups per CTA of gen_split_shift (125 groups), beside its tail warp.
constexpr int kShiftSplitWarps = 4;

// Sequence splitting (Sec. "Parallelizing RNGs") for calls with too few
// streams to fill the device: segment y of the grid produces rows
// [y*rows, min(steps, (y+1)*rows)) of every stream, starting from the state
// jumped ahead by y*rows steps (the MWC part by the handle's tabulated
// multiplier a^(y*rows), the xorshift and LCG parts, which all streams of a
// segment share, composed by each CTA from the device tables: SegmentJump).
// One group of four streams per thread, rows 32-byte aligned (as gen_vec).
//
// Writing the final state back must wait until every segment has read the
// start state, and no segment may wait for another.  So each thread counts
// its arrival on the group's counter right after reading the start state;
// the last segment also stashes its final state and counts once more.  The
// arrival that brings the count to segments + 1 sees every read done and the
// final state ready: it writes the state (from registers or the stash) and
// clears the counter for the next call.
//
// SYNC: rows 16- but not 32-byte aligned.  As in body_vec_sync, a barrier
// every SYNC_ROWS rows keeps the CTA's warps together so that the two halves of
// a shared DRAM sector meet in L2; every thread of the CTA then runs the
// rows (a CTA shares its segment, hence its jump and its row count), and
// threads past the last group store nothing and count no arrival.
template <int KIND, int FMT>
__device__ __forceinline__ uint32_t split_step(uint32_t (&w)[kMaxWords][4],
                                               const uint32_t (&a)[4], int i)
{
    // KISS_XOR is bound by the ALU pipe here (76,636 x 4096, us: u32 194 with
    // kiss_xor_step, 184 with the join alone moved, 192 with both low halves as
    // well; f32, which adds a shift, a conversion and a product, 245, 230, 210)
    if constexpr (KIND == RNG_KISS_XOR) {
        const uint32_t u = (mwc16x2_step_fma<FMT == RNG_F32 ? 2 : 0>(a[i], w[0][i], w[1][i]) ^
                            lcg_step(w[3][i])) +
                           xorshift32_step(w[2][i]);
        return FMT == RNG_F32 ? __float_as_uint(unit_f32(u)) : u;
    } else {
        return step_enc<KIND, FMT>(w, a, i);
    }
}

template <int KIND, int FMT, int HINT, bool SYNC>
__global__ void __launch_bounds__(256)
gen_split(uint32_t *__restrict__ state, const uint32_t *__restrict__ mult, uint64_t n,
          uint32_t steps, uint32_t rows, uint32_t *__restrict__ out, uint64_t ld,
          uint64_t s_begin, uint64_t count, uint32_t *__restrict__ stash,
          uint32_t *__restrict__ counters, const uint64_t *__restrict__ jmul, JumpTables T)
{
    uint64_t c_first = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    const bool live = c_first < count;
    if (!live)
        c_first = 0;  // compute on stream 0's state, never store
    constexpr int W = KindTraits<KIND>::W;
    const uint64_t s0 = s_begin + c_first;
    const uint32_t segs = gridDim.y;
    const uint32_t y = blockIdx.y;
    const uint32_t first = y * rows;
    const uint32_t mine = min(rows, steps - first);
    uint32_t w[kMaxWords][4] = {};
    uint32_t a[4] = {};
#pragma unroll
    for (int k = 0; k < W; ++k)
        load4(state + k * n + s0, w[k]);
    if constexpr (KindTraits<KIND>::MULT)
        load4(mult + s0, a);
    __threadfence();  // the reads above are done before the arrival is counted
    uint32_t *cnt = counters + s0 / 4;
    const bool finish = live && atomicAdd(cnt, 1u) == segs;
    if (finish) {
        // every other arrival, the stash included, came first
        __threadfence();
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const uint4 q = __ldcg(reinterpret_cast<const uint4 *>(stash + k * n + s0));
            *reinterpret_cast<uint4 *>(state + k * n + s0) = q;
        }
        *cnt = 0;
    }
    if (y > 0) {
        __shared__ SegmentJump<KIND> jump;
        jump.fill(first, T);
        // the threads past the last group only help to compose: 24 streams x 15,000
        // rows, us a call with their powers and without, MWC captured 10.2 and 6.7,
        // MWC16X2 11.9 and 7.9, KISS_XOR 16.3 and 12.3
        if (!SYNC && !live)
            return;
        // MWC32 / KISS: the tabulated a^(y*rows) when the handle's table is
        // passed, else powering (calls captured in a CUDA graph)
        bool powers = !SYNC || live;
        if constexpr (KIND == RNG_MWC32 || KIND == RNG_KISS) {
            if (jmul) {
                const uint4 lo =
                    __ldg(reinterpret_cast<const uint4 *>(jmul + (uint64_t)y * n + s0));
                const uint4 hi =
                    __ldg(reinterpret_cast<const uint4 *>(jmul + (uint64_t)y * n + s0 + 2));
                const uint64_t A[4] = {(uint64_t)lo.y << 32 | lo.x, (uint64_t)lo.w << 32 | lo.z,
                                       (uint64_t)hi.y << 32 | hi.x, (uint64_t)hi.w << 32 | hi.z};
                mwc_jump_streams<KIND, 4>(w, a, first, A);
                powers = false;
            }
        }
        if (powers)
            mwc_jump_streams<KIND, 4>(w, a, first, nullptr);
        if (!SYNC || live)
            jump.template apply<4>(w);
    }
    if (!SYNC && !live)
        return;
    uint32_t *row = out + (uint64_t)first * ld + c_first;
    if constexpr (SYNC) {
        for (uint32_t j = 0; j < mine; ++j) {
            if (j % KindTraits<KIND>::SYNC_ROWS == 0)
                __syncthreads();
            const uint32_t o0 = split_step<KIND, FMT>(w, a, 0);
            const uint32_t o1 = split_step<KIND, FMT>(w, a, 1);
            const uint32_t o2 = split_step<KIND, FMT>(w, a, 2);
            const uint32_t o3 = split_step<KIND, FMT>(w, a, 3);
            if (live)
                store16<HINT>(row, o0, o1, o2, o3);
            row += ld;
        }
        if (!live)
            return;  // after the last barrier
    } else {
#pragma unroll 4
        for (uint32_t j = 0; j < mine; ++j) {
            const uint32_t o0 = split_step<KIND, FMT>(w, a, 0);
            const uint32_t o1 = split_step<KIND, FMT>(w, a, 1);
            const uint32_t o2 = split_step<KIND, FMT>(w, a, 2);
            const uint32_t o3 = split_step<KIND, FMT>(w, a, 3);
            store16<HINT>(row, o0, o1, o2, o3);
            row += ld;
        }
    }
    if (y == segs - 1) {
#pragma unroll
        for (int k = 0; k < W; ++k)
            save4(stash + k * n + s0, w[k]);
        __threadfence();  // the stash is visible before its arrival is counted
        if (atomicAdd(cnt, 1u) == segs) {
#pragma unroll
            for (int k = 0; k < W; ++k)
                save4(state + k * n + s0, w[k]);
            *cnt = 0;
        }
    }
}

// Sequence splitting for rows that are not 16-byte aligned: gen_split's
// segments and arrival counts with body_shift's realigned rows.  A CTA holds
// 31K + 1 groups of four streams in K = `warps` warps (one halo lane per warp
// but the last), the same ones in every segment, and, when count % 4 != 0,
// one more warp, whose first lanes take the last count % 4 streams in the
// last CTA of a segment.  A halo lane starts from the same state as its
// group's owner; the barrier after the loads puts its read before the owner's
// arrival, so the arrivals of owners and tail lanes (one counter per first
// stream) cover every read.
//
// The row's alignment r is uniform over the CTA and goes through r, r + dr, ..
// mod 4 (dr = ld mod 4), a cycle of at most four rows: up to three rows with r
// chosen at run time lead to the cycle's fixed start (shift_cycle_start), the
// blocks of four rows that follow have every r at compile time (eight
// sequences, where gen_shift, which starts at any r, has sixteen, in two
// forms), and at most three rows are left.
// MWC powers are taken in the kernel when the handle's table does not already
// hold them: this path never allocates and never waits.
// On GB300, us a call, whole calls -> this: KISS f32 1001 x 16384 1587 -> 30.7
// (46.6 with a run-time alignment and 32 columns per set bit of the jump), KISS
// u32 10,001 x 8192 370 -> 79, MWC 76,633 x 4096 278 -> 194.
template <int KIND, int FMT, int HINT, int R0, int DR>
__device__ __forceinline__ void shift_cycle(uint32_t (&w)[kMaxWords][4], const uint32_t (&a)[4],
                                            uint32_t *&row, uint64_t ld, uint32_t blocks,
                                            bool owner, bool prev, bool next, bool lead,
                                            bool trail)
{
    OutMap m;
    shift_rows<KIND, FMT, HINT, R0, DR, true>(w, a, row, ld, blocks, owner, prev, next, lead,
                                              trail, m);
}

// Rows until the alignment is one that shift_cycle has: 0 for dr = 1 and 3
// (the cycle has all four), 0 or 1 for dr = 2, any for dr = 0.
__device__ __forceinline__ uint32_t shift_cycle_start(uint32_t r, uint32_t dr)
{
    return dr == 0 ? 0 : dr == 1 ? (4 - r) & 3 : dr == 2 ? r >> 1 : r;
}

template <int KIND, int FMT, int HINT>
__global__ void __launch_bounds__(32 * (kShiftSplitWarps + 1))
gen_split_shift(uint32_t *__restrict__ state, const uint32_t *__restrict__ mult, uint64_t n,
                uint32_t steps, uint32_t rows, uint32_t *__restrict__ out, uint64_t ld,
                uint64_t s_begin, uint64_t count, int warps, uint32_t *__restrict__ stash,
                uint32_t *__restrict__ counters, const uint64_t *__restrict__ jmul, JumpTables T)
{
    constexpr int W = KindTraits<KIND>::W;
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
    const uint64_t main = count & ~(uint64_t)3;
    const uint32_t per_cta = warps ? 31 * warps + 1 : 0;
    const uint64_t g0 = (uint64_t)blockIdx.x * per_cta;
    const uint32_t groups = (uint32_t)min((uint64_t)per_cta, main / 4 - g0);
    const bool tail_warp = k == warps;  // count % 4 streams, one per lane
    const uint32_t g = 31u * k + lane;
    const bool live = tail_warp ? blockIdx.x == gridDim.x - 1 && lane < (int)(count - main)
                                : g < groups;
    const bool owner = live && (tail_warp || lane < 31 || k == warps - 1);
    const bool lead = g == 0;
    const bool trail = owner && g == groups - 1;
    const bool prev = live && lane > 0;
    const bool next = owner && lane < 31 && g + 1 < groups;
    // the thread's first stream, counted from s_begin, and how many it has
    const uint64_t c = !live ? 0 : tail_warp ? main + lane : 4 * (g0 + g);
    const int mine = tail_warp ? 1 : 4;
    const uint64_t s0 = s_begin + c;
    const uint32_t segs = gridDim.y, y = blockIdx.y, first = y * rows;
    const uint32_t n_rows = min(rows, steps - first);
    uint32_t w[kMaxWords][4] = {};
    uint32_t a[4] = {};
    if (live) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // a tail lane holds its stream four times
            const uint64_t s = s0 + (tail_warp ? 0 : i);
#pragma unroll
            for (int q = 0; q < W; ++q)
                w[q][i] = state[q * n + s];
            if constexpr (KindTraits<KIND>::MULT)
                a[i] = mult[s];
        }
    }
    __syncthreads();  // halo states are read before any arrival is counted
    auto save = [&](uint32_t *to) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < mine)
#pragma unroll
                for (int q = 0; q < W; ++q)
                    to[q * n + s0 + i] = w[q][i];
    };
    uint32_t *cnt = counters + s0;
    if (owner) {
        __threadfence();
        if (atomicAdd(cnt, 1u) == segs) {  // the stash was ready before
            __threadfence();
            for (int i = 0; i < mine; ++i)
                for (int q = 0; q < W; ++q)
                    state[q * n + s0 + i] = __ldcg(stash + q * n + s0 + i);
            *cnt = 0;
        }
    }
    if (y > 0) {
        __shared__ SegmentJump<KIND> jump;
        jump.fill(first, T);
        if (live) {
            if ((KIND == RNG_MWC32 || KIND == RNG_KISS) && jmul) {
                uint64_t A[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    A[i] = __ldg(jmul + (uint64_t)y * n + s0 + (tail_warp ? 0 : i));
                mwc_jump_streams<KIND, 4>(w, a, first, A);
            } else {
                mwc_jump_streams<KIND, 4>(w, a, first, nullptr);
            }
            jump.template apply<4>(w);
        }
    }
    uint32_t *row = out + (uint64_t)first * ld + c;
    if (!tail_warp && !live)
        row = out;  // never stored to; keeps the alignment's arithmetic in range
    const uint32_t dr = (uint32_t)(ld & 3);
    uint32_t r = (uint32_t)(((uintptr_t)(out + (uint64_t)first * ld) >> 2) & 3);
    const uint32_t lead_in = min(shift_cycle_start(r, dr), n_rows);
    const uint32_t blocks = (n_rows - lead_in) / 4, rest = (n_rows - lead_in) % 4;
    if (tail_warp) {
        auto step = [&] {
            const uint32_t o = step_enc<KIND, FMT>(w, a, 0);
            if (live)
                store4<HINT>(row, o);
            row += ld;
        };
        for (uint32_t j = 0; j < lead_in; ++j)
            step();
        for (uint32_t b = 0; b < blocks; ++b) {
            if (b % (KindTraits<KIND>::SYNC_ROWS / 4) == 0)
                __syncthreads();  // with shift_rows
            step();
            step();
            step();
            step();
        }
        for (uint32_t j = 0; j < rest; ++j)
            step();
    } else {
        OutMap m;
        auto one = [&] {
            shift_row_rt<KIND, FMT, HINT>(w, a, row, r, owner, prev, next, lead, trail, m);
            row += ld;
            r = (r + dr) & 3u;
        };
#pragma unroll 1
        for (uint32_t j = 0; j < lead_in; ++j)
            one();
#define GBRNG_SHIFT_CYCLE(R0_, DR_)                                                             \
    case (DR_) * 4 + (R0_):                                                                     \
        shift_cycle<KIND, FMT, HINT, R0_, DR_>(w, a, row, ld, blocks, owner, prev, next, lead,  \
                                               trail);                                          \
        break;
        if (blocks)
            switch (dr * 4 + r) {
                GBRNG_SHIFT_CYCLE(0, 0) GBRNG_SHIFT_CYCLE(1, 0) GBRNG_SHIFT_CYCLE(2, 0)
                GBRNG_SHIFT_CYCLE(3, 0) GBRNG_SHIFT_CYCLE(0, 1) GBRNG_SHIFT_CYCLE(0, 2)
                GBRNG_SHIFT_CYCLE(1, 2) GBRNG_SHIFT_CYCLE(0, 3)
            default: break;
            }
#undef GBRNG_SHIFT_CYCLE
#pragma unroll 1
        for (uint32_t j = 0; j < rest; ++j)
            one();
    }
    if (y == segs - 1 && owner) {
        save(stash);
        __threadfence();
        if (atomicAdd(cnt, 1u) == segs) {
            save(state);
            *cnt = 0;
        }
    }
}

// Rows 32-byte aligned, outputs staged in shared memory and written by the
// TMA engine (bulk asynchronous copies, shared -> global): a CTA of
// kTmaThreads threads owns 4 * kTmaThreads consecutive streams (one group
// of four per thread), generates kTmaRows rows at a time into one of two
// shared buffers, and one thread writes each row's segment (4 KB for 1024
// streams) with one bulk copy.  A buffer is refilled only after its
// copies have finished reading it (wait_group.read), and the kernel waits
// for every copy before it ends.  Threads past the last stream run the rows
// with the others (the barriers are CTA-wide) and their words are not
// copied.
constexpr int kTmaThreads = 256;
constexpr int kTmaRows = 4;

__device__ __forceinline__ void tma_store_row(uint32_t *gdst, const uint32_t *ssrc,
                                              uint32_t bytes)
{
    const uint32_t saddr = static_cast<uint32_t>(__cvta_generic_to_shared(ssrc));
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                 :
                 : "l"(gdst), "r"(saddr), "r"(bytes)
                 : "memory");
}

template <int KIND, int FMT>
__global__ void __launch_bounds__(kTmaThreads)
gen_tma(uint32_t *__restrict__ state, const uint32_t *__restrict__ mult, uint64_t n,
        uint32_t steps, uint32_t *__restrict__ out, uint64_t ld, uint64_t s_begin,
        uint64_t count)
{
    __shared__ __align__(128) uint32_t buf[2][kTmaRows][4 * kTmaThreads];
    constexpr int W = KindTraits<KIND>::W;
    const uint64_t c0 = (uint64_t)blockIdx.x * 4 * kTmaThreads;  // CTA's first stream
    const uint64_t c_first = c0 + 4 * (uint64_t)threadIdx.x;
    const bool live = c_first < count;
    const uint32_t bytes = (uint32_t)(4 * min((uint64_t)4 * kTmaThreads, count - c0));
    const uint64_t s0 = s_begin + c_first;
    uint32_t w[kMaxWords][4] = {};
    uint32_t a[4] = {};
    if (live) {
#pragma unroll
        for (int k = 0; k < W; ++k)
            load4(state + k * n + s0, w[k]);
        if constexpr (KindTraits<KIND>::MULT)
            load4(mult + s0, a);
    }
    const bool leader = threadIdx.x == 0;
    uint32_t row0 = 0;
    for (int b = 0; row0 < steps; b ^= 1, row0 += kTmaRows) {
        const uint32_t rows = min((uint32_t)kTmaRows, steps - row0);
        if (leader)  // the copies that read this buffer two blocks ago are done
            asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        __syncthreads();
        for (uint32_t r = 0; r < rows; ++r) {
            const uint32_t o0 = step_enc<KIND, FMT>(w, a, 0);
            const uint32_t o1 = step_enc<KIND, FMT>(w, a, 1);
            const uint32_t o2 = step_enc<KIND, FMT>(w, a, 2);
            const uint32_t o3 = step_enc<KIND, FMT>(w, a, 3);
            *reinterpret_cast<uint4 *>(&buf[b][r][4 * threadIdx.x]) = make_uint4(o0, o1, o2, o3);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (leader) {
            for (uint32_t r = 0; r < rows; ++r)
                tma_store_row(out + (uint64_t)(row0 + r) * ld + c0, &buf[b][r][0], bytes);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
    }
    if (leader)
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (live) {
#pragma unroll
        for (int k = 0; k < W; ++k)
            save4(state + k * n + s0, w[k]);
    }
}

constexpr int kSMs = 152;
// 4096 x 128 u32 on GB300, device time of a whole call in us, two groups per
// thread (MWC u32 by TMA: 8.6 for 4096 x 64) against one: MWC 8.7 and 5.4 (3.4),
// KISS 12.9 and 7.3, xor128 9.8 and 4.8, MWC16X2 8.5 and 5.0, KISS_XOR 14.0 and
// 7.6 (9.9 with streaming stores); 4096 x 8: KISS 2.2 and 1.8, MWC16X2 1.9 and
// 1.7, KISS_XOR 2.2 and 1.9; 65,536 x 2: KISS 1.8 and 1.7, the others the same.
constexpr uint64_t kSmallCall = (uint64_t)kSMs * 1024;
// CTA size of the kernels with row barriers: large CTAs leave fewer CTA
// boundaries, where neighbouring CTAs that drift apart split sectors.
constexpr int kSyncBlock = 512;

// CTA size for `units` thread-sized pieces of work: shrink until the grid
// covers every SM (small problems), never below one warp.
inline int fit_threads(int threads, uint64_t units)
{
    while (threads > 32 && (units + threads - 1) / threads < kSMs)
        threads /= 2;
    return threads;
}

// CTAs of one size in whole waves of one per SM.  A call of a few waves ends
// with its last one, which a fixed CTA size leaves nearly empty: 700,000 streams
// in CTAs of 4096 are 171 CTAs, and 19 of 152 SMs write the second half.  Where
// less than kEvenFill of the SMs' time is used, the CTAs are made smaller, equal,
// and at most as many as whole waves hold.  Every size from one to thirteen waves was
// timed both ways; above that fill they differ by a few percent either way.
// GB300, TB/s, fixed and even sizes (r: realigned rows), fill:
//   KISS u32    668,784 x 470  0.54  4.58  6.45    191,762r x 1640 0.64  4.45  6.11
//   KISS f32    200,090r x 1572 0.67 3.87  5.82    373,321r x 842  0.62  3.97  5.16
//   xor128 u32   96,528 x 162  0.62  3.42  4.26    177,530r x 1771 0.59  4.15  6.21
//   xor128 f32  663,488 x 474  0.53  4.46  7.08    348,553r x 902  0.58  4.06  5.29
//   XORSHIFT8   197,272 x 1594 0.63  4.29  5.69    338,148r x 930  0.56  3.74  5.01
//   MWC u32     344,340 x 913  0.57  4.79  6.25    359,769r x 874  0.60  4.95  6.78
//   MWC f32     641,408 x 490  0.52  4.91  7.13    187,794r x 1675 0.62  4.46  5.95
constexpr double kEvenFill = 0.8;

// Groups of four streams a CTA of `threads` holds: one a thread, or for
// realigned rows 31 a warp and one.
inline uint64_t groups_of(int threads, bool realigned)
{
    return realigned ? 31 * (threads / 32) + 1 : threads;
}

// Whether even CTAs keep an SM to themselves (one_cta_smem): the realigned
// FP32 kernels, whose conversions wait longer, and XORSHIFT8 run faster beside
// one another.
inline bool even_alone(int kind, int fmt, bool realigned)
{
    return kind != RNG_XORSHIFT8 && !(realigned && fmt == RNG_F32 && kind != RNG_MWC32);
}

// The CTA size for `groups` groups of four, 0 where CTAs of `per_cta` groups
// fill their waves.  XORSHIFT8, whose steps take the longest, wants the warps of
// whole SMs; the others write in denser streams from at most 256 threads, and
// xor128, whose steps take the shortest, 32-byte rows from 128 (f32 calls of
// 1.2 GB, TB/s in CTAs of 160-224 and of 96-128: 173,440 streams 4.96 6.07,
// 195,160 5.68 6.54, 255,048 6.35 6.38).
// tail: one more CTA follows, for the last streams of realigned rows.  Where the
// others would fill their waves exactly it would run after them, so they leave it
// a place, unless that puts more warps on a scheduler or they are three waves or
// more that share their SMs (us without the place and with it: XORSHIFT8 340,321 x
// 924 363, 246, but 453,409 x 693, 13 warps for 12, 214, 259; xor128 f32 189,537 x
// 1659 278, 217, but 340,929 x 922, three waves, 222, 239; KISS u32 340,929 x 922
// 228, 210).
inline int even_threads(int kind, int fmt, uint64_t groups, uint64_t per_cta, bool sectors,
                        bool realigned, bool tail)
{
    const uint64_t ctas = (groups + per_cta - 1) / per_cta;
    const uint64_t waves = (ctas + kSMs - 1) / kSMs;
    if (groups <= (uint64_t)kSMs * 128 ||  // at most one warp a scheduler in any case
        (double)groups >= kEvenFill * (double)(per_cta * kSMs * waves))
        return 0;
    const uint64_t most =
        kind == RNG_XORSHIFT8 ? 512 : kind == RNG_XOR128 && sectors ? 128 : 256;
    auto threads_for = [&](uint64_t places) {
        const uint64_t each = (groups + places - 1) / places;
        return std::max<uint64_t>(
            32, realigned ? 32 * ((each - 1 + 30) / 31) : 32 * ((each + 31) / 32));
    };
    for (uint64_t k = 1;; ++k) {
        const uint64_t threads = threads_for(kSMs * k);
        if (threads > most)
            continue;
        // the CTA of the last streams, which steps them one to a thread
        const uint64_t each = groups_of((int)threads, realigned);
        if (tail && (groups + each - 1) / each == kSMs * k &&
            (k <= 2 || even_alone(kind, fmt, realigned))) {
            const uint64_t wider = threads_for(kSMs * k - 1);
            if (wider <= most && (wider + 127) / 128 == (threads + 127) / 128)
                return (int)wider;
        }
        return (int)threads;
    }
}

// V = 2 only for kinds of at most four state words: two groups of the
// eight-word XORSHIFT8 would not fit the registers of a 512-thread CTA.
template <int KIND, int FMT>
void pick_vec(int v, int hint,
              void (*&vec)(uint32_t *, const uint32_t *, uint64_t, uint32_t, uint32_t *,
                           uint64_t, uint64_t, uint64_t))
{
    if constexpr (KindTraits<KIND>::W <= 4) {
        if (v == 2) {
            vec = hint ? gen_vec<KIND, FMT, 2, 1> : gen_vec<KIND, FMT, 2, 0>;
            return;
        }
    }
    vec = hint ? gen_vec<KIND, FMT, 1, 1> : gen_vec<KIND, FMT, 1, 0>;
}

// Whether a call on `st` may use the handle's MWC table.  Inside a CUDA graph
// capture it is not (re)built: its kernel would only run at replay while later
// direct calls took it as ready.  Nor does a captured call keep its address:
// it may grow.
inline int table_allowed(cudaStream_t st, bool *allowed)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const int e = cuda_status(cudaStreamIsCapturing(st, &cap));
    *allowed = !e && cap == cudaStreamCaptureStatusNone;
    return e;
}

// A split call with 16-byte rows.  *done: launched (else it would have had a
// single segment).
template <int KIND>
int launch_split(int fmt, int hint, bool sectors, const GenLaunch &p, cudaStream_t st, bool *done)
{
    using Fn = void (*)(uint32_t *, const uint32_t *, uint64_t, uint32_t, uint32_t, uint32_t *,
                        uint64_t, uint64_t, uint64_t, uint32_t *, uint32_t *, const uint64_t *,
                        JumpTables);
    Fn fn;
    if (sectors)
        fn = fmt == RNG_F32 ? (hint ? gen_split<KIND, RNG_F32, 1, false>
                                    : gen_split<KIND, RNG_F32, 0, false>)
                            : (hint ? gen_split<KIND, RNG_U32, 1, false>
                                    : gen_split<KIND, RNG_U32, 0, false>);
    else
        fn = fmt == RNG_F32
                 ? (hint ? gen_split<KIND, RNG_F32, 1, true> : gen_split<KIND, RNG_F32, 0, true>)
                 : (hint ? gen_split<KIND, RNG_U32, 1, true> : gen_split<KIND, RNG_U32, 0, true>);
    Gen *g = p.owner;
    const uint64_t count = p.s_end - p.s_begin, tiles = (count / 4 + 255) / 256;
    const bool dense = KIND != RNG_KISS_XOR && KIND != RNG_XORSHIFT8;
    const int smem = !sectors && dense ? kSyncSplitSmem : 0;
    Segments seg;
    const SplitForm form = sectors ? SplitForm::kAligned : SplitForm::kRows16;
    if (!split_segments(KIND, form, fmt, count, p.steps, tiles,
                        resident_ctas((const void *)fn, 256, smem), g->jmul_segs, &seg))
        return RNG_OK;
    JumpTables T{};
    const uint64_t *jmul = nullptr;
    bool table = false;
    int e = needs_jump_tables(KIND) ? jump_tables(&T) : RNG_OK;
    if (!e && mont_table(KIND) && seg.table)
        e = table_allowed(st, &table);
    if (!e && table)
        e = mwc_jump_table(g, seg.rows, seg.count, st, &jmul);
    if (e)
        return e;
    *done = true;
    fn<<<dim3((unsigned)tiles, (unsigned)seg.count), 256, smem, st>>>(
        p.state, p.a, p.n, (uint32_t)p.steps, (uint32_t)seg.rows, static_cast<uint32_t *>(p.out),
        p.ld, p.s_begin, count, g->d_split, g->d_cnt, jmul, T);
    return cuda_status(cudaGetLastError());
}

// The same for rows that are not 16-byte aligned; never allocates or waits.
template <int KIND>
int launch_split_shift(int fmt, const GenLaunch &p, cudaStream_t st, bool *done)
{
    auto fn =
        fmt == RNG_F32 ? gen_split_shift<KIND, RNG_F32, 1> : gen_split_shift<KIND, RNG_U32, 1>;
    Gen *g = p.owner;
    // groups spread evenly over as few CTAs per segment as hold them
    const uint64_t count = p.s_end - p.s_begin;
    const uint64_t groups = count / 4, most = 31 * kShiftSplitWarps + 1;
    const uint64_t few = std::max<uint64_t>((groups + most - 1) / most, 1);
    const uint64_t per = (groups + few - 1) / few;
    const int warps = per < 2 ? (int)per : (int)((per - 1 + 30) / 31);
    const uint64_t tiles = warps ? (groups + 31 * warps) / (31 * warps + 1) : 1;
    const int threads = 32 * (warps + (count % 4 ? 1 : 0));
    Segments seg;
    if (!split_segments(KIND, SplitForm::kShifted, fmt, count, p.steps, tiles,
                        resident_ctas((const void *)fn, threads, 0), g->jmul_segs, &seg))
        return RNG_OK;
    JumpTables T{};
    const uint64_t *jmul = nullptr;
    bool table = false;
    int e = needs_jump_tables(KIND) ? jump_tables(&T) : RNG_OK;
    if (!e && mont_table(KIND))
        e = table_allowed(st, &table);
    if (!e && table)
        e = ready_jump_table(g, seg.rows, seg.count, st, &jmul);
    if (e)
        return e;
    *done = true;
    fn<<<dim3((unsigned)tiles, (unsigned)seg.count), threads, 0, st>>>(
        p.state, p.a, p.n, (uint32_t)p.steps, (uint32_t)seg.rows, static_cast<uint32_t *>(p.out),
        p.ld, p.s_begin, count, warps, g->d_split, shift_counters(g), jmul, T);
    return cuda_status(cudaGetLastError());
}

// One generate call of a KIND generator: picks the path from how the rows
// sit in memory (aligned / synced / realigned), or splits a few-stream call
// into jumped segments.
template <int KIND>
int launch_kind(int fmt, const GenLaunch &p, cudaStream_t st)
{
    using Fn = void (*)(uint32_t *, const uint32_t *, uint64_t, uint32_t, uint32_t *, uint64_t,
                        uint64_t, uint64_t);
    const uint64_t count = p.s_end - p.s_begin;
    if (p.steps == 0 || count == 0)
        return RNG_OK;
    LaunchShape sh = launch_shape(KIND, fmt, count);
    const int split_hint = sh.hint;
    // 16-byte rows and 16-byte state groups: every group of four streams
    // starts on a 16-byte boundary in the output and in the state words.
    const bool aligned = (count % 4 == 0) && (p.ld % 4 == 0) && ((uintptr_t)p.out % 16 == 0) &&
                         (p.n % 4 == 0) && (p.s_begin % 4 == 0) &&
                         ((uintptr_t)p.state % 16 == 0) &&
                         (p.a == nullptr || (uintptr_t)p.a % 16 == 0);
    // whole 32-byte sectors per warp and row: no barriers needed
    const bool sectors = aligned && (p.ld % 8 == 0) && ((uintptr_t)p.out % 32 == 0);
    // The shape is for calls that fill the device.  Below kSmallCall streams
    // there is less than a CTA of it per SM: one group of four per thread then
    // (two halve the warps), and 16-byte stores (TMA rows come in CTAs of 1024
    // streams).  A single warp holds one group per thread anyway.  The kernels of other rows, which
    // take only the store hint from the shape, keep it: their form without it is
    // up to twice as slow (KISS_XOR u32, 20,000 streams x 100 rows from an odd
    // word, us: 8.2 with streaming stores, 12.3 without).
    if (sectors && !sh.set && count < kSmallCall &&
        (sh.hint == 2 || (sh.v == 2 && count > 128))) {
        sh.v = 1;
        sh.hint = 0;
    }
    const uint64_t main = count & ~(uint64_t)3;
    const int sync_threads = fit_threads(kSyncBlock, main / 4);
    const int vec_threads = fit_threads(sh.block, main / 4 / sh.v);
    // KISS with 32-byte rows: FP32 takes CTAs of 128, as many as fit, which even
    // out by themselves, and so do uint32 CTAs of less than 512 threads (311,776
    // streams: 6.6 TB/s, 5.4 in three even waves).  A caller's own shape stays.
    const bool fixed = sectors ? sh.set || (KIND == RNG_KISS &&
                                            (fmt == RNG_F32 || vec_threads < sh.block))
                               : row_ctas_set(KIND, fmt, !aligned);
    int even = 0;
    if (!fixed)
        even = even_threads(KIND, fmt, main / 4,
                            !sectors       ? groups_of(sync_threads, !aligned)
                            : sh.hint == 2 ? kTmaThreads
                                           : sh.v * vec_threads,
                            sectors, !aligned, !aligned && count > main);
    const bool alone = even && even_alone(KIND, fmt, !aligned);
    if (even && sectors) {
        sh.v = 1;
        sh.hint = sh.hint ? 1 : 0;
    }
    Fn vec, shift, sync;
    if (fmt == RNG_F32) {
        pick_vec<KIND, RNG_F32>(sh.v, sh.hint, vec);
        shift = sh.hint ? gen_shift<KIND, RNG_F32, 1> : gen_shift<KIND, RNG_F32, 0>;
        sync = sh.hint ? gen_vec_sync<KIND, RNG_F32, 1> : gen_vec_sync<KIND, RNG_F32, 0>;
    } else {
        pick_vec<KIND, RNG_U32>(sh.v, sh.hint, vec);
        shift = sh.hint ? gen_shift<KIND, RNG_U32, 1> : gen_shift<KIND, RNG_U32, 0>;
        sync = sh.hint ? gen_vec_sync<KIND, RNG_U32, 1> : gen_vec_sync<KIND, RNG_U32, 0>;
    }
    uint32_t *out = static_cast<uint32_t *>(p.out);
    Gen *g = p.owner;
    const SplitForm form = sectors   ? SplitForm::kAligned
                           : aligned ? SplitForm::kRows16
                                     : SplitForm::kShifted;
    if (g && g->d_split && split_wanted(KIND, form, fmt, count, p.steps)) {
        bool done = false;
        const int e = aligned ? launch_split<KIND>(fmt, split_hint, sectors, p, st, &done)
                              : launch_split_shift<KIND>(fmt, p, st, &done);
        if (e || done)
            return e;
    }
    // Calls longer than 2^31 steps are cut into pieces (the kernels count
    // steps in 32 bits); the state carries from piece to piece.
    for (uint64_t done = 0; done < p.steps;) {
        const uint32_t steps = (uint32_t)std::min<uint64_t>(p.steps - done, 1u << 31);
        uint32_t *o = out + done * p.ld;
        if (aligned && !sectors) {
            const int threads = even ? even : sync_threads;
            uint64_t blocks = (count / 4 + threads - 1) / threads;
            if (blocks > 0x7FFFFFFFull)
                return set_error(RNG_ERR_ARG);
            const int smem = alone || (row_ctas(KIND, fmt, false) && threads == kSyncBlock)
                                 ? one_cta_smem((const void *)sync, threads)
                                 : 0;
            sync<<<(unsigned)blocks, threads, smem, st>>>(p.state, p.a, p.n, steps, o, p.ld,
                                                          p.s_begin, count);
        } else if (aligned && sh.hint == 2) {
            // outputs staged in shared memory, rows written by bulk copies
            const uint64_t blocks = (count + 4 * kTmaThreads - 1) / (4 * kTmaThreads);
            if (blocks > 0x7FFFFFFFull)
                return set_error(RNG_ERR_ARG);
            auto tma = fmt == RNG_F32 ? gen_tma<KIND, RNG_F32> : gen_tma<KIND, RNG_U32>;
            tma<<<(unsigned)blocks, kTmaThreads, 0, st>>>(p.state, p.a, p.n, steps, o, p.ld,
                                                          p.s_begin, count);
        } else if (aligned) {
            int threads = sh.block;
            uint64_t groups = count / 4;
            while (threads > 32 && (groups + (uint64_t)threads * sh.v - 1) /
                                           ((uint64_t)threads * sh.v) < kSMs)
                threads /= 2;
            if (even)
                threads = even;
            uint64_t per_block = (uint64_t)threads * sh.v;
            uint64_t blocks = (groups + per_block - 1) / per_block;
            if (blocks > 0x7FFFFFFFull)
                return set_error(RNG_ERR_ARG);
            // one CTA per SM only for the shape's own CTA size (small calls
            // halve it above to fill the SMs)
            const int smem = alone || (!even && sh.one && threads == sh.block)
                                 ? one_cta_smem((const void *)vec, threads)
                                 : 0;
            vec<<<(unsigned)blocks, threads, smem, st>>>(p.state, p.a, p.n, steps, o, p.ld,
                                                         p.s_begin, count);
        } else {
            // realigned groups plus, when count % 4 != 0, one more CTA for the tail
            const int threads = even ? even : sync_threads;
            const uint64_t per_cta = groups_of(threads, true);
            uint64_t blocks = (main / 4 + per_cta - 1) / per_cta + (count > main ? 1 : 0);
            if (blocks > 0x7FFFFFFFull)
                return set_error(RNG_ERR_ARG);
            const int smem = alone || (row_ctas(KIND, fmt, true) && threads == kSyncBlock)
                                 ? one_cta_smem((const void *)shift, threads)
                                 : 0;
            shift<<<(unsigned)blocks, threads, smem, st>>>(p.state, p.a, p.n, steps, o, p.ld,
                                                           p.s_begin, count);
        }
        int e = cuda_status(cudaGetLastError());
        if (e)
            return e;
        done += steps;
    }
    return RNG_OK;
}

}  // namespace
}  // namespace gbrng
