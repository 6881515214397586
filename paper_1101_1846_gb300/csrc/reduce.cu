// Inline consumers (rng_generate_reduce): every stream advances exactly as
// in rng_generate, each output is consumed in registers where it is made,
// and only one 64-bit result per stream and the final state are written.
// This is the paper's second regime, generation without writing the numbers
// back (Sec. "Performance evaluation"; Tables I-III), with the numbers
// actually used so that no step can be optimised away.  The kernels step
// the streams through Engine<KIND> of the public device header, the same
// path a user kernel takes.
//
// One stream per thread, loaded with coalesced 4-byte accesses across the
// warp.  Few streams with long sequences are split into segments of 2^l
// rows (split_segments; grid y = segment) that start from jumped states; their
// results are added into out with 64-bit atomics (exact, in any order), and
// the final state is written back by the last arrival, as in gen_split.
#include "jump.cuh"

namespace gbrng {
namespace {

constexpr int kThreads = 256;
constexpr unsigned kOneCtaEach = 152;  // CTAs of which every SM has one

// The next output.  MWC32 steps by a wide product and two carrying adds here:
// that takes the adds off the FMA-heavy pipe, which bounds its consumers
// (2^22 x 1024 on GB300: sum_u32 810 -> 699 us a call, disc 1029 -> 934), where
// KISS, whose ALU pipe is as full, would lose 2-5 % by it.
// disc steps the base-2^16 kinds with one part's low half on the FMA pipe
// (76,636 x 4096: MWC16X2 110 us without it, 103 with it, 106 with both parts';
// KISS_XOR 202, 191 and 196; the sums are faster with mwc16x2_step, 682 against
// 693 at 16,384 rows).
template <int KIND, bool DISC = false>
__device__ __forceinline__ uint32_t next_of(Engine<KIND> &e)
{
    if constexpr (KIND == RNG_MWC16X2 && DISC) {
        return mwc16x2_step_fma<1>(e.a, e.z, e.w);
    } else if constexpr (KIND == RNG_KISS_XOR && DISC) {
        return (mwc16x2_step_fma<1>(e.a, e.z, e.w) ^ lcg_step(e.l)) + xorshift32_step(e.y);
    } else if constexpr (KIND == RNG_MWC32) {
        uint32_t lo, hi;
        asm("{\n\t.reg .u64 q;\n\t.reg .u32 l, h;\n\t"
            "mul.wide.u32 q, %2, %3;\n\t"
            "mov.b64 {l, h}, q;\n\t"
            "add.cc.u32 %0, l, %4;\n\t"
            "addc.u32 %1, h, 0;\n\t}"
            : "=r"(lo), "=r"(hi)
            : "r"(e.a), "r"(e.x), "r"(e.c));
        e.x = lo;
        e.c = hi;
        return lo;
    } else {
        return e.next();
    }
}

// A pair (u0, u1) is inside when X^2 + Y^2 < 2^48, X = u0 >> 8, Y = u1 >> 8.
template <int KIND, bool DISC = true>
__device__ __forceinline__ uint32_t disc_pair(Engine<KIND> &e)
{
    const uint64_t X = next_of<KIND, DISC>(e) >> 8;
    const uint64_t Y = next_of<KIND, DISC>(e) >> 8;
    return (X * X + Y * Y) >> 48 == 0 ? 1u : 0u;
}

// kPairs pairs, counted exactly, mostly in FP32.  With f0, f1 the outputs
// rounded to FP32 (no shift), d = f0^2 + (f1^2 - 2^64) is off
// (256 X)^2 + (256 Y)^2 - 2^64 by less than 2^43: f0 is off 256 X by at most
// 255 + 128, hence its square by 383 x 2^33, twice, and the two roundings by
// 2^39 each.  So d's sign decides where |d| >= 2^43, and a block with a
// smaller |d| (16 pi/4 2^-20: one in 83,000 of a thread's blocks) is counted
// again in integers from the state it began with.
// The integer test's two wide multiply-adds share the FMA-heavy pipe with the
// MWC and LCG steps; the conversions, the sign's add and the minimum run on
// the ALU pipe and the FP32 multiply-adds on either half of the FMA pipe.
// 2^22 x 1024 on GB300, us a call, integer test -> this: MWC 1385 -> 1029 (934
// with next_of's step), xor128 2164 -> 1580, KISS 2323 -> 1967.
constexpr int kPairs = 16;

template <int KIND>
__device__ __forceinline__ uint32_t disc_block(Engine<KIND> &e)
{
    const Engine<KIND> begin = e;
    uint32_t inside = 0;
    float least = 0x1p64f;
#pragma unroll
    for (int j = 0; j < kPairs; ++j) {
        const float f0 = __uint2float_rn(next_of<KIND, true>(e));
        const float f1 = __uint2float_rn(next_of<KIND, true>(e));
        const float d = __fmaf_rn(f0, f0, __fmaf_rn(f1, f1, -0x1p64f));
        inside += __float_as_uint(d) >> 31;
        least = fminf(least, fabsf(d));
    }
    if (least < 0x1p43f) {
        e = begin;
        inside = 0;
#pragma unroll 1
        for (int j = 0; j < kPairs; ++j)
            inside += disc_pair(e);
    }
    return inside;
}

// The sums run in chunks with a 32-bit counter and an unroll of 32: loop
// bookkeeping then costs little beside the step (the MWC sum measured 11 %
// faster on GB300 than with a 64-bit counter and an unroll of 8; the other
// kinds were unchanged).  256 values of 24 bits fit 32: their chunks add up
// in 32 bits, one shifted add per output in place of a shift and a 64-bit
// add.
template <int OP, bool SPLIT, int KIND>
__device__ __forceinline__ uint64_t consume(Engine<KIND> &e, uint64_t m)
{
    uint64_t acc = 0;
    if constexpr (OP == RNG_SUM_U32) {
        for (uint64_t done = 0; done < m;) {
            const uint32_t k = (uint32_t)(m - done < (1u << 30) ? m - done : (1u << 30));
#pragma unroll 32
            for (uint32_t j = 0; j < k; ++j)
                acc += next_of(e);
            done += k;
        }
    } else if constexpr (OP == RNG_SUM_U24) {
        for (; m >= 256; m -= 256) {
            uint32_t part = 0;
#pragma unroll 32
            for (int j = 0; j < 256; ++j)
                part += next_of(e) >> 8;
            acc += part;
        }
        uint32_t part = 0;
        for (uint32_t j = 0; j < (uint32_t)m; ++j)
            part += next_of(e) >> 8;
        acc += part;
    } else {
        // kPairs pairs at a time by disc_block, the rest one by one
        uint64_t left = m / 2;
        if constexpr (KIND == RNG_KISS_XOR && !SPLIT) {
            // A whole call of this kind (at most 76,636 streams) has few rows;
            // with at most a CTA per SM it takes the integer test, whose chain is
            // shorter (us, blocks and pairs: 4 x 198 6.9 and 5.0, 20,000 x 256
            // 10.8 and 9.0; 76,636 x 256 15.3 and 15.9).
            if (gridDim.x <= kOneCtaEach)
#pragma unroll 4
                for (; left; --left)
                    acc += disc_pair<KIND, false>(e);
        }
        for (; left >= kPairs; left -= kPairs)
            acc += disc_block(e);
        for (; left; --left)
            acc += disc_pair(e);
        if (m & 1)
            next_of(e);  // the unpaired last output is drawn and ignored
    }
    return acc;
}

// An engine's state as the vector bodies hold one stream (w[word][0], a[0]),
// and back.
template <int KIND>
__device__ __forceinline__ void engine_words(const Engine<KIND> &e, uint32_t (&w)[kMaxWords][4],
                                             uint32_t (&a)[4])
{
    if constexpr (KIND == RNG_MWC32) {
        w[0][0] = e.x, w[1][0] = e.c, a[0] = e.a;
    } else if constexpr (KIND == RNG_XOR128) {
        w[0][0] = e.s0, w[1][0] = e.s1, w[2][0] = e.s2, w[3][0] = e.s3;
    } else if constexpr (KIND == RNG_KISS) {
        w[0][0] = e.x, w[1][0] = e.c, w[2][0] = e.y, w[3][0] = e.z, a[0] = e.a;
    } else if constexpr (KIND == RNG_MWC16X2) {
        w[0][0] = e.z, w[1][0] = e.w, a[0] = e.a;
    } else if constexpr (KIND == RNG_XORSHIFT8) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
            w[q][0] = e.v[q];
    } else {
        w[0][0] = e.z, w[1][0] = e.w, w[2][0] = e.y, w[3][0] = e.l, a[0] = e.a;
    }
}

template <int KIND>
__device__ __forceinline__ void engine_from_words(Engine<KIND> &e,
                                                  const uint32_t (&w)[kMaxWords][4])
{
    if constexpr (KIND == RNG_MWC32) {
        e.x = w[0][0], e.c = w[1][0];
    } else if constexpr (KIND == RNG_XOR128) {
        e.s0 = w[0][0], e.s1 = w[1][0], e.s2 = w[2][0], e.s3 = w[3][0];
    } else if constexpr (KIND == RNG_KISS) {
        e.x = w[0][0], e.c = w[1][0], e.y = w[2][0], e.z = w[3][0];
    } else if constexpr (KIND == RNG_MWC16X2) {
        e.z = w[0][0], e.w = w[1][0];
    } else if constexpr (KIND == RNG_XORSHIFT8) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
            e.v[q] = w[q][0];
    } else {
        e.z = w[0][0], e.w = w[1][0], e.y = w[2][0], e.l = w[3][0];
    }
}

// SPLIT = false: one segment (grid y = 1), the whole call per thread.
template <int KIND, int OP, bool SPLIT>
__global__ void __launch_bounds__(kThreads)
reduce_kernel(rng_device_view v, uint64_t steps, uint64_t rows, uint64_t *__restrict__ out,
              uint32_t *__restrict__ stash, uint32_t *__restrict__ counters,
              const uint64_t *__restrict__ jmul, JumpTables T)
{
    const uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (!SPLIT) {
        if (s >= v.n_streams)
            return;
        Engine<KIND> e;
        e.load(v, s);
        out[s] = consume<OP, SPLIT>(e, steps);
        e.store(v, s);
        return;
    }
    const bool live = s < v.n_streams;
    const uint32_t segs = gridDim.y;
    const uint64_t n = v.n_streams;
    const uint64_t first = (uint64_t)blockIdx.y * rows;
    const uint64_t mine = steps - first < rows ? steps - first : rows;
    uint32_t *state = static_cast<uint32_t *>(v.state);
    uint32_t *cnt = counters + s;
    Engine<KIND> e;
    // Split: the same arrival count as gen_split (one counter per stream).
    if (live) {
        e.load(v, s);
        __threadfence();
        if (atomicAdd(cnt, 1u) == segs) {
            __threadfence();
            for (int k = 0; k < v.state_words; ++k)
                state[k * n + s] = __ldcg(stash + k * n + s);
            *cnt = 0;
        }
    }
    if (blockIdx.y > 0) {
        __shared__ SegmentJump<KIND> jump;
        jump.fill(first, T);
        if (live) {
            uint32_t w[kMaxWords][4] = {}, a[4] = {};
            engine_words(e, w, a);
            uint64_t A = 0;
            if ((KIND == RNG_MWC32 || KIND == RNG_KISS) && jmul)
                A = jmul[blockIdx.y * n + s];
            mwc_jump_streams<KIND, 1>(w, a, first, A ? &A : nullptr);
            jump.template apply<1>(w);
            engine_from_words(e, w);
        }
    }
    if (!live)
        return;  // after the CTA's part of the jump
    atomicAdd(reinterpret_cast<unsigned long long *>(out + s),
              (unsigned long long)consume<OP, SPLIT>(e, mine));
    if (blockIdx.y == segs - 1) {
        rng_device_view f = v;
        f.state = stash;
        e.store(f, s);
        __threadfence();
        if (atomicAdd(cnt, 1u) == segs) {
            e.store(v, s);
            *cnt = 0;
        }
    }
}

using ReduceFn = void (*)(rng_device_view, uint64_t, uint64_t, uint64_t *, uint32_t *,
                          uint32_t *, const uint64_t *, JumpTables);

template <int KIND, bool SPLIT>
ReduceFn pick(int op)
{
    if (op == RNG_SUM_U32)
        return reduce_kernel<KIND, RNG_SUM_U32, SPLIT>;
    if (op == RNG_SUM_U24)
        return reduce_kernel<KIND, RNG_SUM_U24, SPLIT>;
    return reduce_kernel<KIND, RNG_DISC, SPLIT>;
}

template <bool SPLIT>
ReduceFn pick_kind(int kind, int op)
{
    switch (kind) {
    case RNG_MWC32: return pick<RNG_MWC32, SPLIT>(op);
    case RNG_XOR128: return pick<RNG_XOR128, SPLIT>(op);
    case RNG_KISS: return pick<RNG_KISS, SPLIT>(op);
    case RNG_MWC16X2: return pick<RNG_MWC16X2, SPLIT>(op);
    case RNG_XORSHIFT8: return pick<RNG_XORSHIFT8, SPLIT>(op);
    default: return pick<RNG_KISS_XOR, SPLIT>(op);
    }
}

}  // namespace
}  // namespace gbrng

using namespace gbrng;

extern "C" int rng_generate_reduce(rng_handle h, uint64_t n_per_stream, int op, void *out)
{
    Gen *g = reinterpret_cast<Gen *>(h);
    if (!g || !out || (uintptr_t)out % 8 != 0 ||
        (op != RNG_SUM_U32 && op != RNG_SUM_U24 && op != RNG_DISC))
        return set_error(RNG_ERR_ARG);
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != g->device && cudaSetDevice(g->device) != cudaSuccess)
        return set_error(RNG_ERR_CUDA);
    cudaStream_t st = g->stream;
    uint64_t *o = static_cast<uint64_t *>(out);
    rng_device_view v{g->kind, g->device, g->words, g->n, g->d_state, g->d_a};
    // pairs never straddle segments: their rows are an even number
    Segments seg{n_per_stream, 1, false};
    const bool split = g->d_split &&
                       split_wanted(g->kind, SplitForm::kReduce, RNG_U32, g->n, n_per_stream) &&
                       split_segments(g->kind, SplitForm::kReduce, RNG_U32, g->n, n_per_stream,
                                      (g->n + kThreads - 1) / kThreads, 0, g->jmul_segs, &seg);
    const uint64_t rows = seg.rows, segs = seg.count;
    ReduceFn fn = split ? pick_kind<true>(g->kind, op) : pick_kind<false>(g->kind, op);
    JumpTables T{};
    const uint64_t *jmul = nullptr;
    int status = RNG_OK;
    if (split && needs_jump_tables(g->kind))
        status = jump_tables(&T);
    // no table build inside a CUDA graph capture (see gen_kernels.cuh)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (!status && split)
        status = cuda_status(cudaStreamIsCapturing(st, &cap));
    if (!status && split && mont_table(g->kind) && cap == cudaStreamCaptureStatusNone)
        status = mwc_jump_table(g, rows, segs, st, &jmul);
    if (!status && split)
        status = cuda_status(cudaMemsetAsync(o, 0, g->n * 8, st));
    if (!status) {
        const dim3 grid((unsigned)((g->n + kThreads - 1) / kThreads), (unsigned)segs);
        fn<<<grid, kThreads, 0, st>>>(v, n_per_stream, rows, o, g->d_split, g->d_cnt, jmul, T);
        status = cuda_status(cudaGetLastError());
    }
    if (prev >= 0 && prev != g->device)
        cudaSetDevice(prev);
    return status;
}
