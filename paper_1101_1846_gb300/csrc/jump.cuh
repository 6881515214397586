// Jump-ahead on the device: the state of a stream k steps later without
// the steps in between (sequence splitting, Sec. "Parallelizing RNGs").
//
//   MWC     With p = a 2^32 - 1, the state as one number z = x + c 2^32
//           (0 < z < p) steps to a x + c = a z mod p (a 2^32 = 1 mod p;
//           Lehmer's generator in disguise), so k steps multiply z by
//           a^k mod p and no division is needed.  In Montgomery form with
//           R = 2^64, a R = 2^32 (mod p), and -p^-1 = 1 (mod 2^32): a
//           reduction step adds (low word) * a one word up (mwc_mont).
//           Multiplying a residue X by a is one MWC step of it.
//   xor128, xorshift32
//           GF(2)-linear: k steps apply M^k, the product of the tables'
//           M^(2^m) over the set bits m of k (powers of one matrix commute).
//   LCG     affine: the composed maps (A_m, C_m) of 2^m steps.
//   MWC16X2 each base-2^16 part by the same Lehmer argument with
//           p = a 2^16 - 1 < 2^32 and the packed word as z.
//   XORSHIFT8  GF(2) with 256 x 256 matrices (the tables' third part).
#pragma once

#include "gen_body.cuh"
#include "modarith.cuh"

namespace gbrng {

__device__ __forceinline__ uint64_t mwc_mul_a(uint64_t X, uint32_t a)
{
    return (uint64_t)a * (uint32_t)X + (X >> 32);
}

// A residue X Y 2^-64 (mod p = a 2^32 - 1), below 2^64 for any X, Y below
// 2^64: schoolbook words with the two reductions folded in, six wide
// multiply-adds where mont_mul for any modulus takes about twelve.  The sum
// before the last step is below 2^64 + p, so p comes off when it carried.
__device__ __forceinline__ uint64_t mwc_mont(uint64_t X, uint64_t Y, uint32_t a)
{
    const uint32_t x0 = (uint32_t)X, x1 = (uint32_t)(X >> 32);
    const uint32_t y0 = (uint32_t)Y, y1 = (uint32_t)(Y >> 32);
    const uint64_t t = (uint64_t)x0 * y0;
    const uint64_t s = (uint64_t)x0 * y1 + (t >> 32);
    const uint64_t s2 = (uint64_t)x1 * y0 + (uint32_t)s;
    const uint64_t s3 = (uint64_t)(uint32_t)t * a + (uint32_t)s2;  // clears word 0
    // at most (2^32 - 1)^2 + 2 (2^32 - 1) = 2^64 - 1
    const uint64_t u = (uint64_t)x1 * y1 + (s >> 32) + (s2 >> 32);
    uint32_t lo, hi, carry;
    asm("{\n\t.reg .u32 l, h, c;\n\t"
        "add.cc.u32 l, %3, %5;\n\t"          // u + (s3 >> 32)
        "addc.cc.u32 h, %4, 0;\n\t"
        "addc.u32 c, 0, 0;\n\t"
        "mad.lo.cc.u32 %0, %6, %7, l;\n\t"   // + (low word of s3) a: clears word 1
        "madc.hi.cc.u32 %1, %6, %7, h;\n\t"
        "addc.u32 %2, c, 0;\n\t}"
        : "=&r"(lo), "=&r"(hi), "=r"(carry)
        : "r"((uint32_t)u), "r"((uint32_t)(u >> 32)), "r"((uint32_t)(s3 >> 32)),
          "r"((uint32_t)s3), "r"(a));
    const uint64_t r = (uint64_t)hi << 32 | lo;
    return carry ? r + 1 - ((uint64_t)a << 32) : r;
}

// A residue of a^k (mod p), below 2^64, in Montgomery form, k >= 1.
__device__ __forceinline__ uint64_t mwc_power(uint32_t a, uint64_t k)
{
    uint64_t A = (uint64_t)1 << 32;  // a^1 in Montgomery form: the top bit of k
    for (int bit = 62 - __clzll((long long)k); bit >= 0; --bit) {
        A = mwc_mont(A, A, a);
        if ((k >> bit) & 1)
            A = mwc_mul_a(A, a);
    }
    return A;
}

// (x, c) <- the state k steps on, for A = a^k in Montgomery form.
__device__ __forceinline__ void mwc_apply(uint64_t A, uint32_t a, uint32_t &x, uint32_t &c)
{
    uint64_t z = mwc_mont(A, (uint64_t)c << 32 | x, a);  // below 2^64
    const uint64_t p = ((uint64_t)a << 32) - 1;
    while (z >= p)  // at most 2^64 / p times: 4 for the table's multipliers
        z -= p;
    x = (uint32_t)z;
    c = (uint32_t)(z >> 32);
}

__device__ __forceinline__ void mwc_jump(uint32_t a, uint32_t &x, uint32_t &c, uint64_t k)
{
    if (k != 0)
        mwc_apply(mwc_power(a, k), a, x, c);
}

// One base-2^16 part z = x + c 2^16, multiplier a < 2^16: k steps make it
// a^k z mod p, p = a 2^16 - 1.  The power is taken in Montgomery form with
// R = 2^32, where a is 2^16 and -p^-1 mod 2^32 is 1 + a 2^16, so nothing needs
// a division; left to right from k's top bit.
__device__ __forceinline__ void mwc16_jump(uint32_t a, uint32_t &z, uint64_t k)
{
    if (k == 0)
        return;
    const uint32_t p = (a << 16) - 1u;
    const uint32_t ninv = (a << 16) + 1u;
    uint32_t A = 1u << 16;  // a in Montgomery form
    for (int bit = 62 - __clzll((long long)k); bit >= 0; --bit) {
        A = mont_mul32(A, A, p, ninv);
        if ((k >> bit) & 1u)  // times a: h 2^16 + l -> a l + h
            A = a * (A & 0xFFFFu) + (A >> 16);
    }
    z = mont_mul32(A, z, p, ninv);  // a^k R z R^-1 mod p
}

__device__ __forceinline__ uint32_t gf2_apply32(const uint32_t *__restrict__ col, uint32_t y)
{
    uint32_t r = 0;
#pragma unroll 8
    for (int b = 0; b < 32; ++b)
        r ^= __ldg(col + b) & (0u - ((y >> b) & 1u));
    return r;
}

// Copies 16 bytes to shared memory without waiting.
__device__ __forceinline__ void copy16_async(void *shared, const void *global)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;"
                 :
                 : "r"((uint32_t)__cvta_generic_to_shared(shared)), "l"(global)
                 : "memory");
}

// Waits for the CTA's copies.
__device__ __forceinline__ void copies_done()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// v <- M v for a (32 W)-square GF(2) matrix in shared memory (column j at
// col[W j], W words) and one vector that every lane of the warp holds: lane l
// takes column l of each group of 32 and the lanes' parts are reduced, about
// 30 instructions at W = 4.
template <int W>
__device__ __forceinline__ void gf2_apply_warp(const uint32_t *col, uint32_t (&v)[W], int lane)
{
    uint32_t r[W] = {};
#pragma unroll
    for (int q = 0; q < W; ++q) {
        const uint32_t mask = 0u - ((v[q] >> lane) & 1u);
        if constexpr (W == 1) {
            r[0] ^= col[lane] & mask;
        } else {
#pragma unroll
            for (int h = 0; h < W / 4; ++h) {
                const uint4 m = reinterpret_cast<const uint4 *>(col + W * (32 * q + lane))[h];
                r[4 * h] ^= m.x & mask;
                r[4 * h + 1] ^= m.y & mask;
                r[4 * h + 2] ^= m.z & mask;
                r[4 * h + 3] ^= m.w & mask;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < W; ++q)
        v[q] = __reduce_xor_sync(0xFFFFFFFFu, r[q]);
}

// The xorshift32 and LCG parts of a jump by k, the same for every stream of a
// CTA: X^k as four byte tables (the image of byte value b at byte q of the
// word is xs[256 q + b]) and the affine map z -> A z + C.
struct __align__(16) KissJump {
    union {
        uint32_t level[64][32];  // the set bits' matrices, while X^k is composed
        uint32_t xs[1024];
    };
    uint32_t col[32];
    uint32_t A, C;
};

// Fills J for k >= 1; every thread of the CTA (a multiple of 32) calls this.
// The columns' chains run side by side, four per warp at 256 threads, on
// matrices copied in ahead of them (a chain of reads from L2 took 0.3 us a
// set bit).
__device__ __forceinline__ void kiss_jump_fill(KissJump &J, uint64_t k, const JumpTables &T)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int levels = __popcll(k);
    uint32_t A = 1, C = 0;
    int i = 0;
    for (uint64_t r = k; r; r &= r - 1, ++i) {
        const int m = __ffsll((long long)r) - 1;
        if (threadIdx.x < 8)
            copy16_async(&J.level[i][4 * threadIdx.x], T.xs32 + 32 * m + 4 * threadIdx.x);
        if (threadIdx.x == 8) {
            const uint2 map = __ldg(T.lcg + m);
            C = map.x * C + map.y;
            A = map.x * A;
        }
    }
    if (threadIdx.x == 8) {
        J.A = A;
        J.C = C;
    }
    copies_done();
    for (int j0 = 4 * warp; j0 < 32; j0 += 4 * warps) {
        uint32_t v[4][1];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            v[c][0] = 1u << (j0 + c);
        for (int m = 0; m < levels; ++m) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                gf2_apply_warp<1>(J.level[m], v[c], lane);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (lane == c)
                J.col[j0 + c] = v[c][0];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 1024; e += blockDim.x) {
        uint32_t x = 0;
#pragma unroll
        for (int b = 0; b < 8; ++b)
            x ^= J.col[8 * (e >> 8) + b] & (0u - ((uint32_t)(e >> b) & 1u));
        J.xs[e] = x;
    }
    __syncthreads();
}

__device__ __forceinline__ void kiss_jump_apply(const KissJump &J, uint32_t &y, uint32_t &z)
{
    y = J.xs[y & 255u] ^ J.xs[256 + ((y >> 8) & 255u)] ^ J.xs[512 + ((y >> 16) & 255u)] ^
        J.xs[768 + (y >> 24)];
    z = J.A * z + J.C;
}

// The same for one stream, a matrix per set bit of k.
__device__ __forceinline__ void kiss_jump_bits(uint32_t &y, uint32_t &z, uint64_t k,
                                               const JumpTables &T)
{
    for (uint64_t r = k; r; r &= r - 1) {
        const int m = __ffsll((long long)r) - 1;
        const uint2 lc = __ldg(T.lcg + m);
        y = gf2_apply32(T.xs32 + 32 * m, y);
        z = lc.x * z + lc.y;
    }
}

// The columns of M^k of a kind with a big GF(2) part, composed by the CTA from
// the set bits' matrices, a few of which are in shared memory at a time.
template <int W>
struct __align__(16) Gf2Jump {
    static constexpr int kAtOnce = W == 4 ? 4 : 2;
    uint32_t level[kAtOnce][32 * W * W];
    uint32_t col[32 * W * W];
};

// r <- M w for the G vectors of a thread (word q of vector i in w[q][i]; they
// share every column read) and a matrix in shared memory.
template <int W, int G, int N>
__device__ __forceinline__ void gf2_apply(const uint32_t *col, uint32_t (&w)[N][G])
{
    uint32_t r[W][G] = {};
#pragma unroll
    for (int word = 0; word < W; ++word) {
#pragma unroll 8
        for (int b = 0; b < 32; ++b) {
            const uint4 *c = reinterpret_cast<const uint4 *>(col + W * (32 * word + b));
#pragma unroll
            for (int h = 0; h < W / 4; ++h) {
                const uint4 m = c[h];
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    const uint32_t mask = 0u - ((w[word][i] >> b) & 1u);
                    r[4 * h][i] ^= m.x & mask;
                    r[4 * h + 1][i] ^= m.y & mask;
                    r[4 * h + 2][i] ^= m.z & mask;
                    r[4 * h + 3][i] ^= m.w & mask;
                }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < W; ++q)
#pragma unroll
        for (int i = 0; i < G; ++i)
            w[q][i] = r[q][i];
}

// Fills J for k >= 1; every thread of the CTA (a multiple of 32) calls this.
// A thread takes a column at a time through the levels in shared memory.
template <int W>
__device__ __forceinline__ void gf2_jump_fill(Gf2Jump<W> &J, uint64_t k,
                                              const uint32_t *__restrict__ table)
{
    constexpr int kWords = 32 * W * W;
    for (int i = threadIdx.x; i < kWords; i += blockDim.x)  // the identity
        J.col[i] = (i % W) == (i / W) / 32 ? 1u << (i / W % 32) : 0u;
    for (uint64_t r = k; r;) {
        int levels = 0;
        for (; levels < Gf2Jump<W>::kAtOnce && r; ++levels, r &= r - 1) {
            const uint32_t *src = table + (size_t)kWords * (__ffsll((long long)r) - 1);
            for (int i = 4 * threadIdx.x; i < kWords; i += 4 * blockDim.x)
                copy16_async(&J.level[levels][i], src + i);
        }
        copies_done();
#pragma unroll 1
        for (int j = threadIdx.x; j < 32 * W; j += blockDim.x) {
            uint32_t v[W][1];
#pragma unroll
            for (int q = 0; q < W; ++q)
                v[q][0] = J.col[W * j + q];
#pragma unroll 1
            for (int m = 0; m < levels; ++m)
                gf2_apply<W, 1, W>(J.level[m], v);
#pragma unroll
            for (int q = 0; q < W; ++q)
                J.col[W * j + q] = v[q][0];
        }
        __syncthreads();
    }
}

// w <- M w for the first G of a thread's four streams.
template <int W, int G>
__device__ __forceinline__ void gf2_jump_apply(const Gf2Jump<W> &J, uint32_t (&w)[kMaxWords][4])
{
    uint32_t v[W][G];
#pragma unroll
    for (int q = 0; q < W; ++q)
#pragma unroll
        for (int i = 0; i < G; ++i)
            v[q][i] = w[q][i];
    gf2_apply<W, G, W>(J.col, v);
#pragma unroll
    for (int q = 0; q < W; ++q)
#pragma unroll
        for (int i = 0; i < G; ++i)
            w[q][i] = v[q][i];
}

// The part of a segment's jump that all its streams share, composed once per
// CTA: a call's segments jump by first = y * rows, which has several set bits,
// and each cost every stream a matrix before.
template <int KIND>
struct SegmentJump {
    __device__ __forceinline__ void fill(uint64_t, const JumpTables &) {}
    template <int G>
    __device__ __forceinline__ void apply(uint32_t (&)[kMaxWords][4]) const
    {
    }
};
struct KissSegmentJump {
    KissJump J;
    __device__ __forceinline__ void fill(uint64_t k, const JumpTables &T)
    {
        kiss_jump_fill(J, k, T);
    }
    template <int G>
    __device__ __forceinline__ void apply(uint32_t (&w)[kMaxWords][4]) const
    {
#pragma unroll
        for (int i = 0; i < G; ++i)
            kiss_jump_apply(J, w[2][i], w[3][i]);
    }
};
template <>
struct SegmentJump<RNG_KISS> : KissSegmentJump {
};
template <>
struct SegmentJump<RNG_KISS_XOR> : KissSegmentJump {
};
template <>
struct SegmentJump<RNG_XOR128> {
    Gf2Jump<4> J;
    __device__ __forceinline__ void fill(uint64_t k, const JumpTables &T)
    {
        gf2_jump_fill<4>(J, k, reinterpret_cast<const uint32_t *>(T.xor128));
    }
    template <int G>
    __device__ __forceinline__ void apply(uint32_t (&w)[kMaxWords][4]) const
    {
        gf2_jump_apply<4, G>(J, w);
    }
};
template <>
struct SegmentJump<RNG_XORSHIFT8> {
    Gf2Jump<8> J;
    __device__ __forceinline__ void fill(uint64_t k, const JumpTables &T)
    {
        gf2_jump_fill<8>(J, k, reinterpret_cast<const uint32_t *>(T.xs8));
    }
    template <int G>
    __device__ __forceinline__ void apply(uint32_t (&w)[kMaxWords][4]) const
    {
        gf2_jump_apply<8, G>(J, w);
    }
};

// Jumps the MWC parts of G streams held as w[word][i] (the vector bodies'
// layout) with multipliers a[i] by k steps; A (MWC32, KISS): the tabulated
// powers a[i]^k in Montgomery form, or nullptr.
template <int KIND, int G>
__device__ __forceinline__ void mwc_jump_streams(uint32_t (&w)[kMaxWords][4],
                                                 const uint32_t (&a)[4], uint64_t k,
                                                 const uint64_t *A)
{
#pragma unroll
    for (int i = 0; i < G; ++i) {
        if constexpr (KIND == RNG_MWC32 || KIND == RNG_KISS) {
            if (A)
                mwc_apply(A[i], a[i], w[0][i], w[1][i]);
            else
                mwc_jump(a[i], w[0][i], w[1][i], k);
        }
        if constexpr (KIND == RNG_MWC16X2 || KIND == RNG_KISS_XOR) {
            mwc16_jump(a[i] & 0xFFFFu, w[0][i], k);
            mwc16_jump(a[i] >> 16, w[1][i], k);
        }
    }
}

}  // namespace gbrng
