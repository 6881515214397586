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

// v <- M v for a 128 x 128 GF(2) matrix given by columns (word w of column j
// in col[j]); the four streams of a group share every column load.
template <int G>
__device__ __forceinline__ void gf2_apply128(const uint4 *__restrict__ col,
                                             uint32_t (&w)[kMaxWords][4])
{
    uint32_t r[4][G];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < G; ++i)
            r[q][i] = 0;
#pragma unroll
    for (int word = 0; word < 4; ++word) {
#pragma unroll 4
        for (int b = 0; b < 32; ++b) {
            const uint4 m = __ldg(col + 32 * word + b);
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const uint32_t mask = 0u - ((w[word][i] >> b) & 1u);
                r[0][i] ^= m.x & mask;
                r[1][i] ^= m.y & mask;
                r[2][i] ^= m.z & mask;
                r[3][i] ^= m.w & mask;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < G; ++i)
            w[q][i] = r[q][i];
}

// v <- M v for a 256 x 256 GF(2) matrix: column j is col[2j] (words 0-3)
// and col[2j + 1] (words 4-7).
template <int G>
__device__ __forceinline__ void gf2_apply256(const uint4 *__restrict__ col,
                                             uint32_t (&w)[kMaxWords][4])
{
    uint32_t r[8][G];
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int i = 0; i < G; ++i)
            r[q][i] = 0;
#pragma unroll
    for (int word = 0; word < 8; ++word) {
#pragma unroll 2
        for (int b = 0; b < 32; ++b) {
            const uint4 lo = __ldg(col + 2 * (32 * word + b));
            const uint4 hi = __ldg(col + 2 * (32 * word + b) + 1);
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const uint32_t mask = 0u - ((w[word][i] >> b) & 1u);
                r[0][i] ^= lo.x & mask;
                r[1][i] ^= lo.y & mask;
                r[2][i] ^= lo.z & mask;
                r[3][i] ^= lo.w & mask;
                r[4][i] ^= hi.x & mask;
                r[5][i] ^= hi.y & mask;
                r[6][i] ^= hi.z & mask;
                r[7][i] ^= hi.w & mask;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int i = 0; i < G; ++i)
            w[q][i] = r[q][i];
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

// Jumps G streams held as w[word][i] (the vector bodies' layout; G = 1 for
// a single stream) with multipliers a[i] by k steps.  With MWC_DONE the
// base-2^32 MWC words are left alone (the caller has applied a tabulated
// multiplier).
template <int KIND, int G, bool MWC_DONE = false>
__device__ __forceinline__ void jump_streams(uint32_t (&w)[kMaxWords][4],
                                             const uint32_t (&a)[4], uint64_t k,
                                             const JumpTables &T)
{
    if (k == 0)
        return;
    if constexpr ((KIND == RNG_MWC32 || KIND == RNG_KISS) && !MWC_DONE) {
#pragma unroll
        for (int i = 0; i < G; ++i)
            mwc_jump(a[i], w[0][i], w[1][i], k);
    }
    if constexpr (KIND == RNG_MWC16X2 || KIND == RNG_KISS_XOR) {
#pragma unroll
        for (int i = 0; i < G; ++i) {
            mwc16_jump(a[i] & 0xFFFFu, w[0][i], k);
            mwc16_jump(a[i] >> 16, w[1][i], k);
        }
    }
    if constexpr (KIND == RNG_XOR128) {
        for (uint64_t r = k; r; r &= r - 1)
            gf2_apply128<G>(T.xor128 + 128 * (__ffsll((long long)r) - 1), w);
    }
    if constexpr (KIND == RNG_XORSHIFT8) {
        for (uint64_t r = k; r; r &= r - 1)
            gf2_apply256<G>(T.xs8 + 512 * (__ffsll((long long)r) - 1), w);
    }
    if constexpr (KIND == RNG_KISS || KIND == RNG_KISS_XOR) {
        for (uint64_t r = k; r; r &= r - 1) {
            const int m = __ffsll((long long)r) - 1;
            const uint2 lc = __ldg(T.lcg + m);
#pragma unroll
            for (int i = 0; i < G; ++i) {
                w[2][i] = gf2_apply32(T.xs32 + 32 * m, w[2][i]);
                w[3][i] = lc.x * w[3][i] + lc.y;
            }
        }
    }
}

// The same for one stream in an Engine.  A != 0 (MWC32, KISS): the MWC part
// is multiplied by A = a^k in Montgomery form (a tabulated power) instead of
// powering.
template <int KIND>
__device__ __forceinline__ void jump_engine(Engine<KIND> &e, uint64_t k, const JumpTables &T,
                                            uint64_t A = 0)
{
    uint32_t w[kMaxWords][4] = {};
    uint32_t a[4] = {};
    if constexpr (KIND == RNG_MWC32) {
        w[0][0] = e.x;
        w[1][0] = e.c;
        a[0] = e.a;
    } else if constexpr (KIND == RNG_XOR128) {
        w[0][0] = e.s0;
        w[1][0] = e.s1;
        w[2][0] = e.s2;
        w[3][0] = e.s3;
    } else if constexpr (KIND == RNG_KISS) {
        w[0][0] = e.x;
        w[1][0] = e.c;
        w[2][0] = e.y;
        w[3][0] = e.z;
        a[0] = e.a;
    } else if constexpr (KIND == RNG_MWC16X2) {
        w[0][0] = e.z;
        w[1][0] = e.w;
        a[0] = e.a;
    } else if constexpr (KIND == RNG_XORSHIFT8) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
            w[q][0] = e.v[q];
    } else {
        w[0][0] = e.z;
        w[1][0] = e.w;
        w[2][0] = e.y;
        w[3][0] = e.l;
        a[0] = e.a;
    }
    if constexpr (KIND == RNG_MWC32 || KIND == RNG_KISS) {
        if (A != 0 && k != 0) {
            mwc_apply(A, a[0], w[0][0], w[1][0]);
            jump_streams<KIND, 1, true>(w, a, k, T);
        } else {
            jump_streams<KIND, 1>(w, a, k, T);
        }
    } else {
        jump_streams<KIND, 1>(w, a, k, T);
    }
    if constexpr (KIND == RNG_MWC32) {
        e.x = w[0][0];
        e.c = w[1][0];
    } else if constexpr (KIND == RNG_XOR128) {
        e.s0 = w[0][0];
        e.s1 = w[1][0];
        e.s2 = w[2][0];
        e.s3 = w[3][0];
    } else if constexpr (KIND == RNG_KISS) {
        e.x = w[0][0];
        e.c = w[1][0];
        e.y = w[2][0];
        e.z = w[3][0];
    } else if constexpr (KIND == RNG_MWC16X2) {
        e.z = w[0][0];
        e.w = w[1][0];
    } else if constexpr (KIND == RNG_XORSHIFT8) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
            e.v[q] = w[q][0];
    } else {
        e.z = w[0][0];
        e.w = w[1][0];
        e.y = w[2][0];
        e.l = w[3][0];
    }
}

}  // namespace gbrng
