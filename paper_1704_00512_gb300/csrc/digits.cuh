// Fixed-point digits of FP32 and FP64 values for f16 tensor-core products (what they
// are and why: colstep.cu, which runs the recursion on them; product.cu has the FP64
// masked products).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"

namespace cheb {

// Tiles of an element type: NT n8-tiles (2 block columns each) per panel, and the
// grid exponents that the recursion takes: of T's columns, to the end of the finite
// numbers, and of the operator's scalar rows (a byte each; FP64: OP_MAX + EX_MAX - 47 is
// an exponent too).
template <typename T>
struct Dig;
template <>
struct Dig<float> {
    static constexpr int NT = 2, EX_MIN = -90, EX_MAX = 128, OP_MIN = -80, OP_MAX = 30;
};
template <>
struct Dig<double> {
    static constexpr int NT = 1, EX_MIN = -400, EX_MAX = 1024, OP_MIN = -127, OP_MAX = 46;
};

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// --- digits ----------------------------------------------------------------

// |x| as an unsigned that orders like |x| and is largest for infinities and NaN
__device__ __forceinline__ uint32_t mag_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t mag_bits(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

// mag_bits of infinities and NaN and no others is at least this
template <typename T>
constexpr uint32_t NOT_FINITE = sizeof(T) == 4 ? 0x7f800000u : 0x7ff00000u;

// Grid exponent e of values with largest magnitude bits m: every |x| < 0.997 2^e
// (0 for all zeros).  false: not finite, or e outside [lo, hi].
template <typename T>
__device__ __forceinline__ bool grid_exp(uint32_t m, int lo, int hi, int &e) {
    e = 0;
    if (m == 0u) return true;
    if constexpr (sizeof(T) == 4) {
        e = (int)(m >> 23) - 126 + ((m & 0x7fffffu) >= 0x7f0000u ? 1 : 0);
    } else {
        e = (int)(m >> 20) - 1022 + ((m & 0xfffffu) >= 0xfe000u ? 1 : 0);
    }
    return m < NOT_FINITE<T> && e >= lo && e <= hi;
}
// 2^e as a float / double (e within the normal range)
__device__ __forceinline__ float pow2(int e, float) { return __int_as_float((e + 127) << 23); }
__device__ __forceinline__ double pow2(int e, double) { return __hiloint2double((e + 1023) << 20, 0); }

// x on the grid of exponent e with an offset that makes every digit
// non-negative.  FP32: 30 bits of x 2^(29 - e); FP64: 60 bits of x 2^(59 - e),
// 512 in each of the six digits.
__device__ __forceinline__ int grid_value(float x, int e) { return __float2int_rn(x * pow2(29 - e, 0.f)); }
__device__ __forceinline__ uint64_t grid_value(double x, int e) {
    const uint64_t bits = (uint64_t)__double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7ff), sh = ex - 1016 - e;
    const uint64_t mant = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
    uint64_t mag = 0;
    if (ex > 0 && sh > -54) mag = sh >= 0 ? mant << sh : (mant + (1ull << (-sh - 1))) >> -sh;
    const int64_t q = (bits >> 63) ? -(int64_t)mag : (int64_t)mag;
    return (uint64_t)q + 0x0802008020080200ull;
}

// fp16x2 arithmetic on packed digits (all values and results exact)
__device__ __forceinline__ uint32_t h2_sub(uint32_t x, uint32_t y) {
    uint32_t r;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(y));
    return r;
}
__device__ __forceinline__ uint32_t h2_fma(uint32_t x, uint32_t y, uint32_t z) {
    uint32_t r;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(y), "r"(z));
    return r;
}
// Two 10-bit biased digits (bits 0-9 and 16-25) as f16 integers: the bits under
// the f16 exponent of 1024, less 1024 + 512.
__device__ __forceinline__ uint32_t f16_digits(uint32_t d) { return h2_sub(d | 0x64006400u, 0x66006600u); }

// FP32 operator digits of a pair, packed (q = h_0 2^20 + h_1 2^10 + h_2, 10 bits
// each): h_0 of both in word 0 and h_1 in word 1 (bits 0-9, 16-25), h_2 spread
// over bits 10-15 / 26-31 of word 0 (its upper 6) and 10-13 / 26-29 of word 1.
__device__ __forceinline__ void pack_pair(uint32_t (&w)[2], int q0, int q1) {
    const uint32_t u = (uint32_t)q0 + 0x20080200u, v = (uint32_t)q1 + 0x20080200u;
    w[0] = ((u >> 20) & 0x3ffu) | ((u & 0x3f0u) << 6) | (((v >> 20) & 0x3ffu) << 16) | ((v & 0x3f0u) << 22);
    w[1] = ((u >> 10) & 0x3ffu) | ((u & 0xfu) << 10) | (((v >> 10) & 0x3ffu) << 16) | ((v & 0xfu) << 26);
}
__device__ __forceinline__ uint32_t spread_digit(uint32_t w0, uint32_t w1) {
    return f16_digits(((w1 >> 10) & 0x000f000fu) | ((w0 >> 6) & 0x03f003f0u));
}
// FP32 panel digits of a pair: q = d_0 2^19 + d_1 2^8 + d_2, 11, 11 and 8 bits;
// w[0] = d_0, w[1] = d_1 / 2 as f16, the third digits + 128 as bytes in third.
// (d_1 / 2 and 2 d_2 carry the weights that the operator's 10-bit digits have.)
__device__ __forceinline__ void panel_digits(uint32_t (&w)[2], uint32_t &third, int q0, int q1) {
    const uint32_t off = (1024u << 19) + (1024u << 8) + 128u;
    const uint32_t u = (uint32_t)q0 + off, v = (uint32_t)q1 + off;
    auto h2 = [](int a, int b) {
        const __half2 h = __floats2half2_rn((float)a, (float)b);  // (off the conversion unit)
        return *reinterpret_cast<const uint32_t *>(&h);
    };
    w[0] = h2((int)(u >> 19) - 1024, (int)(v >> 19) - 1024);
    w[1] = h2((int)((u >> 8) & 0x7ffu) - 1024, (int)((v >> 8) & 0x7ffu) - 1024);
    w[1] = h2_fma(w[1], 0x38003800u, 0u);  // * 0.5
    third = (u & 0xffu) | ((v & 0xffu) << 8);
}
// 2 d_2 of a pair from its bytes: selected under the exponent of 1024
template <int SEL>
__device__ __forceinline__ uint32_t third_digits(uint32_t bytes) {
    return h2_fma(__byte_perm(bytes, 0x64646464u, SEL), 0x40004000u, 0xe880e880u);  // 2 (1024 + b) - 2304
}

// FP64 panel digits of a pair: w[i] = digit i of both as f16.
__device__ __forceinline__ void panel_digits(uint32_t (&w)[6], double x0, double x1, int e) {
    const uint64_t u = grid_value(x0, e), v = grid_value(x1, e);
#pragma unroll
    for (int i = 0; i < 6; ++i)
        w[i] = f16_digits(((uint32_t)(u >> (10 * (5 - i))) & 0x3ffu) | (((uint32_t)(v >> (10 * (5 - i))) & 0x3ffu) << 16));
}
// FP64 operator digits of a pair, packed: digits 0-3 in words 0-3 (bits 0-9,
// 16-25), digit 4 spread over words 0 and 1, digit 5 over words 2 and 3.
__device__ __forceinline__ void pack_pair(uint32_t (&w)[4], double x0, double x1, int e) {
    const uint64_t u = grid_value(x0, e), v = grid_value(x1, e);
    auto d = [](uint64_t z, int i) { return (uint32_t)(z >> (10 * (5 - i))) & 0x3ffu; };
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int j = 4 + i / 2;  // the spread digit of this word
        const uint32_t pu = i % 2 == 0 ? d(u, j) >> 4 : d(u, j) & 0xfu, pv = i % 2 == 0 ? d(v, j) >> 4 : d(v, j) & 0xfu;
        w[i] = d(u, i) | (pu << 10) | (d(v, i) << 16) | (pv << 26);
    }
}
__device__ __forceinline__ uint32_t packed_digit(const uint32_t (&w)[4], int i) {
    if (i < 4) return f16_digits(w[i] & 0x03ff03ffu);
    return spread_digit(w[2 * (i - 4)], w[2 * (i - 4) + 1]);
}

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2],
                                         const float (&c)[4]) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

// The operator's digits, each scalar row on the grid of its largest element (exponent
// opexp[4 block row + row], within [lo, hi]): one warp per block row; block nnzL is the
// zero block that pads the lists.  A block holds, per scalar row r, the words of its
// pairs (H[r][0], H[r][1]) and (H[r][2], H[r][3]): 16 bytes in FP32, 32 in FP64.
// (Unpacked f16 digits would save the unpacking and take half as much again from
// L2 and, counted in the 128-byte lines that a load touches, from L1.)
template <typename T>
__global__ void k_opdig(const int64_t *rp, const double *v, int64_t nbr, int64_t nnzL, int round_bf16, int lo, int hi,
                        uint4 *opd, int32_t *opexp, int32_t *opflag) {
    constexpr bool F64 = sizeof(T) == 8;
    const int64_t I = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (I == nbr) {
        constexpr int N = F64 ? 8 : 4;
        if (lane < N) opd[nnzL * N + lane] = make_uint4(0x82008200u, 0x02000200u, 0x82008200u, 0x02000200u);
        return;
    }
    if (I > nbr) return;
    const int64_t e0 = rp[I] * BB, e1 = rp[I + 1] * BB;
    uint32_t m = 0;  // of scalar row (lane / 4) % 4, whose elements the lane reads
    for (int64_t i = e0 + lane; i < e1; i += 32) {
        if constexpr (F64) m = max(m, mag_bits(v[i]));
        else m = max(m, mag_bits(round_bf16 ? bf16r((float)v[i]) : (float)v[i]));
    }
#pragma unroll
    for (int o = 1; o < 32; o = o == 2 ? 16 : 2 * o) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    int e;
    if (__any_sync(0xffffffffu, !grid_exp<T>(m, lo, hi, e))) {
        if (lane == 0) atomicOr(opflag, 1);
        return;
    }
    if (lane < 16 && (lane & 3) == 0) opexp[4 * I + (lane >> 2)] = e;
    e = __shfl_sync(0xffffffffu, e, 4 * (lane & 3));
    for (int64_t i = e0 / 4 + lane; i < e1 / 4; i += 32) {  // scalar rows (lane % 4) of the blocks
        const double2 x = make_double2(v[4 * i], v[4 * i + 1]), y = make_double2(v[4 * i + 2], v[4 * i + 3]);
        if constexpr (F64) {
            uint32_t w[4];
            pack_pair(w, x.x, x.y, e);
            opd[2 * i] = make_uint4(w[0], w[1], w[2], w[3]);
            pack_pair(w, y.x, y.y, e);
            opd[2 * i + 1] = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
            // 30 bits of the FP64 element (BF16: of the rounded one)
            const double sc = pow2(29 - e, 0.0);
            auto q = [&](double z) { return __double2int_rn((round_bf16 ? (double)bf16r((float)z) : z) * sc); };
            uint32_t w0[2], w1[2];
            pack_pair(w0, q(x.x), q(x.y));
            pack_pair(w1, q(y.x), q(y.y));
            opd[i] = make_uint4(w0[0], w0[1], w1[0], w1[1]);
        }
    }
}

// A scalar row of an operator block's digits, in one load (an L1 access costs a
// cycle for each line it touches, and a warp's rows lie in 8 blocks)
__device__ __forceinline__ void ld_row(uint32_t (&w)[4], const uint4 *opd, uint32_t blk) {
    const uint4 v = __ldg(opd + (uint64_t)blk * 4);
    w[0] = v.x;
    w[1] = v.y;
    w[2] = v.z;
    w[3] = v.w;
}
__device__ __forceinline__ void ld_row(uint32_t (&w)[8], const uint4 *opd, uint32_t blk) {
    asm("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
        : "l"(opd + (uint64_t)blk * 8));
}

}  // namespace cheb
