// Residue planes of ring words: the number system of combine_residue_kernel.
//
// A product of ring words needs 36 of the 64 products of their bytes (kernels_limb.cuh).  Through residues it needs 18: write
// x = x_l + 2^56 x_h with x_l the signed low 56 bits and x_h a byte; then mod 2^64
//     x y = x_l y_l + 2^56 (x_h y_l + x_l y_h),
// where the second term needs only the low bytes of x_l and y_l.  The sum of the x_l y_l over the contraction index is an
// integer of less than 2^(110 + log2 depth) and is found from its residues modulo 16 pairwise coprime numbers of at most 256
// (Chinese remainder theorem), each of them a product of signed bytes that a tensor core accumulates exactly in 32 bits.  The
// two cross products are two more.  All 64 bits through residues would take 18 moduli as well, but 18 planes instead of 17 and
// half the depth.
//
// Planes of a word: 0..15 the residues of x_l (plane 0, modulo 256, is its low byte), 16 the byte x_h.  The right operand's
// residues 1..15 are multiplied by the inverse of M / m_i modulo m_i, so that the product's residue is already the factor that
// the Chinese remainder theorem puts before M / m_i.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace comet {

typedef unsigned long long u64;

namespace residue {
constexpr int MODULI = 16, PLANES = 17, JOBS = 18;       // JOBS: byte products per operand pair
constexpr int KC = 64;                                   // contraction depth of a block
constexpr int GROUP_BYTES = 8 * KC;                      // 8 rows of one plane and block, as the tensor cores read them
constexpr int CELL_BYTES = PLANES * GROUP_BYTES;         // all planes of 8 rows and a block
// Twice the depth of a product (two operand pairs) times 2^110 stays below M / 2, M = 2^125.48, with 2^-12 of M to spare for
// the quotient's rounding (residue_recombine_kernel); the byte products then stay below 2^29.
constexpr int MAX_DEPTH = 11424;

__host__ __device__ constexpr int modulus(int i) {
    constexpr int m[MODULI] = {256, 253, 251, 247, 245, 243, 241, 239, 233, 229, 227, 223, 211, 199, 197, 193};
    return m[i];
}
// M / m_i modulo 2^64, and modulo m_i the inverse of it
__host__ __device__ constexpr u64 cofactor(int i) {
    u64 p = 1;
    for (int k = 0; k < MODULI; ++k)
        if (k != i) p *= (u64)modulus(k);
    return p;
}
__host__ __device__ constexpr u64 product() { return cofactor(0) * 256ull; }
__host__ __device__ constexpr int inverse(int i) {
    int p = 1;
    for (int k = 0; k < MODULI; ++k)
        if (k != i) p = p * (modulus(k) % modulus(i)) % modulus(i);
    for (int v = 1; v < modulus(i); ++v)
        if (p * v % modulus(i) == 1) return v;
    return 0;
}
// What byte b of a word (0..6) counts in residue i, as a signed byte.
__host__ __device__ constexpr int weight(int i, int b, bool right) {
    int w = 1;
    for (int k = 0; k < b; ++k) w = w * 256 % modulus(i);
    if (right) w = w * inverse(i) % modulus(i);
    return w > modulus(i) / 2 ? w - modulus(i) : w;
}
__host__ __device__ constexpr unsigned weights(int i, int first, bool right) {       // of four bytes, packed
    unsigned packed = 0;
    for (int b = 0; b < 4 && first + b < 7; ++b) packed |= (unsigned)(weight(i, first + b, right) & 255) << (8 * b);
    return packed;
}
// The reduction works in floats of [2^23, 2^24), whose unit is 1: BASE + t with BASE a multiple of 256 m near 1.5 * 2^23 and
// |t| < 2^18 the weighted sum of the bytes.
__host__ __device__ constexpr int base(int i) { return 12582912 / (256 * modulus(i)) * (256 * modulus(i)); }
// ... as the word that the sum starts from.  Byte 6 is signed: its sign bit is flipped, and 128 of its weight taken off here.
__host__ __device__ constexpr unsigned start(int i, bool right) {
    return 0x4B000000u + (unsigned)(base(i) - 8388608 - 128 * weight(i, 6, right));
}
}  // namespace residue

__device__ __forceinline__ unsigned residue_dot(unsigned bytes, unsigned weights, unsigned acc) {
    unsigned d;
    asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(bytes), "r"(weights), "r"(acc));
    return d;
}

// Residue I of x_l, in the low byte: t - m * round(t / m).  The quotient comes out of one fused multiply-add, as the low bits
// of a float near 1.5 * 2^23; its error before rounding is below 0.004, so the residue fits a signed byte for m <= 253.
template <int I, bool RIGHT>
__device__ __forceinline__ unsigned residue_of(unsigned lo, unsigned hi) {
    constexpr int m = residue::modulus(I), base = residue::base(I);
    constexpr unsigned w_lo = residue::weights(I, 0, RIGHT), w_hi = residue::weights(I, 4, RIGHT), start = residue::start(I, RIGHT);
    const unsigned t = residue_dot(hi, w_hi, residue_dot(lo, w_lo, start));
    const float q = __fmaf_rn(__uint_as_float(t), 1.0f / (float)m, (float)(12582912 - base / m));
    return t - __float_as_uint(q) * (unsigned)m;
}

__device__ __forceinline__ unsigned residue_pack(unsigned a, unsigned b, unsigned c, unsigned d) {
    return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

template <bool RIGHT, int I>
__device__ __forceinline__ void residue_emit_from(uint8_t* dst, const unsigned* lo, const unsigned* hi) {
    if constexpr (I < residue::MODULI) {
        *reinterpret_cast<unsigned*>(dst + I * residue::GROUP_BYTES) =
            residue_pack(residue_of<I, RIGHT>(lo[0], hi[0]), residue_of<I, RIGHT>(lo[1], hi[1]), residue_of<I, RIGHT>(lo[2], hi[2]),
                         residue_of<I, RIGHT>(lo[3], hi[3]));
        residue_emit_from<RIGHT, I + 1>(dst, lo, hi);
    }
}

// Four words of one row -> 17 planes, four bytes each, GROUP_BYTES apart.
template <bool RIGHT>
__device__ __forceinline__ void residue_emit4(uint8_t* dst, const u64* w) {
    unsigned lo[4], hi[4], top[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        lo[e] = (unsigned)w[e];
        hi[e] = (unsigned)(w[e] >> 32) ^ 0x00800000u;            // byte 6 without its sign
        top[e] = (unsigned)(w[e] >> 32) + 0x00800000u;           // x_h = (x + 2^55) / 2^56, in byte 3
    }
    *reinterpret_cast<unsigned*>(dst) = residue_pack(lo[0], lo[1], lo[2], lo[3]);
    *reinterpret_cast<unsigned*>(dst + residue::MODULI * residue::GROUP_BYTES) =
        __byte_perm(__byte_perm(top[0], top[1], 0x0073), __byte_perm(top[2], top[3], 0x0073), 0x5410);
    residue_emit_from<RIGHT, 1>(dst, lo, hi);
}

}  // namespace comet
