// Element-wise Beaver product (Section 2.1 "Multiplication", Eq. 1, one element at a time), e.g. the product
// ReLU(gate) * up of a gated FFN:
//   open   : [d]_i = [x]_i - [a]_i,  [e]_i = [y]_i - [b]_i                       (before the exchange)
//   combine: d = [d]_0 + [d]_1, e = [e]_0 + [e]_1,
//            [z]_i = [c]_i + d*[b]_i + e*[a]_i + i*d*e                           (after it)
// Bound by memory: eight words per element and party (five in, two messages and the result out).  One pass: a thread has
// both parties' words of its elements, which is the exchange, so nobody reads a message back (as two passes, with the
// messages read by both parties, eleven words and a second launch).  16-byte accesses when the word count is even and the
// pointers allow it.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "pdl.cuh"

namespace comet {

typedef unsigned long long u64;

struct MulArgs {
    const u64* x[2]; const u64* y[2];
    const u64* a[2]; const u64* b[2]; const u64* c[2];
    u64* d[2]; u64* e[2];        // the messages
    u64* z[2];
    long long pieces;            // 16-byte pairs, or single words
};

__device__ __forceinline__ ulonglong2 mul_sub(ulonglong2 p, ulonglong2 q) { return make_ulonglong2(p.x - q.x, p.y - q.y); }
__device__ __forceinline__ u64 mul_sub(u64 p, u64 q) { return p - q; }
__device__ __forceinline__ u64 mul_eq1(u64 c, u64 d, u64 e, u64 a, u64 b, int party) {
    return c + d * b + e * a + (party ? d * e : 0ull);
}
__device__ __forceinline__ u64 mul_combine(u64 c, u64 d0, u64 d1, u64 e0, u64 e1, u64 a, u64 b, int party) {
    return mul_eq1(c, d0 + d1, e0 + e1, a, b, party);
}
__device__ __forceinline__ ulonglong2 mul_combine(ulonglong2 c, ulonglong2 d0, ulonglong2 d1, ulonglong2 e0,
                                                  ulonglong2 e1, ulonglong2 a, ulonglong2 b, int party) {
    return make_ulonglong2(mul_eq1(c.x, d0.x + d1.x, e0.x + e1.x, a.x, b.x, party),
                           mul_eq1(c.y, d0.y + d1.y, e0.y + e1.y, a.y, b.y, party));
}

template <typename PIECE>
__global__ void __launch_bounds__(256)
beaver_mul_kernel(const __grid_constant__ MulArgs g) {
    pdl_wait();
    pdl_launch_dependents();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < g.pieces; t += stride) {
        PIECE x[2], y[2], a[2], b[2], c[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            x[p] = __ldcs(reinterpret_cast<const PIECE*>(g.x[p]) + t);
            a[p] = __ldcs(reinterpret_cast<const PIECE*>(g.a[p]) + t);
            y[p] = __ldcs(reinterpret_cast<const PIECE*>(g.y[p]) + t);
            b[p] = __ldcs(reinterpret_cast<const PIECE*>(g.b[p]) + t);
            c[p] = __ldcs(reinterpret_cast<const PIECE*>(g.c[p]) + t);
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            x[p] = mul_sub(x[p], a[p]);                      // [d]_i
            y[p] = mul_sub(y[p], b[p]);                      // [e]_i
            reinterpret_cast<PIECE*>(g.d[p])[t] = x[p];
            reinterpret_cast<PIECE*>(g.e[p])[t] = y[p];
        }
#pragma unroll
        for (int p = 0; p < 2; ++p)
            reinterpret_cast<PIECE*>(g.z[p])[t] = mul_combine(c[p], x[0], x[1], y[0], y[1], a[p], b[p], p);
    }
}

// Truncation by f bits with a dealer's pair (r, r' = floor(r / 2^f), r read as signed).  Not a protocol of the
// paper; it is Section 2.1's "Reconstruction" of m = z - r followed by its "Addition" of the public value
// floor(m / 2^f):
//   open   : [m]_i = [z]_i - [r]_i                                      (before the exchange)
//   combine: m = [m]_0 + [m]_1,  [z]_i <- [r']_i + i * (m >> f, arithmetic)  (after it)
struct TruncPairArgs {
    u64* z[2];                   // in: shares at scale 2f; out: shares at scale f
    const u64* r[2]; const u64* rp[2];
    u64* m[2];                   // the messages
    long long pieces;
    int f;
};

__device__ __forceinline__ u64 trunc_floor(u64 m, int f) { return (u64)((long long)m >> f); }
__device__ __forceinline__ u64 trunc_pair_out(u64 rp, u64 m0, u64 m1, int f, int party) {
    return party ? rp + trunc_floor(m0 + m1, f) : rp;
}
__device__ __forceinline__ ulonglong2 trunc_pair_out(ulonglong2 rp, ulonglong2 m0, ulonglong2 m1, int f, int party) {
    return make_ulonglong2(trunc_pair_out(rp.x, m0.x, m1.x, f, party), trunc_pair_out(rp.y, m0.y, m1.y, f, party));
}

// One pass over both parties, as above.
template <typename PIECE>
__global__ void __launch_bounds__(256)
trunc_pair_kernel(const __grid_constant__ TruncPairArgs g) {
    pdl_wait();
    pdl_launch_dependents();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < g.pieces; t += stride) {
        PIECE m[2], rp[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            rp[p] = __ldcs(reinterpret_cast<const PIECE*>(g.rp[p]) + t);
            m[p] = mul_sub(reinterpret_cast<const PIECE*>(g.z[p])[t], __ldcs(reinterpret_cast<const PIECE*>(g.r[p]) + t));
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            reinterpret_cast<PIECE*>(g.m[p])[t] = m[p];
            reinterpret_cast<PIECE*>(g.z[p])[t] = trunc_pair_out(rp[p], m[0], m[1], g.f, p);
        }
    }
}

// Section 2.1 "Addition": a shared bias [cols] added to every row of a shared matrix, in place; purely local.
// Bound by memory (one word in, one out per element); 16-byte pieces when the column count and the pointers allow it, and
// the position in the row is carried along instead of divided out per element.
struct BiasArgs {
    u64* z[2];
    const u64* bias[2];
    long long total;             // pieces of the whole matrix
    int pieces;                  // pieces per row
    int stride_pieces;           // (gridDim.x * blockDim.x) % pieces
};

__device__ __forceinline__ ulonglong2 mul_add(ulonglong2 p, ulonglong2 q) { return make_ulonglong2(p.x + q.x, p.y + q.y); }
__device__ __forceinline__ u64 mul_add(u64 p, u64 q) { return p + q; }

template <typename PIECE>
__global__ void __launch_bounds__(256)
add_bias_kernel(const __grid_constant__ BiasArgs g) {
    pdl_wait();
    pdl_launch_dependents();
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int piece = (int)(t % g.pieces);
    for (; t < g.total; t += stride) {
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            PIECE* z = reinterpret_cast<PIECE*>(g.z[p]) + t;
            *z = mul_add(*z, __ldca(reinterpret_cast<const PIECE*>(g.bias[p]) + piece));
        }
        piece += g.stride_pieces;
        if (piece >= g.pieces) piece -= g.pieces;
    }
}

}  // namespace comet
