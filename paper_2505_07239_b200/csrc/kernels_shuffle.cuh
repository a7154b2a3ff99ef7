// Oblivious shuffle, online stage (Section 4.2, Protocol 1): a row gather through a
// party's sub-permutation plus or minus a one-time mask,
//   mask step  : [y]_i = tau_i([x]_i) + a_i
//   finish step: [z]_i = rho_i([y]_other) - b_i
// with (p(x))[j] = x[p[j]] acting on the rows of a [rows, cols] matrix of ring
// words.  Pure HBM work: 16-byte accesses, consecutive threads on consecutive
// pieces of a row; blockIdx.y is the party.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "pdl.cuh"

namespace comet {

typedef unsigned long long u64;

struct ShuffleArgs {
    const u64* in[2];          // source matrix read by party 0 / party 1 (already swapped for the finish step)
    const int32_t* perm[2];    // the party's sub-permutation, `rows` entries
    const u64* mask[2];        // a_i or b_i, [rows, cols]
    u64* out[2];
    long long rows;
    int pieces;                // pieces per row: cols / 2 (16-byte pieces) or cols (8-byte pieces)
    int subtract;              // 0: out = gathered + mask, 1: out = gathered - mask
    long long stride_rows;     // (gridDim.x * blockDim.x) / pieces
    int stride_pieces;         // (gridDim.x * blockDim.x) % pieces
    int* bad_index;            // optional: set to 1 when a permutation entry is outside [0, rows)
};

// PIECE = ulonglong2 (even cols, 16-byte aligned pointers) or u64.
template <typename PIECE>
__device__ __forceinline__ PIECE shuffle_combine(PIECE g, PIECE m, int subtract);
template <>
__device__ __forceinline__ ulonglong2 shuffle_combine<ulonglong2>(ulonglong2 g, ulonglong2 m, int subtract) {
    return subtract ? make_ulonglong2(g.x - m.x, g.y - m.y) : make_ulonglong2(g.x + m.x, g.y + m.y);
}
template <>
__device__ __forceinline__ u64 shuffle_combine<u64>(u64 g, u64 m, int subtract) {
    return subtract ? g - m : g + m;
}
template <typename PIECE>
__device__ __forceinline__ PIECE shuffle_zero();
template <>
__device__ __forceinline__ ulonglong2 shuffle_zero<ulonglong2>() { return make_ulonglong2(0ull, 0ull); }
template <>
__device__ __forceinline__ u64 shuffle_zero<u64>() { return 0ull; }

template <typename PIECE>
__global__ void __launch_bounds__(256)
shuffle_rows_kernel(ShuffleArgs a) {
    pdl_wait();
    pdl_launch_dependents();
    const int party = blockIdx.y;
    const PIECE* __restrict__ in = reinterpret_cast<const PIECE*>(party ? a.in[1] : a.in[0]);
    const PIECE* __restrict__ mask = reinterpret_cast<const PIECE*>(party ? a.mask[1] : a.mask[0]);
    const int32_t* __restrict__ perm = party ? a.perm[1] : a.perm[0];
    PIECE* __restrict__ out = reinterpret_cast<PIECE*>(party ? a.out[1] : a.out[0]);
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long row = first / a.pieces;
    int piece = (int)(first - row * a.pieces);
    while (row < a.rows) {
        const long long src = perm[row];
        const long long at = row * a.pieces + piece;
        PIECE g;
        if (src >= 0 && src < a.rows) {
            g = __ldca(in + src * a.pieces + piece);
        } else {
            g = shuffle_zero<PIECE>();              // never read out of bounds; the caller sees the flag
            if (a.bad_index) *a.bad_index = 1;
        }
        out[at] = shuffle_combine<PIECE>(g, __ldca(mask + at), a.subtract);
        row += a.stride_rows;
        piece += a.stride_pieces;
        if (piece >= a.pieces) { piece -= a.pieces; ++row; }
    }
}

// Both steps in one pass: [y]_i = tau_i([x]_i) + a_i is written as the message, and [z]_i = rho_i([y]_other) - b_i takes its
// rows of the other party's message from the words they are made of instead of waiting for them: row j of z_i is
// x_other[tau_other[r]] + a_other[r] - b_i[j] with r = rho_i[j].  Five words per element and party cross HBM, as the protocol
// has it, as long as X and a stay in L2 for their second use; see shuffle_in_one_pass in comet_api.cu.
struct ShuffleBothArgs {
    const u64* x[2];
    const int32_t* tau[2];
    const int32_t* rho[2];
    const u64* a[2];
    const u64* b[2];
    u64* y[2];
    u64* z[2];
    long long rows;
    int pieces;
    long long stride_rows;
    int stride_pieces;
    int* bad_index;
};

template <typename PIECE>
__global__ void __launch_bounds__(256)
shuffle_both_kernel(const __grid_constant__ ShuffleBothArgs g) {
    pdl_wait();
    pdl_launch_dependents();
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long row = first / g.pieces;
    int piece = (int)(first - row * g.pieces);
    while (row < g.rows) {
        const long long at = row * g.pieces + piece;
        // A permutation entry out of range is never followed: the row it would have fetched counts as zero.  (Row 0 is read in
        // its place, so that every load of a piece is in flight before the first is needed.)
        long long src[2], r[2], far[2];
        bool src_ok[2], r_ok[2], far_ok[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            src[p] = g.tau[p][row];
            r[p] = g.rho[p][row];
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            src_ok[p] = src[p] >= 0 && src[p] < g.rows;
            r_ok[p] = r[p] >= 0 && r[p] < g.rows;
            if (!src_ok[p]) src[p] = 0;
            if (!r_ok[p]) r[p] = 0;
            far[p] = g.tau[p ^ 1][r[p]];
            far_ok[p] = r_ok[p] && far[p] >= 0 && far[p] < g.rows;
            if (!far_ok[p]) far[p] = 0;
            if ((!src_ok[p] || !r_ok[p]) && g.bad_index) *g.bad_index = 1;
        }
        PIECE xv[2], av[2], bv[2], xo[2], ao[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            xv[p] = __ldca(reinterpret_cast<const PIECE*>(g.x[p]) + src[p] * g.pieces + piece);
            av[p] = __ldca(reinterpret_cast<const PIECE*>(g.a[p]) + at);
            bv[p] = __ldcs(reinterpret_cast<const PIECE*>(g.b[p]) + at);
            xo[p] = __ldca(reinterpret_cast<const PIECE*>(g.x[p ^ 1]) + far[p] * g.pieces + piece);
            ao[p] = __ldca(reinterpret_cast<const PIECE*>(g.a[p ^ 1]) + r[p] * g.pieces + piece);
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            if (!src_ok[p]) xv[p] = shuffle_zero<PIECE>();
            if (!far_ok[p]) xo[p] = shuffle_zero<PIECE>();
            if (!r_ok[p]) ao[p] = shuffle_zero<PIECE>();
            reinterpret_cast<PIECE*>(g.y[p])[at] = shuffle_combine<PIECE>(xv[p], av[p], 0);
            reinterpret_cast<PIECE*>(g.z[p])[at] = shuffle_combine<PIECE>(shuffle_combine<PIECE>(xo[p], ao[p], 0), bv[p], 1);
        }
        row += g.stride_rows;
        piece += g.stride_pieces;
        if (piece >= g.pieces) { piece -= g.pieces; ++row; }
    }
}

// inverse[perm[j]] = j: what a party does locally to obtain the sub-permutations of the unshuffle.
__global__ void __launch_bounds__(256)
invert_permutation_kernel(const int32_t* perm, int32_t* inverse, long long rows,
                          int* bad_index) {
    pdl_wait();
    pdl_launch_dependents();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < rows; j += stride) {
        const long long p = perm[j];
        if (p >= 0 && p < rows) inverse[p] = (int32_t)j;
        else if (bad_index) *bad_index = 1;
    }
}

}  // namespace comet
