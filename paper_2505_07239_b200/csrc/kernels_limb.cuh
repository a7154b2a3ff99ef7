// K4, tensor-core variant: the gathered ring matmul + Beaver combine
//   Z_i = C_i + E*B_i + A_i*F + i*E*F = C_i + E*B_i + V_i*F,   V_i = A_i + i*E   (Eq. 1, party i)
// on the int8 tensor cores of sm_100a (tcgen05.mma kind::i8, accumulators in TMEM).
//
// A 64-bit ring word is eight unsigned 8-bit limbs, x = sum_p x_p 2^(8p).  Mod 2^64 only limb pairs with
// p + q <= 7 matter: x*y = sum_{s=0..7} 2^(8s) D_s, D_s = sum_{p+q=s} x_p y_q (36 of the 64 limb products).
// Each D_s summed over the contraction index is one 32-bit accumulator per output element: 8 accumulators
// of 128 x 64 fill the 512 TMEM columns of an SM exactly.  Only D_s mod 2^(64-8s) is needed, so 32-bit
// wrap-around is harmless for s >= 4, and for s <= 3 the exact sum (s+1)*K*255^2 stays below 2^32 while a
// segment accumulates at most 16384 contraction elements.
//
// Operands are kept as "blocked limb planes": for a tile of R rows (128 left, 64 right) and a block of 32
// contraction elements, 8 planes of R x 32 bytes, each stored as the tensor core's K-major no-swizzle
// canonical layout (8-row x 16-byte core matrices; the two 16-byte K halves of a row group adjacent).  One
// block is one contiguous bulk copy into shared memory.  With the planes of the right operand stacked
// along N, limb plane p of the left operand meets planes 0..7-p of the right operand in ONE instruction
// whose N spans accumulators D_p..D_7 (split in two when N > 256): 12 instructions per 32-deep step.
//
// Work is split stream-K style over a persistent grid: the (party, tile, k-block) space is cut into equal
// contiguous ranges, or every tile into parts of its own (LimbArgs::parts), every segment's partial sums are added to Z by 64-bit integer reductions of the copy
// engine -- exact and order-independent in the ring -- and Z is pre-loaded with C_i.
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "pdl.cuh"
#include "residue_planes.cuh"

namespace comet {

namespace limb {
constexpr int BM = 128, BN = 64, KC = 32, PLANES = 8;
constexpr int A_BLOCK_BYTES = PLANES * BM * KC;   // 32 KiB
constexpr int B_BLOCK_BYTES = PLANES * BN * KC;   // 16 KiB
constexpr int STAGES = 3;
constexpr int MAX_SEGMENT_UNITS = 16384 / KC;     // keeps the limb sums for s <= 3 below 2^32
constexpr int EPI_WARPS = 8;                      // warp w drains TMEM lanes 32*(w%4).., columns 32*(w/4)..
constexpr int THREADS = 32 * (EPI_WARPS + 2);     // warps 0-7 epilogue, warp 8 copy producer, warp 9 MMA issuer
constexpr int EX_THREADS = 128, EX_ROWS = 16, EX_MAX_KB_PER_CTA = 16;      // exchange kernel: four rows per warp
constexpr int EX_STAGES = 2, EX_STAGE_BYTES = EX_THREADS * 8 * 16;           // eight 16-byte pieces per lane and k-block
constexpr size_t EX_SMEM_BYTES = (size_t)EX_STAGES * EX_STAGE_BYTES;        // 32 KiB at most: fits beside a tensor-core CTA
constexpr int OUT_COLS = 16;                      // words per staged output row (a thread's 32 go in two rounds)
constexpr int OUT_ROW_BYTES = OUT_COLS * 8 + 16;  // padded against bank conflicts (grouped kernel: one copy per row)
constexpr int OUT_TILE_BYTES = 32 * OUT_COLS * 8; // swizzled instead (one tensor copy per warp and round), 1 KiB aligned
constexpr size_t SMEM_BYTES = (size_t)STAGES * (A_BLOCK_BYTES + B_BLOCK_BYTES) + (size_t)EPI_WARPS * 32 * OUT_ROW_BYTES + 1024;
constexpr long long WAIT_CYCLES = 4000000000ll;   // ~2 s at 1.9 GHz: every wait gives up after this
constexpr unsigned LBO_BYTES = 128, SBO_BYTES = 256;
}  // namespace limb

// ---------------------------------------------------------------------------
// Blocked limb planes from words: 4 x 4 byte transposition, and four words of one row -> eight planes, four bytes each,
// `stride` bytes apart.
//
// Inside a 32-deep k-block the contraction indices sit in the order in which a warp reads words: a lane holds two 16-byte
// pieces of a row, words 2c, 2c+1, 16+2c, 17+2c (c = lane mod 8, so eight lanes read whole 128-byte lines), and writes
// their bytes next to each other, at bytes 4c .. 4c+3 of the row's 32.  Every operand uses that order, so sums over a
// k-block are the same.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void limb_transpose4(unsigned x0, unsigned x1, unsigned x2, unsigned x3,
                                                unsigned& p0, unsigned& p1, unsigned& p2, unsigned& p3) {
    const unsigned t0 = __byte_perm(x0, x1, 0x5140), t1 = __byte_perm(x2, x3, 0x5140);
    const unsigned t2 = __byte_perm(x0, x1, 0x7362), t3 = __byte_perm(x2, x3, 0x7362);
    p0 = __byte_perm(t0, t1, 0x5410);
    p1 = __byte_perm(t0, t1, 0x7632);
    p2 = __byte_perm(t2, t3, 0x5410);
    p3 = __byte_perm(t2, t3, 0x7632);
}

__device__ __forceinline__ void limb_emit4(uint8_t* dst, int stride, const u64* w) {
    uint32_t p[8];
    limb_transpose4((uint32_t)w[0], (uint32_t)w[1], (uint32_t)w[2], (uint32_t)w[3], p[0], p[1], p[2], p[3]);
    limb_transpose4((uint32_t)(w[0] >> 32), (uint32_t)(w[1] >> 32), (uint32_t)(w[2] >> 32), (uint32_t)(w[3] >> 32),
                    p[4], p[5], p[6], p[7]);
#pragma unroll
    for (int i = 0; i < 8; ++i) *reinterpret_cast<uint32_t*>(dst + i * stride) = p[i];
}

// 16-byte asynchronous copy global -> shared that bypasses L1; with `bytes` = 0 nothing is read and the 16 bytes are
// filled with zeros.
__device__ __forceinline__ void limb_copy16_async(uint32_t dst_smem, const void* src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst_smem), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void limb_copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void limb_copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }

// ---------------------------------------------------------------------------
// Masking and exchange for the tensor-core kernel, one launch (Section 2.1 "Multiplication"; IndexCols of Protocol 2,
// IndexRow of Protocol 3):
//   left  rows: E_i = X_i - A_i        -> message;  planes of E = E_0 + E_1 and of V_i = A_i + i*E
//   right rows: F_i = gather(W_i) - B_i -> message;  planes of F = F_0 + F_1 and of B_i
//   copy      : Z_i <- C_i (the accumulation target starts from the triple's C share)
// gather: up   (down = 0): row c of the right operand is row neuron(c) of W (whole rows of `ldw` words);
//         down (down = 1): contraction index c is column neuron(c) of W (strips of `bs` words in every row).
// What is written for a party depends on that party's shares and on the two messages; both parties' words of one place
// are in the same thread, which is the exchange, so a message is written once and read by nobody on the path, and the
// planes of E and F exist once for both parties.
//
// Bound by memory: per word and party 16 bytes in, 8 out as the message, 12 out as planes (the sum's planes are shared).
// A warp owns four rows and walks k-blocks of 32 words.  A lane's 16-byte pieces land in shared memory by asynchronous
// copies, EX_STAGES k-blocks ahead, and only that lane reads them: no barriers, and loads in flight cost neither registers
// nor L1 lines.  (Plain loads, eight per lane in flight: 48 us on [512 | 832, 2048] and 329 us on [512 | 8192, 2048] with the
// L1 that the tensor-core kernels' carve-out leaves, 37 and 271 us with all of it; 33 and 258 us this way.)
// It replaces an opening kernel and a preparation kernel that read the messages back and built every plane of E and F
// twice: 112 bytes per word of both parties, now 72.
// With RESIDUE the planes are those of combine_residue_kernel: 17 instead of 8, 99 bytes per word of both parties; [512 | 832,
// 2048] 45 us in the step, [512 | 8192, 2048] 281, 5.9 TB/s (about 1000 instructions a warp and k-block, a third of its time).
// grid = left_blocks + right_blocks + copy_blocks; a left / right block owns 16 rows x kb_per_cta k-blocks.
// ---------------------------------------------------------------------------
struct LimbExchangeArgs {
    const u64* X[2]; const u64* A[2];
    u64* E[2];
    uint8_t* Epl;
    uint8_t* Vpl[2];
    const u64* W0[2];        // weights of group 0 (gate when gated, else the only matrix)
    const u64* W1[2];        // weights of group 1 (up-projection of a gated FFN)
    const u64* W2[2];        // weights of group 2 (third stacked matrix, e.g. the value projection)
    const u64* B[2];
    u64* F[2];
    uint8_t* Fpl;
    uint8_t* Bpl[2];
    const u64* C[2];
    u64* Z[2];
    long long copy_pairs;
    const int32_t* ids;      // ascending active block ids, or null: they are in the launch's BlockIds
    int n, bs;               // active neurons, neurons per block
    int M, N, K;             // rows of the left and right operand, contraction length
    int ldw, down;
    int left_blocks, right_blocks, copy_blocks;
    int kblocks, kb_per_cta, kchunks;      // kchunks = ceil(kblocks / kb_per_cta)
    // Protocol 3 with per-column row sets: per-token mask over the active blocks, [M, tmask_ld] bytes, or null.  Where
    // it is zero X and A_i have no entry: E_i is zero there and the party's A_i counts as zero.
    const uint8_t* tmask;
    int tmask_ld;
    // Protocol 2 over connected components: component label per row of X and per active block (-1 = in no
    // component), or null.  A row / column outside every component is not opened: its message words are zero.
    // Protocol 3 (down) uses blk_label alone: a block no token uses holds no non-zero column of X, and the rows of
    // the right operand that belong to it are not opened either.
    const int32_t* row_label;
    const int32_t* blk_label;
    // One multiplication per component: the planes are written in component order while the messages keep the compact
    // order.  Plane row r of the left operand is row row_map[r]; of the right operand (up) compact row
    // col_map[r / bs] * bs + r % bs; contraction index k (down) is compact index kmap[k / bs] * bs + k % bs.
    // Null: identity.
    const int32_t* row_map;
    const int32_t* col_map;
    const int32_t* kmap;
};

// The ascending active block ids of a mask that the host held: they travel in the parameter block of every kernel that gathers
// (2 KiB), which takes the compaction launch (a few us of host time, one hop of the chain) off the step.  Longer masks and
// masks in device memory are compacted by a kernel, and `ids` of the arguments points to its result.
struct BlockIds {
    static constexpr int CAPACITY = 1024;
    uint16_t id[CAPACITY];
};
__device__ __forceinline__ int block_id(const int32_t* ids, const BlockIds& held, int blk) {
    return ids ? __ldg(ids + blk) : (int)held.id[blk];
}

// The list written out, for a caller who reads it: from the parameter block too, so that the call can be captured.
__global__ void __launch_bounds__(BlockIds::CAPACITY)
held_ids_kernel(const __grid_constant__ BlockIds held, int count, int32_t* __restrict__ out) {
    pdl_wait();
    pdl_launch_dependents();
    if ((int)threadIdx.x < count) out[threadIdx.x] = held.id[threadIdx.x];
}

template <bool LEFT, bool RESIDUE>
__device__ __forceinline__ void limb_exchange_rows(const LimbExchangeArgs& a, const BlockIds& held, int block, uint8_t* smem) {
    using namespace limb;
    constexpr int TILE = LEFT ? BM : BN, BLOCK_BYTES = PLANES * TILE * KC;
    const int c = threadIdx.x & 7;
    const int r = (block / a.kchunks) * EX_ROWS + (threadIdx.x >> 3);                         // plane row
    const int kb0 = (block % a.kchunks) * a.kb_per_cta, kb1 = min(kb0 + a.kb_per_cta, a.kblocks);
    if (r >= (LEFT ? a.M : a.N)) return;         // planes of rows past the operand are never looked at
    int at = r;                                  // compact row: where it lies in the operands and in the message
    bool closed = false;                         // the row is not part of the message
    const u64* src[2];                           // the row of X_i / the gathered row of W_i
    if (LEFT) {
        if (a.row_map) at = __ldg(a.row_map + r);
        closed = a.row_label && __ldg(a.row_label + at) < 0;
        src[0] = a.X[0] + (size_t)at * a.K;
        src[1] = a.X[1] + (size_t)at * a.K;
    } else {
        if (a.col_map) {
            const int sb = r / a.bs;
            at = __ldg(a.col_map + sb) * a.bs + (r - sb * a.bs);
        }
        if (a.down) {
            src[0] = a.W0[0] + (size_t)at * a.ldw;
            src[1] = a.W0[1] + (size_t)at * a.ldw;
        } else {
            const int grp = (at >= a.n) + (at >= 2 * a.n), j = at - grp * a.n, blk = j / a.bs;
            const size_t off = (size_t)(block_id(a.ids, held, blk) * a.bs + (j - blk * a.bs)) * a.ldw;
            closed = a.blk_label && __ldg(a.blk_label + blk) < 0;
            src[0] = (grp == 0 ? a.W0[0] : grp == 1 ? a.W1[0] : a.W2[0]) + off;
            src[1] = (grp == 0 ? a.W0[1] : grp == 1 ? a.W1[1] : a.W2[1]) + off;
        }
    }
    const u64* own[2];                           // the row of A_i / B_i
    u64* msg[2];                                 // the row of E_i / F_i
    uint8_t* pl[3];                              // this lane's cell in the planes of V_0 / B_0, V_1 / B_1, E / F
    // (residue planes: blocks of 64, all rows of a block together; see ResidueMaps)
    const size_t next_block = (size_t)(((LEFT ? a.M : a.N) + 7) / 8) * residue::CELL_BYTES;
    const size_t cell = (RESIDUE ? (size_t)(kb0 >> 1) * next_block + (size_t)(r >> 3) * residue::CELL_BYTES + (kb0 & 1) * 256
                                 : ((size_t)(r / TILE) * a.kblocks + kb0) * BLOCK_BYTES + (size_t)(r % TILE >> 3) * 256) +
                        (size_t)((c >> 2) * 128 + (r & 7) * 16 + (c & 3) * 4);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        own[p] = (LEFT ? a.A[p] : a.B[p]) + (size_t)at * a.K;
        msg[p] = (LEFT ? a.E[p] : a.F[p]) + (size_t)at * a.K;
        pl[p] = (LEFT ? a.Vpl[p] : a.Bpl[p]) + cell;
    }
    pl[2] = (LEFT ? a.Epl : a.Fpl) + cell;

    // This lane's piece h of k-block kb: compact index of its first word, its column in W, and whether it exists and is part
    // of the message.  Sixteen indices aligned to 16 lie in one block.
    struct Piece { int ks, col; bool in, open; };
    auto piece = [&](int kb, int h) {
        Piece q;
        const int k = kb * KC + 16 * h;
        q.ks = q.col = k + 2 * c;
        q.in = q.ks < a.K;
        q.open = q.in && !closed;
        if (a.down && q.in) {
            int blk = k / a.bs;
            const int within = k - blk * a.bs + 2 * c;
            if (a.kmap) blk = __ldg(a.kmap + blk);
            q.ks = q.col = blk * a.bs + within;
            if (!LEFT) {
                q.col = block_id(a.ids, held, blk) * a.bs + within;
                if (a.blk_label && __ldg(a.blk_label + blk) < 0) q.open = false;
            } else if (a.tmask && a.tmask[(size_t)at * a.tmask_ld + blk] == 0) {
                q.open = q.in = false;           // an entry off the support is none of the triple either
            }
        }
        return q;
    };
    const uint32_t mine = (uint32_t)__cvta_generic_to_shared(smem) + threadIdx.x * 16;
    auto issue = [&](int kb) {
        const uint32_t stage = mine + (uint32_t)((kb - kb0) % EX_STAGES) * EX_STAGE_BYTES;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const Piece q = piece(kb, h);
            const uint32_t bytes = q.in ? 16u : 0u;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                limb_copy16_async(stage + (uint32_t)(4 * h + 2 * p) * (16 * EX_THREADS), q.in ? src[p] + q.col : own[p], bytes);
                limb_copy16_async(stage + (uint32_t)(4 * h + 2 * p + 1) * (16 * EX_THREADS), q.in ? own[p] + q.ks : own[p], bytes);
            }
        }
    };
#pragma unroll
    for (int s = 0; s < EX_STAGES - 1; ++s) {
        if (kb0 + s < kb1) issue(kb0 + s);
        limb_copy_commit();
    }
    for (int kb = kb0; kb < kb1; ++kb) {
        if (kb + EX_STAGES - 1 < kb1) issue(kb + EX_STAGES - 1);
        limb_copy_commit();
        limb_copy_wait<EX_STAGES - 1>();
        const uint8_t* stage = smem + (size_t)((kb - kb0) % EX_STAGES) * EX_STAGE_BYTES + threadIdx.x * 16;
        u64 f[2][4], b[2][4];                    // X_i / W_i, then the message; A_i / B_i
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const Piece q = piece(kb, h);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(stage + (4 * h + 2 * p) * (16 * EX_THREADS));
                const ulonglong2 m = *reinterpret_cast<const ulonglong2*>(stage + (4 * h + 2 * p + 1) * (16 * EX_THREADS));
                b[p][2 * h] = m.x;
                b[p][2 * h + 1] = m.y;
                f[p][2 * h] = q.open ? x.x - m.x : 0ull;
                f[p][2 * h + 1] = q.open ? x.y - m.y : 0ull;
                if (kb * KC + 16 * h + 2 * c < a.K)
                    *reinterpret_cast<ulonglong2*>(msg[p] + q.ks) = make_ulonglong2(f[p][2 * h], f[p][2 * h + 1]);
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            f[0][e] += f[1][e];                  // the exchange
            if (LEFT) b[1][e] += f[0][e];        // V_1 = A_1 + E  (V_0 = A_0)
        }
        if (RESIDUE) {
            residue_emit4<!LEFT>(pl[0], b[0]);
            residue_emit4<!LEFT>(pl[1], b[1]);
            residue_emit4<!LEFT>(pl[2], f[0]);
        } else {
            limb_emit4(pl[0], TILE * KC, b[0]);
            limb_emit4(pl[1], TILE * KC, b[1]);
            limb_emit4(pl[2], TILE * KC, f[0]);
        }
        const size_t step = !RESIDUE ? BLOCK_BYTES : (kb & 1) ? next_block - 256 : 256;
#pragma unroll
        for (int i = 0; i < 3; ++i) pl[i] += step;
    }
    limb_copy_wait<0>();
}

template <bool RESIDUE>
__device__ __forceinline__ void limb_exchange_block(const LimbExchangeArgs& a, const BlockIds& held, int block, uint8_t* smem) {
    if (block < a.left_blocks) return limb_exchange_rows<true, RESIDUE>(a, held, block, smem);
    block -= a.left_blocks;
    if (block < a.right_blocks) return limb_exchange_rows<false, RESIDUE>(a, held, block, smem);
    block -= a.right_blocks;
    const int party = block & 1;
    const ulonglong2* __restrict__ s = reinterpret_cast<const ulonglong2*>(party ? a.C[1] : a.C[0]);
    ulonglong2* __restrict__ d = reinterpret_cast<ulonglong2*>(party ? a.Z[1] : a.Z[0]);
    const long long stride = (long long)(a.copy_blocks >> 1) * limb::EX_THREADS;
    for (long long t = (long long)(block >> 1) * limb::EX_THREADS + threadIdx.x; t < a.copy_pairs; t += stride) {
        if (a.col_map) {                         // entries outside the components stay zero (see LimbArgs)
            const unsigned row = (unsigned)(t / (unsigned)(a.N / 2)), blk = ((unsigned)t - row * (a.N / 2)) * 2 % a.n / a.bs;
            if (__ldg(a.row_label + row) != __ldg(a.blk_label + blk) || __ldg(a.blk_label + blk) < 0) {
                d[t] = make_ulonglong2(0ull, 0ull);
                continue;
            }
        }
        d[t] = __ldcs(s + t);
    }
}

// The first `first_blocks` CTAs work on `a`, the others on `b` (another product's operands).
template <bool RESIDUE>
__global__ void __launch_bounds__(limb::EX_THREADS, 7)
limb_exchange_kernel(const __grid_constant__ LimbExchangeArgs a, const __grid_constant__ LimbExchangeArgs b, int first_blocks,
                     const __grid_constant__ BlockIds held) {
    extern __shared__ __align__(16) uint8_t ex_smem[];
    pdl_wait();
    pdl_launch_dependents();
    const int block = blockIdx.x;
    if (block < first_blocks) limb_exchange_block<RESIDUE>(a, held, block, ex_smem);
    else limb_exchange_block<RESIDUE>(b, held, block - first_blocks, ex_smem);
}

// ---------------------------------------------------------------------------
// PTX wrappers (sm_100a)
// ---------------------------------------------------------------------------
namespace ptx {
// One lane of a converged warp, the same one every time.  Single-thread instructions (copies of the copy engine, MMAs, commits)
// stand under this and not under `lane == 0`: the compiler then knows that one thread runs them, and makes no loop over the
// lanes of each: an issuer at `lane == 0` takes some 100 cycles an MMA, whatever its size.  (In the kernel of this file, whose MMAs
// take about that long themselves, it makes no difference that shows: QKV of 203 tokens, 512 tokens in four groups and 128 tokens
// x 320 within 1 % of what they were, less than two runs of one side differ.)
__device__ __forceinline__ bool elect_one() {
    uint32_t elected;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(elected));
    return elected != 0;
}
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void bulk_s2g(void* dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
// shared -> global bulk reduction: 64-bit integer add of `bytes` (multiple of 16) contiguous bytes
__device__ __forceinline__ void bulk_reduce_add_u64(void* dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.u64 [%0], [%1], %2;"
                 ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
// shared -> global tensor reduction: add a box of 64-bit integers at (column x, row y) of the map's matrix; what lies outside
// the matrix is left out
__device__ __forceinline__ void tensor_reduce_add(const CUtensorMap* map, uint32_t src, int x, int y) {
    asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_group_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_group0() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// D[tmem] (+)= A[smem desc] * B[smem desc], u8 x u8 -> s32.  The descriptors are passed as (low, high) words: only
// the low word (the shared-memory address field) changes between instructions.
#define COMET_MMA_I8(NAME, QUAL)                                                                                   \
    __device__ __forceinline__ void NAME(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,            \
                                         uint32_t b_hi, uint32_t idesc, uint32_t acc) {                           \
        asm volatile(                                                                                              \
            "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"                                                           \
            "setp.ne.b32 p, %6, 0;\n\t"                                                                            \
            "mov.b64 da, {%1, %2};\n\t"                                                                            \
            "mov.b64 db, {%3, %4};\n\t"                                                                            \
            "tcgen05.mma.cta_group::1.kind::i8" QUAL " [%0], da, db, %5, p;\n\t}"                                  \
            ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc) : "memory");          \
    }
COMET_MMA_I8(mma_i8, "")                               // A operand fetched for this instruction only
COMET_MMA_I8(mma_i8_keep_a, ".collector::a::fill")     // A operand kept in the collector for the next instruction
COMET_MMA_I8(mma_i8_reuse_a, ".collector::a::lastuse") // A operand taken from the collector, then dropped
#undef COMET_MMA_I8
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* d) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* d) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
}  // namespace ptx

// ---------------------------------------------------------------------------
// What a per-token mask S [T, nab] (non-zero byte = token t uses active block b) implies, in one launch of one CTA.
//
// 1. The first step of Protocol 2: the connected components of the bipartite graph (token rows) x (active
//    blocks) with the non-zero bytes as edges.  The paper uses depth-first search; here S becomes a bit matrix,
//    every row joins the blocks it uses in a union-find forest over the blocks (hooking by compare-and-swap, the
//    larger root under the smaller), and one pass afterwards reads the roots.  A node's label is the smallest token
//    index of its component; nodes without an edge get -1.
//
// 2. (plan != 0) Protocols 2 and 3 ask for one multiplication per component / per non-zero column entry, over the
//    rows and columns that take part only (the multiplication counts of Theorems 1 and 2).  On the tensor cores
//    this becomes ONE launch over component-sorted operands: token rows and active blocks are ordered by
//    component label (ties by index), so every component is a contiguous rectangle, and
//      up   (Protocol 2): an output tile has work only if the label ranges of its rows and of its columns
//                         intersect; per row tile these column tiles form an interval;
//      down (Protocol 3): a row tile's contraction runs only over the blocks of the components its rows belong
//                         to, an interval of k-blocks in the sorted order of the contraction index.
//    row_map [T]           sorted row position -> token row; rows of no component come last
//    col_map [groups*nab]  sorted block position -> compact block (group * nab + active block) of the
//                          up-projection's columns; inside a component the order is (group, block); blocks of no
//                          component last
//    kmap    [nab]         sorted block position -> active block, for the down-projection's contraction index
//    up, dn  [row tiles]   the work of every tile of 128 sorted rows (LimbGroupRow); needs at most 32768 tokens
//
// report (mapped host memory): [0] edges, [1] components, [2] rows with an edge, [3] blocks with an edge,
// [4] k-block units of the up-projection per party, [5] sum over components of rows x blocks, [6] units of the
// down-projection per party ([4] and [6] only with plan).  Every word carries the launch's ticket above its value, so that the
// host sees by itself which have arrived and no fence over the bus (2 us) orders them.
//
// What bounds it: the host waits for the report, so it is a chain of latencies in one CTA: reading S, the joins, the sort, the
// report.  Rows are sorted by counting, per 32 rows and component.  Comparing every row with every other and spreading minimum
// labels until nothing changed took 26 us of 512 tokens x 26 blocks in four groups, this 14 us.
//
// Working storage (token_plan_words): in dynamic shared memory when `in_smem`, else in `scratch` (global).
// ---------------------------------------------------------------------------
struct LimbGroupRow {
    int unit0;       // units (k-blocks, both operand pairs) of the row tiles before this one, per party
    int tn0, ntn;    // interval of column tiles with work
    int klo, kcnt;   // interval of k-blocks with work; a tile runs over 2 * kcnt units
};

constexpr int PLAN_WORDS = 7, PLAN_VALUE_BITS = 40;          // of the report

struct TokenPlanArgs {
    const uint8_t* S;            // [T, nab]
    uint8_t* copy;               // where S is kept, or null: it is the kept one
    int T, nab, wpr;             // wpr = ceil(nab / 32)
    int32_t* row_label;          // out [T]
    int32_t* blk_label;          // out [nab]
    unsigned long long* report;
    unsigned long long ticket;
    int in_smem;
    uint32_t* scratch;
    int plan, groups, bs, kb_up, nt_dn;
    int32_t* row_map;
    int32_t* col_map;
    int32_t* kmap;
    LimbGroupRow* up;
    LimbGroupRow* dn;
};

// Words of working storage: bit matrix; rows per 32 rows and component; components of the rows; and per block the forest, the
// smallest row, the rows and their first position, the label, and the sorted labels.
__host__ __device__ inline size_t token_plan_words(size_t T, size_t nab, size_t wpr, size_t groups) {
    return T * wpr + (T + 31) / 32 * (nab + 1) + T + nab * 5 + 2 + groups * nab;
}

// Root of block b; every second pointer on the way is shortened (others may do the same: all of them point to ancestors).
__device__ __forceinline__ int plan_root(volatile int* parent, int b) {
    int p = parent[b];
    while (p != b) {
        const int q = parent[p];
        if (q != p) parent[b] = q;
        b = p;
        p = q;
    }
    return b;
}

__global__ void __launch_bounds__(1024, 1)
token_plan_kernel(TokenPlanArgs a) {
    constexpr int TM = limb::BM, TN = limb::BN, KC = limb::KC, MAX_TILES = 32768 / TM, WARPS = 32;
    extern __shared__ __align__(16) uint32_t plan_smem[];
    __shared__ int components, live_blocks;
    __shared__ unsigned edges, pairs;            // at most T * nab, which the host keeps below 2^31 / 16
    __shared__ int tile_lo[MAX_TILES], tile_hi[MAX_TILES], units_up[MAX_TILES], units_dn[MAX_TILES];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int T = a.T, nab = a.nab, wpr = a.wpr, groups = a.groups, bs = a.bs, chunks = (T + 31) / 32;
    const int INF = 0x7fffffff;
    uint32_t* bits = a.in_smem ? plan_smem : a.scratch;
    int* count = reinterpret_cast<int*>(bits + (size_t)T * wpr);      // [chunks][nab + 1], the last for rows of no component
    int* comp = count + (size_t)chunks * (nab + 1);                   // [T] root of the row's blocks, nab: none
    int* parent = comp + T;                                           // [nab] the forest
    int* least = parent + nab;                                        // [nab] smallest row of the component, at its root
    int* rows_of = least + nab;                                         // [nab + 1] rows of a component, at its root
    int* first_row = rows_of + nab + 1;                                 // [nab + 1] where they go in the sorted order
    int* bl = first_row + nab + 1;                                    // [nab] label of the block
    int* sorted_bl = bl + nab;                                        // [groups * nab]

    pdl_wait();
    for (int w = tid; w < T * wpr + chunks * (nab + 1); w += 1024) bits[w] = 0u;
    for (int b = tid; b < nab; b += 1024) {
        parent[b] = b;
        least[b] = INF;
    }
    if (tid == 0) { components = live_blocks = 0; edges = pairs = 0u; }
    __syncthreads();
    {
        // S is read (and kept) 16 bytes at a time where it lies on such a boundary, the rest singly
        const int total = T * nab, quads = (reinterpret_cast<uintptr_t>(a.S) & 15) == 0 ? total >> 4 : 0;
        const uint4* S16 = reinterpret_cast<const uint4*>(a.S);
        for (int q = tid; q < quads; q += 1024) {
            const uint4 v = __ldg(S16 + q);
            if (a.copy) reinterpret_cast<uint4*>(a.copy)[q] = v;
            int r = 16 * q / nab, b = 16 * q - r * nab;
            uint32_t found = 0u;                 // of word b / 32 of row r
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const uint32_t word = k < 4 ? v.x : k < 8 ? v.y : k < 12 ? v.z : v.w;
                if (word >> (8 * (k & 3)) & 0xffu) found |= 1u << (b & 31);
                ++b;
                if (k == 15 || b == nab || (b & 31) == 0) {
                    if (found) atomicOr(&bits[r * wpr + ((b - 1) >> 5)], found);
                    found = 0u;
                    if (b == nab) { b = 0; ++r; }
                }
            }
        }
        for (int t = 16 * quads + tid; t < total; t += 1024) {
            const uint8_t v = a.S[t];
            if (a.copy) a.copy[t] = v;
            if (v != 0) {
                const int r = t / nab, b = t - r * nab;
                atomicOr(&bits[r * wpr + (b >> 5)], 1u << (b & 31));
            }
        }
    }
    __syncthreads();
    // Every row joins its blocks.  First the first 64 rows, a thread per edge, which settles most of the forest; then, with every
    // block pointing at its root, the others, a thread per row, which mostly find their blocks joined.
    auto join = [&](int x, int y) {              // returns their root
        x = plan_root(parent, x);
        y = plan_root(parent, y);
        while (x != y) {
            const int hi = max(x, y), lo = min(x, y);
            if (atomicCAS(parent + hi, hi, lo) == hi) return lo;
            x = plan_root(parent, x);
            y = plan_root(parent, y);
        }
        return x;
    };
    for (int e = tid; e < min(T, 64) * nab; e += 1024) {
        const int r = e / nab, b = e - r * nab;
        const uint32_t* row = bits + r * wpr;
        if ((row[b >> 5] >> (b & 31) & 1u) == 0u) continue;
        int w = 0;
        while (row[w] == 0u) ++w;
        const int first = w * 32 + __ffs(row[w]) - 1;
        if (first != b) join(first, b);
    }
    __syncthreads();
    for (int b = tid; b < nab; b += 1024) parent[b] = plan_root(parent, b);
    __syncthreads();
    unsigned mine = 0;
    for (int r = tid; r < T; r += 1024) {
        int root = nab;
        for (int w = 0; w < wpr; ++w) {
            uint32_t v = bits[r * wpr + w];
            mine += __popc(v);
            for (; v; v &= v - 1) {
                const int y = *(volatile int*)(parent + w * 32 + __ffs(v) - 1);
                if (root == nab) root = y;
                if (root != y) root = join(root, y);
            }
        }
        comp[r] = root;                          // of the moment
    }
    __syncthreads();
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0 && mine) atomicAdd(&edges, mine);
    for (int chunk = warp; chunk < chunks; chunk += WARPS) {
        const int r = chunk * 32 + lane;
        int root = r < T ? comp[r] : -1;
        if (root >= 0 && root < nab) root = plan_root(parent, root);
        const unsigned same = __match_any_sync(0xffffffffu, root);
        if (r < T) {
            comp[r] = root;
            if (lane == __ffs(same) - 1) {
                count[chunk * (nab + 1) + root] = __popc(same);
                if (root < nab) atomicMin(least + root, r);
            }
        }
    }
    __syncthreads();
    // rows per component, and of those the rows before each chunk
    for (int b = tid; b <= nab; b += 1024) {
        int sum = 0;
        for (int k = 0; k < chunks; ++k) {
            const int n = count[k * (nab + 1) + b];
            count[k * (nab + 1) + b] = sum;
            sum += n;
        }
        rows_of[b] = sum;
    }
    __syncthreads();
    {
        int comps = 0, live_b = 0;
        unsigned my_pairs = 0;
        for (int b = tid; b < nab; b += 1024) {
            const int root = plan_root(parent, b), l = least[root] == INF ? -1 : least[root];
            bl[b] = l;
            a.blk_label[b] = l;
            live_b += l >= 0;
            comps += rows_of[b] > 0;
            my_pairs += l >= 0 ? rows_of[root] : 0;
        }
        if (tid - lane < nab) {
            comps = __reduce_add_sync(0xffffffffu, comps);
            live_b = __reduce_add_sync(0xffffffffu, live_b);
            my_pairs = __reduce_add_sync(0xffffffffu, my_pairs);
            if (lane == 0) {
                atomicAdd(&components, comps);
                atomicAdd(&live_blocks, live_b);
                atomicAdd(&pairs, my_pairs);
            }
        }
        for (int r = tid; r < T; r += 1024) a.row_label[r] = comp[r] < nab ? least[comp[r]] : -1;
    }
    const int M = T - rows_of[nab];                // rows with an edge; the others come after them
    __syncthreads();
    const int NB = live_blocks;
    // ---- component-sorted order
    for (int b = tid; a.plan && b < nab; b += 1024) {
        const int l = bl[b];
        int less = 0, same = 0, before = 0, rows = 0;
        for (int q = 0; q < nab; ++q) {
            const int lq = bl[q];
            less += lq >= 0 && lq < l;
            same += lq == l;
            before += lq == l && q < b;
            rows += lq < l ? rows_of[q] : 0;       // zero but at a root
        }
        first_row[b] = rows;
        if (l >= 0) {
            for (int g = 0; g < groups; ++g) {
                a.col_map[groups * less + g * same + before] = g * nab + b;
                sorted_bl[groups * less + g * same + before] = l;
            }
            a.kmap[less + before] = b;
        } else {
            for (int g = 0; g < groups; ++g) {
                a.col_map[groups * NB + g * (nab - NB) + before] = g * nab + b;
                sorted_bl[groups * NB + g * (nab - NB) + before] = -1;
            }
            a.kmap[NB + before] = b;
        }
    }
    if (tid == 0) first_row[nab] = M;
    __syncthreads();
    for (int chunk = warp; a.plan && chunk < chunks; chunk += WARPS) {
        const int r = chunk * 32 + lane, c = r < T ? comp[r] : -1;
        const unsigned same = __match_any_sync(0xffffffffu, c);
        if (c < 0) continue;
        const int pos = first_row[c] + count[chunk * (nab + 1) + c] + __popc(same & ((1u << lane) - 1u));
        a.row_map[pos] = r;
        if (c < nab) {
            if (pos % TM == 0) tile_lo[pos / TM] = least[c];
            if (pos % TM == TM - 1 || pos == M - 1) tile_hi[pos / TM] = least[c];
        }
    }
    __syncthreads();

    // ---- the work of every row tile, a warp per tile
    const int N = groups * NB * bs, mt = a.plan ? (M + TM - 1) / TM : 0, nt = (N + TN - 1) / TN;
    for (int tm = warp; tm < mt; tm += WARPS) {
        const int lo_m = tile_lo[tm], hi_m = tile_hi[tm];
        int first = -1, count = 0;
        for (int t0 = 0; t0 < nt; t0 += 32) {
            const int tn = t0 + lane;
            const bool hit = tn < nt && sorted_bl[(min(tn * TN + TN, N) - 1) / bs] >= lo_m && sorted_bl[(tn * TN) / bs] <= hi_m;
            const unsigned hits = __ballot_sync(0xffffffffu, hit);
            if (first < 0 && hits) first = t0 + __ffs(hits) - 1;
            count += __popc(hits);
        }
        int blk_begin = 0, blk_end = 0;          // sorted block positions of the components lo_m .. hi_m
        for (int q = lane; q < nab; q += 32) {
            const int lq = bl[q];
            blk_begin += lq >= 0 && lq < lo_m;
            blk_end += lq >= 0 && lq <= hi_m;
        }
        blk_begin = __reduce_add_sync(0xffffffffu, blk_begin);
        blk_end = __reduce_add_sync(0xffffffffu, blk_end);
        const int klo = (blk_begin * bs) / KC, khi = (blk_end * bs + KC - 1) / KC;
        if (lane == 0) {
            a.up[tm].tn0 = max(first, 0);
            a.up[tm].ntn = count;
            a.up[tm].klo = 0;
            a.up[tm].kcnt = a.kb_up;
            units_up[tm] = count * 2 * a.kb_up;
            a.dn[tm].tn0 = 0;
            a.dn[tm].ntn = a.nt_dn;
            a.dn[tm].klo = klo;
            a.dn[tm].kcnt = khi - klo;
            units_dn[tm] = a.nt_dn * 2 * (khi - klo);
        }
    }
    __syncthreads();
    if (tid == 0) {
        int off_up = 0, off_dn = 0;
        for (int tm = 0; tm < mt; ++tm) {
            a.up[tm].unit0 = off_up;
            a.dn[tm].unit0 = off_dn;
            off_up += units_up[tm];
            off_dn += units_dn[tm];
        }
        const unsigned long long words[PLAN_WORDS] = {edges, (unsigned)components, (unsigned)M, (unsigned)NB, (unsigned)off_up,
                                                      pairs, (unsigned)off_dn};
#pragma unroll
        for (int k = 0; k < PLAN_WORDS; ++k)
            reinterpret_cast<volatile unsigned long long*>(a.report)[k] = a.ticket << PLAN_VALUE_BITS | words[k];
    }
}

struct LimbArgs {
    const uint8_t* Epl;      // left planes of E = E_0 + E_1: [m-tile][k-block][32 KiB]
    const uint8_t* Vpl[2];   // left planes of V_i = A_i + i*E
    const uint8_t* Bpl[2];   // right planes of B_i: [n-tile][k-block][16 KiB]
    const uint8_t* Fpl;      // right planes of F = F_0 + F_1
    u64* Z[2];               // [M, N], pre-loaded with C_i; partial sums are added with bulk reductions
    int M, N;                // N a multiple of 16
    int mt, nt, kb;          // tiles and k-blocks per operand pair; one tile runs over 2*kb blocks
    int parts;               // CTAs to a tile (limb_parts), or 0: all tiles' blocks in equal ranges
    int* error_flag;         // set to 1 if a bounded wait ran out
    int* error_host;         // the same report in mapped host memory, so that the host sees it without a copy
    // Only read by the grouped kernel (one multiplication per connected component): the planes hold the operands
    // in component-sorted order, M counts the rows that lie in a component (and N the columns, when col_map is
    // given), and every row tile runs over the column tiles and k-blocks its LimbGroupRow names.  kb stays the
    // number of k-blocks per plane tile in memory.  A finished row piece goes to row row_map[r] of Z, whose rows are
    // ldz words long, and the 16 columns from sorted column c on to compact columns
    // col_map[c / bs] * bs + c % bs.. (bs is a multiple of 16; col_map null: column c itself).
    int ldz, bs;
    int group_units;             // units per party: sum over row tiles of ntn * 2 * kcnt
    const LimbGroupRow* groups;  // [mt]
    const int32_t* row_map;      // [M] sorted row -> row of Z
    const int32_t* col_map;      // [N / bs] sorted block -> compact block of Z, or null
    // Component labels of Z's rows and of the active blocks, with col_map: the Merge step of Protocol 2.  A tile may touch
    // several components; what it holds outside them (a piece of a row whose block has another label) is left out, and Z holds
    // zero there (limb_exchange_kernel).  As a pass over Z after the product it took 5 us and a launch of 512 tokens x 832.
    const int32_t* row_label;
    const int32_t* blk_label;
    int blocks;                  // active blocks
};

// Slow path of a bounded wait, kept out of line so that the polling loops of the three roles stay short.
__device__ __noinline__ bool limb_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    const long long t0 = clock64();
    for (;;) {
        for (int i = 0; i < 128; ++i)
            if (ptx::mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > limb::WAIT_CYCLES) {
            *abort_flag = 1;
            return false;
        }
    }
}

// Bounded wait: false (and the CTA-wide abort flag raised) if the barrier did not flip in time or another
// role already gave up.
__device__ __forceinline__ bool limb_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    return limb_wait_slow(bar, parity, abort_flag);
}

// The epilogue warps' wait for a finished segment lasts tens of microseconds and involves 256 threads: one lane
// per warp polls, sleeping between polls so that the warp leaves the issue slots to whoever shares the SM (a
// co-resident memory-side CTA), and then every lane acquires the completed phase with one (succeeding) poll.
__device__ __noinline__ bool limb_wait_sleeping(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    const long long t0 = clock64();
    for (;;) {
        if (ptx::mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > limb::WAIT_CYCLES) {
            *abort_flag = 1;
            return false;
        }
        __nanosleep(40);
    }
}

__device__ __forceinline__ bool limb_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    bool ok = true;
    if ((threadIdx.x & 31) == 0) ok = limb_wait_sleeping(bar, parity, abort_flag);
    ok = __shfl_sync(0xffffffffu, ok, 0);      // also reconverges the warp for the aligned TMEM loads
    if (ok) ok = limb_wait(bar, parity, abort_flag);
    return __all_sync(0xffffffffu, ok);
}

// Z = sum_s 2^(8s) D_s mod 2^64 from the eight 32-bit accumulators of one output element: the terms with s <= 3 are
// 32 x 32 -> 64-bit multiply-adds by 2^(8s), the terms with s >= 4 only reach the high word (32-bit shifts and adds).
__device__ __forceinline__ u64 limb_recombine(uint32_t d0, uint32_t d1, uint32_t d2, uint32_t d3, uint32_t d4,
                                              uint32_t d5, uint32_t d6, uint32_t d7) {
    u64 v = (u64)d0;
    v += (u64)d1 * (u64)(1u << 8);
    v += (u64)d2 * (u64)(1u << 16);
    v += (u64)d3 * (u64)(1u << 24);
    const uint32_t hi = (uint32_t)(v >> 32) + d4 + (d5 << 8) + (d6 << 16) + (d7 << 24);
    return ((u64)hi << 32) | (u64)(uint32_t)v;
}

// One contiguous piece of a CTA's share of the (party, tile, k-block) space: a run of k-blocks of one tile.
struct LimbSegment {
    int party, tm, tn;
    int kpos;        // first k-block, in [0, 2*kb): blocks [0,kb) pair E with B_i, [kb,2kb) pair V_i with F
    int count;       // k-blocks in this segment, <= MAX_SEGMENT_UNITS
    int kb, klo;     // grouped kernel only: k-blocks per operand pair of this tile and the first of them
};

template <bool GROUPED = false>
__device__ __forceinline__ LimbSegment limb_segment(const LimbArgs& a, long long u, long long u_end) {
    LimbSegment s;
    long long seg_end;
    if (GROUPED) {
        s.party = (int)(u / a.group_units);
        const int ul = (int)(u - (long long)s.party * a.group_units);
        int tm = 0;
        while (tm + 1 < a.mt && __ldg(&a.groups[tm + 1].unit0) <= ul) ++tm;     // row tiles without work are passed over
        const int unit0 = __ldg(&a.groups[tm].unit0);
        s.kb = __ldg(&a.groups[tm].kcnt);
        s.klo = __ldg(&a.groups[tm].klo);
        const int tile_units = 2 * s.kb, r = ul - unit0, ti = r / tile_units;
        s.tm = tm;
        s.tn = __ldg(&a.groups[tm].tn0) + ti;
        s.kpos = r - ti * tile_units;
        seg_end = u - s.kpos + tile_units;
    } else {
        const long long tile_units = 2ll * a.kb;
        const long long tile = u / tile_units;
        seg_end = (tile + 1) * tile_units;
        const int per_party = a.mt * a.nt;
        s.party = (int)(tile / per_party);
        const int t2 = (int)(tile - (long long)s.party * per_party);
        s.tm = t2 / a.nt;
        s.tn = t2 - s.tm * a.nt;
        s.kpos = (int)(u - tile * tile_units);
        s.kb = a.kb;
        s.klo = 0;
    }
    if (seg_end > u_end) seg_end = u_end;
    if (seg_end > u + limb::MAX_SEGMENT_UNITS) seg_end = u + limb::MAX_SEGMENT_UNITS;
    s.count = (int)(seg_end - u);
    return s;
}

// Low / high word of a shared-memory matrix descriptor, K-major, no swizzle: bits 0-13 address>>4, 16-29 leading
// byte offset>>4 (between the two 16-byte K halves), 32-45 stride byte offset>>4 (between 8-row groups), 46-47
// descriptor version 1.
__device__ __forceinline__ uint32_t limb_desc_lo(uint32_t addr) {
    return ((addr & 0x3FFFFu) >> 4) | ((uint32_t)(limb::LBO_BYTES >> 4) << 16);
}
constexpr uint32_t LIMB_DESC_HI = (uint32_t)(limb::SBO_BYTES >> 4) | (1u << 14);

template <bool GROUPED>
__device__ __forceinline__ void combine_limb_body(const LimbArgs& a, const CUtensorMap* z_maps) {
    using namespace limb;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[STAGES];
    __shared__ __align__(8) uint64_t empty_bar[STAGES];
    __shared__ __align__(8) uint64_t accum_full_bar, accum_empty_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = smem;
    uint8_t* sB = smem + (size_t)STAGES * A_BLOCK_BYTES;
    uint8_t* sOut = sB + (size_t)STAGES * B_BLOCK_BYTES;      // EPI_WARPS x 32 rows x OUT_ROW_BYTES

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long total_units = GROUPED ? 2ll * a.group_units : 2ll * a.mt * a.nt * 2ll * a.kb;
    long long u_begin, u_end;
    if (!GROUPED && a.parts) {                   // one part of one tile
        const unsigned tile = blockIdx.x / (unsigned)a.parts, part = blockIdx.x - tile * a.parts;
        const long long first = 2ll * a.kb * tile;
        u_begin = first + 2u * (unsigned)a.kb * part / (unsigned)a.parts;
        u_end = first + 2u * (unsigned)a.kb * (part + 1) / (unsigned)a.parts;
    } else {
        u_begin = total_units * blockIdx.x / gridDim.x;
        u_end = total_units * (blockIdx.x + 1) / gridDim.x;
    }

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&full_bar[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&empty_bar[s]), 1);
        }
        ptx::mbar_init(ptx::smem_u32(&accum_full_bar), 1);
        ptx::mbar_init(ptx::smem_u32(&accum_empty_bar), 32 * EPI_WARPS);
        abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 0) {
        ptx::tmem_alloc(ptx::smem_u32(&tmem_slot), 512);
        ptx::tmem_relinquish();
    }
    ptx::fence_before_sync();
    __syncthreads();
    ptx::fence_after_sync();
    const uint32_t tmem_base = tmem_slot;
    // barriers and tensor memory are set up; from here on the kernel touches what its predecessors wrote
    pdl_wait();

    if (warp == EPI_WARPS) {
        // ---------------- producer: one bulk copy per operand block ----------------
        if (ptx::elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            int issued = 0;
            bool ok = true;
            const uint32_t full0 = ptx::smem_u32(&full_bar[0]), empty0 = ptx::smem_u32(&empty_bar[0]);
            const uint32_t sA0 = ptx::smem_u32(sA), sB0 = ptx::smem_u32(sB);
            for (long long u = u_begin; u < u_end && ok;) {
                const LimbSegment sg = limb_segment<GROUPED>(a, u, u_end);
                u += sg.count;
                int kpos = sg.kpos;
                const int kbe = GROUPED ? sg.kb : a.kb;       // k-blocks per operand pair of this tile
                const int klo = GROUPED ? sg.klo : 0;         // and where they start in the plane tile
                bool second = kpos >= kbe;
                if (second) kpos -= kbe;
                const uint8_t* left = (second ? (sg.party ? a.Vpl[1] : a.Vpl[0]) : a.Epl) +
                                      ((size_t)sg.tm * a.kb + klo + kpos) * A_BLOCK_BYTES;
                const uint8_t* right = (second ? a.Fpl : (sg.party ? a.Bpl[1] : a.Bpl[0])) +
                                       ((size_t)sg.tn * a.kb + klo + kpos) * B_BLOCK_BYTES;
                for (int it = 0; it < sg.count; ++it) {
                    ok = limb_wait(empty0 + 8 * stage, phase ^ 1u, &abort_flag);
                    if (!ok) break;
                    const uint32_t bar = full0 + 8 * stage;
                    ptx::mbar_expect_tx(bar, A_BLOCK_BYTES + B_BLOCK_BYTES);
                    ptx::bulk_g2s(sA0 + stage * A_BLOCK_BYTES, left, A_BLOCK_BYTES, bar);
                    ptx::bulk_g2s(sB0 + stage * B_BLOCK_BYTES, right, B_BLOCK_BYTES, bar);
                    ++issued;
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                    left += A_BLOCK_BYTES;
                    right += B_BLOCK_BYTES;
                    if (++kpos == kbe && !second) {
                        // the tile's first product (E with B_i) is done: go on with the second (V_i with F)
                        second = true;
                        kpos = 0;
                        left = (sg.party ? a.Vpl[1] : a.Vpl[0]) + ((size_t)sg.tm * a.kb + klo) * A_BLOCK_BYTES;
                        right = a.Fpl + ((size_t)sg.tn * a.kb + klo) * B_BLOCK_BYTES;
                    }
                }
            }
            if (!ok) {
                // gave up: let the copies already in flight land before the CTA leaves
                const int back = issued < STAGES ? issued : STAGES;
                for (int j = 1; j <= back; ++j) {
                    int s = stage - j;
                    uint32_t ph = phase;
                    if (s < 0) { s += STAGES; ph ^= 1u; }
                    const long long t0 = clock64();
                    while (!ptx::mbar_try_wait(ptx::smem_u32(&full_bar[s]), ph) && clock64() - t0 < 20000000ll) {}
                }
            }
        }
    } else if (warp == EPI_WARPS + 1) {
        // ---------------- MMA issuer: 12 instructions per k-block, as little else as possible ----------------
        if (ptx::elect_one()) {
            // instruction descriptor: s32 accumulate, u8 x u8, both K-major, M = 128, N filled in per instruction
            constexpr uint32_t IDESC = (2u << 4) | ((uint32_t)(BM >> 4) << 24);
            const uint32_t full0 = ptx::smem_u32(&full_bar[0]), empty0 = ptx::smem_u32(&empty_bar[0]);
            const uint32_t accum_full = ptx::smem_u32(&accum_full_bar), accum_empty = ptx::smem_u32(&accum_empty_bar);
            const uint32_t a_lo0 = limb_desc_lo(ptx::smem_u32(sA)), b_lo0 = limb_desc_lo(ptx::smem_u32(sB));
            int stage = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            for (long long u = u_begin; u < u_end && ok;) {
                const LimbSegment sg = limb_segment<GROUPED>(a, u, u_end);
                u += sg.count;
                ok = limb_wait(accum_empty, acc_phase ^ 1u, &abort_flag);
                if (!ok) break;
                ptx::fence_after_sync();
                uint32_t acc = 0;                         // the segment's first block overwrites the accumulators
                for (int it = 0; it < sg.count; ++it) {
                    ok = limb_wait(full0 + 8 * stage, phase, &abort_flag);
                    if (!ok) break;
                    ptx::fence_after_sync();
                    const uint32_t a_lo = a_lo0 + stage * (A_BLOCK_BYTES >> 4);
                    const uint32_t b_lo = b_lo0 + stage * (B_BLOCK_BYTES >> 4);
                    const uint32_t b_lo_hi = b_lo + ((256 * KC) >> 4);         // right-operand rows 256.. (planes 4..7)
                    // Left plane p meets right planes 0..7-p, whose products land in accumulators D_p..D_7: one
                    // instruction of N = 64*(8-p), cut at 256.  When a plane issues two instructions the second
                    // takes the left operand from the collector instead of shared memory.
#pragma unroll
                    for (int i = 0; i < PLANES; ++i) {
                        // wide and narrow instructions alternate (plane 0, which overwrites every accumulator when a
                        // segment starts, stays first)
                        const int p = (i & 1) ? PLANES - 1 - (i >> 1) : (i >> 1);
                        const uint32_t ap = a_lo + ((p * BM * KC) >> 4);
                        const int n_total = BN * (PLANES - p);
                        const uint32_t acc_p = p == 0 ? acc : 1u;
                        if (n_total > 256) {
                            ptx::mma_i8_keep_a(tmem_base + BN * p, ap, LIMB_DESC_HI, b_lo, LIMB_DESC_HI,
                                               IDESC | ((uint32_t)(256 >> 3) << 17), acc_p);
                            ptx::mma_i8_reuse_a(tmem_base + BN * p + 256, ap, LIMB_DESC_HI, b_lo_hi, LIMB_DESC_HI,
                                                IDESC | ((uint32_t)((n_total - 256) >> 3) << 17), acc_p);
                        } else {
                            ptx::mma_i8(tmem_base + BN * p, ap, LIMB_DESC_HI, b_lo, LIMB_DESC_HI,
                                        IDESC | ((uint32_t)(n_total >> 3) << 17), acc_p);
                        }
                    }
                    ptx::mma_commit(empty0 + 8 * stage);    // frees the stage once the MMAs have read it
                    acc = 1u;
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                ptx::mma_commit(accum_full);
                acc_phase ^= 1u;
            }
            // the main loop is over: the next kernel of the stream may be brought in beside the last drain
            pdl_launch_dependents();
        }
    } else {
        // ---------------- epilogue: TMEM -> registers -> recombine mod 2^64 -> release TMEM ->
        //                  stage the rows in shared memory -> one bulk add-reduction per row into Z ----------------
        uint32_t acc_phase = 0;
        bool ok = true;
        const int quarter = warp & 3, chalf = warp >> 2;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16) + chalf * 32;
        // this lane's row in the warp's staging tile
        uint8_t* my_row = GROUPED ? sOut + ((size_t)warp * 32 + lane) * OUT_ROW_BYTES
                                  : sOut + (size_t)warp * OUT_TILE_BYTES + lane * (OUT_COLS * 8);
        const uint32_t my_row_s = ptx::smem_u32(my_row);
        for (long long u = u_begin; u < u_end && ok;) {
            const LimbSegment sg = limb_segment<GROUPED>(a, u, u_end);
            u += sg.count;
            ok = limb_wait_warp(ptx::smem_u32(&accum_full_bar), acc_phase, &abort_flag);
            if (!ok) break;
            ptx::fence_after_sync();
            const int row = sg.tm * BM + quarter * 32 + lane;
            const int col0 = sg.tn * BN + chalf * 32;
            u64* zrow = nullptr;
            int label = 0;
            if (GROUPED) {
                const int at = row < a.M ? __ldg(a.row_map + row) : 0;
                zrow = (sg.party ? a.Z[1] : a.Z[0]) + (size_t)at * a.ldz;
                if (a.col_map) label = __ldg(a.row_label + at);
            }
#pragma unroll
            for (int h = 0; h < 32 / OUT_COLS; ++h) {          // this thread's 32 columns, OUT_COLS at a time
                u64 v[OUT_COLS];
#pragma unroll
                for (int c = 0; c < OUT_COLS / 8; ++c) {
                    uint32_t d[PLANES][8];
#pragma unroll
                    for (int s = 0; s < PLANES; ++s) ptx::tmem_ld8(lane_base + BN * s + h * OUT_COLS + c * 8, d[s]);
                    ptx::tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        v[c * 8 + j] = limb_recombine(d[0][j], d[1][j], d[2][j], d[3][j], d[4][j], d[5][j], d[6][j],
                                                      d[7][j]);
                }
                if (h == 32 / OUT_COLS - 1) {
                    // every accumulator has been read: hand TMEM back before anything that waits on the copy engine
                    ptx::fence_before_sync();
                    ptx::mbar_arrive(ptx::smem_u32(&accum_empty_bar));
                }
                if (GROUPED) {
                    ptx::bulk_wait_group_read0();              // the previous reduction has read this thread's staging row
#pragma unroll
                    for (int j = 0; j < OUT_COLS; j += 2)
                        *reinterpret_cast<ulonglong2*>(my_row + j * 8) = make_ulonglong2(v[j], v[j + 1]);
                    int cols = a.N - col0 - h * OUT_COLS;
                    if (cols > OUT_COLS) cols = OUT_COLS;
                    if (row < a.M && cols > 0) {
                        ptx::fence_proxy_async_smem();     // this thread's row, written above, is read by the copy engine
                        const int c = col0 + h * OUT_COLS, blk = c / a.bs;
                        u64* dst = zrow + c;
                        bool inside = true;
                        if (a.col_map) {
                            const int at = __ldg(a.col_map + blk);
                            dst = zrow + (size_t)at * a.bs + (c - blk * a.bs);
                            inside = __ldg(a.blk_label + at % a.blocks) == label;
                        }
                        if (inside) ptx::bulk_reduce_add_u64(dst, my_row_s, (uint32_t)cols * 8u);
                    }
                    ptx::bulk_commit_group();
                } else {
                    // One tensor reduction takes the warp's 32 x 16 words.  (One bulk reduction per row costs some 70 cycles
                    // of issue each, 64 of them per warp and tile: a product of two k-blocks' work per CTA took 13.7 us, with
                    // this 11.2.)
                    if (lane == 0) ptx::bulk_wait_group_read0();
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < OUT_COLS; j += 2)
                        *reinterpret_cast<ulonglong2*>(my_row + (((j >> 1) ^ (lane & 7)) << 4)) = make_ulonglong2(v[j], v[j + 1]);
                    ptx::fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        const int x = col0 + h * OUT_COLS, y = sg.tm * BM + quarter * 32;
                        if (x < a.N && y < a.M) ptx::tensor_reduce_add(z_maps + sg.party, my_row_s, x, y);
                        ptx::bulk_commit_group();
                    }
                }
            }
            acc_phase ^= 1u;
        }
        ptx::bulk_wait_group0();                       // every reduction of this thread has completed
    }

    ptx::fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) {
        *a.error_flag = 1;
        *reinterpret_cast<volatile int*>(a.error_host) = 1;
        __threadfence_system();
    }
    if (warp == 0) {
        ptx::fence_after_sync();
        ptx::tmem_dealloc(tmem_base, 512);
    }
}

struct LimbMaps {
    CUtensorMap z[2];            // Z_0, Z_1 as [M, N] matrices of 64-bit integers, boxes of 32 rows x 16 words, 128-byte swizzle
};

__global__ void __launch_bounds__(limb::THREADS, 1)
combine_limb_kernel(const __grid_constant__ LimbArgs a, const __grid_constant__ LimbMaps maps) {
    combine_limb_body<false>(a, maps.z);
}

// One multiplication per connected component (Protocols 2 and 3 under a per-token mask): the same kernel over the
// tiles and k-blocks of the component-sorted operands that have work, scattering the result rows back to Z.
__global__ void __launch_bounds__(limb::THREADS, 1)
combine_limb_grouped_kernel(const __grid_constant__ LimbArgs a) {
    combine_limb_body<true>(a, nullptr);
}

}  // namespace comet
