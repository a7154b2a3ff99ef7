// One Pi_MatMul for few token rows (the decode step) in one kernel: mask, exchange and combine without a pass over
// memory in between.
//   before the exchange   E_i = X_i - A_i,  F_i = gather(W_i) - B_i          (Section 2.1 "Multiplication", the gathers
//                                                                             of Protocols 2 and 3), written as messages
//   the exchange          E = E_0 + E_1,  F = F_0 + F_1
//   after it              Z_i += E*B_i + V_i*F,  V_i = A_i + i*E              (Eq. 1; Z_i holds C_i when it starts)
//
// What bounds it: with at most 32 token rows a weight word takes part in 2 * 32 multiply-adds per party, so the kernel
// is bound by streaming the weight side.  Per word of the right operand and party that is W_i and B_i in and F_i out,
// 24 bytes, and this kernel moves nothing else of that size: the limb planes the tensor cores read exist in shared
// memory only.  (Its predecessor wrote the planes of B_i and F_i to memory and read them back: 56 bytes per word.)
// Measured, both parties: [32, 4096] x [4096, 1312] 50 us and [7, 4096] x [4096, 3328] 104 us from a CTA's start to its end,
// where 24 bytes per weight word at the measured copy rate are 39 and 100 us; a step of 192 KiB takes 8400 cycles, 95 % of that
// rate, the rest is 2 us until the first bytes arrive and 4 us from the last planes to the end (MMAs 3100 cycles, drain of 32
// tokens 4000, of 7 tokens 1200, the reductions' completion 900).
//
// A CTA carries both parties' share of a tile of 128 output features (the rows of the MMA; 32 of them in small products, see the
// kernel's FEATURES) x 32 tokens, and walks it in
// steps of 32 contraction indices.  What is computed for a party depends on that party's shares and on the two messages
// alone; both parties' words of one place pass through the same thread, which is the exchange.
//   warps 16-17   raw producers, one per party: 16-byte asynchronous copies of W_i, B_i (32 rows x 32 words of each per
//                 slot) into a ring of three 32 KiB slots
//   warps 0-15    converters, two groups of eight that take the four slots of a step in turn: words -> messages F_0, F_1
//                 (to memory) and their sum -> limb planes of B_0, B_1, F
//   warps 18-25   the token side, four rows each: X_i, A_i straight from L2, a step ahead -> messages E_0, E_1 -> limb
//                 planes of E, A_0, A_1 + E; at the end of a segment the same warps are the epilogue (four per party): TMEM
//                 -> recombine mod 2^64 -> rows staged in shared memory -> tensor add-reductions into Z
//   warp 26       issues the MMAs: F is the same for both parties, so three weight-side plane sets serve four products
//   warp 27       Z_i <- C_i for the tiles that begin in this CTA's range, and a flag on each, which every CTA that adds to the
//                 tile waits for.  (As a kernel of its own before this one it cost a launch, and 1.5 us between two products.)
// Shared memory: 96 KiB weight planes, 24 KiB token planes, 96 KiB raw ring, 8 KiB result rows; all 512 TMEM columns (two
// parties x eight accumulators x 32 tokens).  The planes are single-buffered: converting a step and multiplying it take
// turns, while the ring and the converters' registers keep up to 160 KiB of loads in flight.
//
// The contraction indices of a step sit in the planes in limb_emit4's order (kernels_limb.cuh).
//
// Work is cut stream-K style like the other tensor-core kernel's: the (feature tile, token tile, step) space in equal
// contiguous ranges, a step weighted by the number of raw slots it takes (a ragged last tile takes fewer) and a constant; with
// no more steps than SMs every CTA has one.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "kernels_limb.cuh"
#include "pdl.cuh"

namespace comet {

namespace limb_stream {
constexpr int BW = 128, BT = 32, KC = limb::KC, PLANES = limb::PLANES, QROWS = 32, QUARTERS = BW / QROWS;
constexpr int CONV_GROUPS = 2, GROUP_WARPS = 8, CONV_WARPS = CONV_GROUPS * GROUP_WARPS;
constexpr int RAW_WARP0 = CONV_WARPS, TOK_WARP0 = RAW_WARP0 + 2, TOK_WARPS = 8, MMA_WARP = TOK_WARP0 + TOK_WARPS;
constexpr int EPI_WARPS = TOK_WARPS / 2;                 // per party
constexpr int SMALL_WORKERS = 3;                         // warps per party that drain a small tile
constexpr int INIT_WARP = MMA_WARP + 1, THREADS = 32 * (INIT_WARP + 1);
constexpr int RAW_ARRAY_BYTES = QROWS * KC * 8;          // 8 KiB: one array of a slot
constexpr int RAW_SLOT_BYTES = 4 * RAW_ARRAY_BYTES;      // party 0: W | B, party 1: W | B
constexpr int RAW_SLOTS = 3;
constexpr int W_PLANE_BYTES = BW * KC;
constexpr int W_SET_BYTES = PLANES * W_PLANE_BYTES;      // 32 KiB: limb planes of B_0, B_1 or F
constexpr int T_SET_BYTES = PLANES * BT * KC;            //  8 KiB: limb planes of V_0, V_1 or E
constexpr int OUT_TOKENS = 4;                            // tokens an epilogue thread recombines at a time
constexpr int OUT_BYTES = OUT_TOKENS * 32 * 8;           // an epilogue warp's staging buffer: a row of 32 features per token
constexpr int ACC_COLS = PLANES * BT;                    // 256 TMEM columns per party
constexpr int SYNC_WORDS = 2;                            // of StreamArgs::sync before the tiles' flags
// A step adds two products to an accumulator, so the bound on a segment's depth (16384 contraction indices keep the
// limb sums for s <= 3 below 2^32) allows half as many steps.
constexpr int MAX_SEGMENT_STEPS = limb::MAX_SEGMENT_UNITS / 2;
// What a step costs besides its slots, in slots: the MMAs and the hand-over of the planes take turns with the conversion.
// Measured on [32, 4096] x [4096, 1312]: 8600 cycles with four slots, 4800 to 5600 with one (the last tile's).  Counted as one
// slot, the CTAs of that tile ran 67 us where the others took 52, and the layer 134 us; as three 124.4, as five 122.2.
constexpr int STEP_SLOTS = 5;
// And what Z <- C costs for one token row of a tile, in sixteenths of a slot: 4 KiB of traffic are three, and the first planes
// wait for it.  Counted as nothing the opt6.7b decode layer takes 122 us, as three 119.5, as five 116.6.
constexpr int OWN_SIXTEENTHS = 5;
constexpr size_t SMEM_BYTES = 3 * (size_t)W_SET_BYTES + 3 * (size_t)T_SET_BYTES + (size_t)RAW_SLOTS * RAW_SLOT_BYTES +
                              (size_t)TOK_WARPS * OUT_BYTES + 128;
}  // namespace limb_stream

struct StreamArgs {
    const u64* X[2]; const u64* A[2];                     // token side, [M, K]
    u64* E[2];                                            // message, [M, K]
    const u64* W0[2]; const u64* W1[2]; const u64* W2[2]; // weights of the stacked groups (down: W0 alone)
    const u64* B[2];                                      // [N, K]
    u64* F[2];                                            // message, [N, K]
    u64* Z[2];                                            // [M, N]
    const u64* C[2];                                      // [M, N]: what the sums are added to
    // [SYNC_WORDS + tiles] words of one context, or null (then Z holds C when the kernel before this one has completed).  The
    // first two are one 64-bit word: the number of launches so far, above the tickets taken of this one.  Then, per tile, the
    // epoch (launches before it plus one, never 0) of the last launch in which its part of Z became C.  All zero to begin with,
    // and advanced on the device alone: a launch may be captured once and run any number of times.
    uint32_t* sync;
    int gather;              // 0: the right operand is W0 itself, [N, K]
    const int32_t* ids;      // ascending active block ids, or null: they are in the launch's BlockIds
    int n, bs;               // active neurons, neurons per block (a multiple of 16 when there are ids)
    int M, N, K;             // K a multiple of 8
    int ldw, down;           // words per row of W; gather rows (up) or strips of bs words of every row (down)
    int mt, nt, kb;          // token tiles, feature tiles, steps per tile
    // how the steps are dealt out: a step costs the raw slots it takes, and STEP_SLOTS for what does not depend on them
    int last_cost;           // of a step of the last, possibly ragged, feature tile
    unsigned own_cost;       // of Z <- C for a tile, before its first step
    unsigned cta_cost, cta_extra;   // total cost = gridDim.x * cta_cost + cta_extra, cta_extra < gridDim.x; 0: a step per CTA
    const uint8_t* tmask;    // per-token mask [M, tmask_ld] over the active blocks of the contraction index, or null:
    int tmask_ld;            // where it is zero, neither X nor A_i has an entry
    const int32_t* row_label;   // component label per token (negative: the row is not opened), or null
    const int32_t* blk_label;   // likewise per active block (up: rows of the right operand, down: its columns), or null
    int* error_flag;
    int* error_host;         // or null
};

// Z_i <- C_i for both parties, so that the product kernel behind it can add partial sums.
__global__ void __launch_bounds__(256)
result_init_kernel(const u64* __restrict__ c0, const u64* __restrict__ c1, u64* __restrict__ z0, u64* __restrict__ z1,
                   long long pairs) {
    pdl_launch_dependents();             // the product's CTAs are set up meanwhile; they wait for this kernel's end
    pdl_wait();
    const ulonglong2* __restrict__ s = reinterpret_cast<const ulonglong2*>(blockIdx.y ? c1 : c0);
    ulonglong2* __restrict__ d = reinterpret_cast<ulonglong2*>(blockIdx.y ? z1 : z0);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < pairs; t += stride) d[t] = __ldcs(s + t);
}

// A run of steps of one tile, at most MAX_SEGMENT_STEPS of them.
struct StreamSegment {
    int tile, tm, tn, step, count;
};

__device__ __forceinline__ StreamSegment stream_segment(const StreamArgs& a, unsigned u, unsigned u_end) {
    StreamSegment s;
    const unsigned tile = u / (unsigned)a.kb;
    s.tile = (int)tile;
    s.step = (int)(u - tile * a.kb);
    s.tn = a.mt == 1 ? (int)tile : (int)(tile / (unsigned)a.mt);
    s.tm = (int)tile - s.tn * a.mt;
    s.count = min(min(a.kb - s.step, (int)(u_end - u)), limb_stream::MAX_SEGMENT_STEPS);
    return s;
}

// Raw slots the weight side of a feature tile takes per step.
template <int FEATURES>
__device__ __forceinline__ int stream_quarters(const StreamArgs& a, int tn) {
    if (FEATURES < limb_stream::BW) return 1;
    return tn + 1 < a.nt ? limb_stream::QUARTERS : a.last_cost - limb_stream::STEP_SLOTS;
}

// First step of the range that begins at cost b * cta_cost + min(b, cta_extra).
__device__ __forceinline__ unsigned stream_cut(const StreamArgs& a, unsigned b) {
    if (a.cta_cost == 0) return b;
    constexpr unsigned FULL = limb_stream::QUARTERS + limb_stream::STEP_SLOTS;
    const unsigned kb = (unsigned)a.kb, full_tiles = (unsigned)a.mt * (unsigned)(a.nt - 1);
    unsigned cost = b * a.cta_cost + min(b, a.cta_extra), step_cost = FULL, tile = 0;
    if (cost >= full_tiles * (a.own_cost + kb * FULL)) {
        cost -= full_tiles * (a.own_cost + kb * FULL);
        step_cost = (unsigned)a.last_cost;
        tile = full_tiles;
    }
    const unsigned tile_cost = a.own_cost + kb * step_cost, t = cost / tile_cost, in = cost - t * tile_cost;
    return (tile + t) * kb + (in > a.own_cost ? (in - a.own_cost) / step_cost : 0u);
}

// 16-byte asynchronous copy global -> shared that bypasses L1, and this thread's arrival on `bar` once all its copies so
// far have landed.
__device__ __forceinline__ void stream_copy16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void stream_copies_arrive(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];" ::"r"(bar) : "memory");
}

// Whether the first step of some tile is in the range.
__device__ __forceinline__ bool stream_owns(const StreamArgs& a, unsigned u_begin, unsigned u_end) {
    return (u_begin + a.kb - 1) / a.kb < (u_end + a.kb - 1) / a.kb;
}

// The bounded wait for a tile's flag, one lane per warp (the one that issues the warp's reductions).
__device__ __forceinline__ bool stream_tile_ready(const uint32_t* flag, uint32_t epoch, int lane, volatile int* abort_flag) {
    bool ok = true;
    if (lane == 0) {
        const long long t0 = clock64();
        for (;;) {
            uint32_t seen;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(flag) : "memory");
            if (seen == epoch) break;
            if (*abort_flag || clock64() - t0 > limb::WAIT_CYCLES) {
                *abort_flag = 1;
                ok = false;
                break;
            }
            __nanosleep(40);
        }
        asm volatile("fence.proxy.async;" ::: "memory");
    }
    return __all_sync(0xffffffffu, ok);
}

// COLS = 16 for up to 16 tokens, else 32: the width of the token planes and of the accumulators.  With half the columns the MMAs
// take half the time, which the conversion of a step otherwise waits for: llama7b decode (7 tokens) 202 -> 188 us.  (As a
// value of the launch instead of a template's it cost the 32-token layer 2 %.)
// FEATURES = 32 where the device has room for a CTA per step even of such tiles (launch_stream), else BW: a CTA's first planes wait for
// all of its words, and its end for its own sums, and a quarter of either is there sooner; the MMAs have a quarter of their rows
// in use, which costs nothing.  With so few steps latency is all there is, so the rest is cut short too: the first rows are found
// before the wait for the kernel before this one, Z <- C goes through registers, and three warps a party drain.  From that wait
// to the end, 16 tokens x 256 deep x 96: 7.8 -> 6.5 us.  A layer of 256 x 96, 32 tokens: 29.9 -> 21.9 us; 16 tokens: 22.3 to 22.9 -> 19.6 to
// 21.9, which is what the host's calls take; of 448 x 320, 32 tokens: 31.2 -> 28.8.
template <int COLS, int FEATURES>
__global__ void __launch_bounds__(limb_stream::THREADS, 1)
combine_stream_kernel(const __grid_constant__ StreamArgs a, const __grid_constant__ LimbMaps maps,
                      const __grid_constant__ BlockIds held) {
    using namespace limb_stream;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t raw_full[RAW_SLOTS], raw_empty[RAW_SLOTS];
    __shared__ __align__(8) uint64_t planes_full, own_empty[2], shared_empty;     // own: B_0 / B_1; shared: F, E, V_i
    __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2];
    __shared__ __align__(8) uint64_t own_landed, own_stored;                      // C of a tile of this CTA's: in, and out again
    __shared__ uint32_t tmem_slot, ticket, epoch;
    __shared__ int abort_flag;

    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
    uint8_t* sB = smem;                                   // planes of B_0, B_1, F
    uint8_t* sV = sB + 3 * W_SET_BYTES;                   // planes of V_0, V_1, E
    uint8_t* sRaw = sV + 3 * T_SET_BYTES;
    uint8_t* sOut = sRaw + RAW_SLOTS * RAW_SLOT_BYTES;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 32) {
        const u64 word = a.sync ? atomicAdd(reinterpret_cast<u64*>(a.sync), 1ull) : blockIdx.x;
        ticket = (uint32_t)word;
        epoch = (uint32_t)(word >> 32) + 1;
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < RAW_SLOTS; ++s) {
            ptx::mbar_init(ptx::smem_u32(&raw_full[s]), 64);                // every producer lane
            ptx::mbar_init(ptx::smem_u32(&raw_empty[s]), GROUP_WARPS);
        }
        ptx::mbar_init(ptx::smem_u32(&planes_full), CONV_WARPS + TOK_WARPS);
        ptx::mbar_init(ptx::smem_u32(&shared_empty), 1);
        for (int p = 0; p < 2; ++p) {
            ptx::mbar_init(ptx::smem_u32(&own_empty[p]), 1);
            ptx::mbar_init(ptx::smem_u32(&acc_full[p]), 1);
            ptx::mbar_init(ptx::smem_u32(&acc_empty[p]), EPI_WARPS);
        }
        ptx::mbar_init(ptx::smem_u32(&own_landed), 1);
        ptx::mbar_init(ptx::smem_u32(&own_stored), 1);
        abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if (warp == MMA_WARP) {
        ptx::tmem_alloc(ptx::smem_u32(&tmem_slot), 2 * ACC_COLS);
        ptx::tmem_relinquish();
    }
    ptx::fence_before_sync();
    __syncthreads();
    ptx::fence_after_sync();
    const uint32_t tmem_base = tmem_slot;
    // A ticket beyond the launch means that the words are not what the launches before it left: nothing is touched then.
    const bool valid = ticket < gridDim.x;
    if (!valid && threadIdx.x == 0) abort_flag = 1;
    const unsigned cta = valid ? ticket : 0u, u_begin = stream_cut(a, cta), u_end = valid ? stream_cut(a, cta + 1) : u_begin;
    constexpr bool SMALL = FEATURES < BW;
    const bool raw_warp = warp >= RAW_WARP0 && warp < RAW_WARP0 + 2;
    // the list of blocks may be the work of the kernel before this one
    if (!SMALL || !raw_warp || a.ids) pdl_wait();

    // A party's sums of a segment have arrived, and its part of Z may be added to.
    auto arrived = [&](const StreamSegment& sg, int party, uint32_t seg_phase) {
        bool ok = true;
        if (a.sync) ok = stream_tile_ready(a.sync + SYNC_WORDS + sg.tile, epoch, lane, &abort_flag);
        return ok && limb_wait_warp(ptx::smem_u32(&acc_full[party]), seg_phase, &abort_flag);
    };
    // ---------------- epilogue of a segment: lane = output feature, registers = tokens ----------------
    // Result rows go through shared memory, OUT_TOKENS of them at a time, and one tensor reduction adds them into Z.  (A bulk reduction
    // per row: 7400 cycles for 32 tokens.)
    auto drain_round = [&](int party, uint32_t acc, int col0, int row0, int t0, u64* stage, bool reused) {
        uint32_t d[PLANES][OUT_TOKENS];
#pragma unroll
        for (int s = 0; s < PLANES; ++s) ptx::tmem_ld4(acc + COLS * s + t0, d[s]);
        ptx::tmem_wait_ld();
        if (lane == 0 && reused) ptx::bulk_wait_group_read0();           // the last reduction has read its rows
        __syncwarp();
#pragma unroll
        for (int j = 0; j < OUT_TOKENS; ++j)
            stage[j * 32 + lane] = limb_recombine(d[0][j], d[1][j], d[2][j], d[3][j], d[4][j], d[5][j], d[6][j], d[7][j]);
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0 && col0 < a.N) {
            ptx::tensor_reduce_add(&maps.z[party], ptx::smem_u32(stage), col0, row0 + t0);
            ptx::bulk_commit_group();
        }
    };
    // Of a small tile, a CTA's only one: a worker, a warp that may read the first TMEM lanes, takes every SMALL_WORKERS-th round.  They stage
    // in the raw ring, which nothing uses any more.
    auto drain_small = [&](const StreamSegment& sg, int party, int worker) {
        const int tokens = min(a.M - sg.tm * BT, BT);
        ptx::fence_after_sync();
        for (int t0 = worker * OUT_TOKENS; t0 < tokens; t0 += SMALL_WORKERS * OUT_TOKENS)
            drain_round(party, tmem_base + party * ACC_COLS, sg.tn * FEATURES, sg.tm * BT, t0,
                        reinterpret_cast<u64*>(sRaw + (size_t)(party * (BT / OUT_TOKENS) + t0 / OUT_TOKENS) * OUT_BYTES), false);
    };

    if (raw_warp) {
        // ---------------- raw producer of one party: 16 lanes per row of a slot ----------------
        const int party = warp - RAW_WARP0, half = (lane >> 3) & 1, piece = lane & 15, rsub = lane >> 4;
        const uint32_t raw0 = ptx::smem_u32(sRaw) + party * 2 * RAW_ARRAY_BYTES + lane * 16;
        const u64* __restrict__ W0 = party ? a.W0[1] : a.W0[0];
        const u64* __restrict__ Bi = party ? a.B[1] : a.B[0];
        int slot = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (unsigned u = u_begin; u < u_end && ok;) {
            const StreamSegment sg = stream_segment(a, u, u_end);
            u += sg.count;
            const int quarters = stream_quarters<FEATURES>(a, sg.tn);
            // Sixteen rows aligned to 16 lie in one block (block sizes are multiples of 16), so they are `ldw` apart in W:
            // lane h of a warp's first eight knows where rows 16h .. 16h+15 of the tile begin
            const u64* w_row16 = W0;
            {
                const int row = sg.tn * FEATURES + (lane & 7) * 16;
                if (row < a.N) {
                    if (!a.gather || a.down) {
                        w_row16 = W0 + (size_t)row * a.ldw;
                    } else {
                        const int grp = (row >= a.n) + (row >= 2 * a.n), j = row - grp * a.n, blk = j / a.bs;
                        w_row16 = (grp == 0 ? W0 : grp == 1 ? (party ? a.W1[1] : a.W1[0]) : (party ? a.W2[1] : a.W2[0])) +
                                  (size_t)(block_id(a.ids, held, blk) * a.bs + (j - blk * a.bs)) * a.ldw;
                    }
                }
            }
            if (SMALL) pdl_wait();
            for (int it = 0; it < sg.count && ok; ++it) {
                const int k = (sg.step + it) * KC + 2 * piece;
                const bool kv = k < a.K;
                int col = k;                                      // this lane's column of W
                if (a.down && a.gather && kv) {
                    const int blk = ((sg.step + it) * KC + 16 * half) / a.bs;
                    col = block_id(a.ids, held, blk) * a.bs + (k - blk * a.bs);
                }
                for (int q = 0; q < quarters; ++q) {
                    const int row0 = sg.tn * FEATURES + q * QROWS + rsub;
                    const int rows = kv ? a.N - row0 : 0;                          // this lane's rows: row0 + 2i, 2i < rows
                    const u64* right = Bi + (size_t)row0 * a.K + k;
                    const u64* left[2];                                            // rows 0-15 and 16-31 of the slot
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        left[h] = reinterpret_cast<const u64*>(
                                      __shfl_sync(0xffffffffu, (unsigned long long)w_row16, 2 * q + h)) +
                                  (size_t)rsub * a.ldw + col;
                    const size_t left_step = 2 * (size_t)a.ldw, right_step = 2 * (size_t)a.K;
                    ok = limb_wait(ptx::smem_u32(&raw_empty[slot]), phase ^ 1u, &abort_flag);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    const uint32_t dst = raw0 + slot * RAW_SLOT_BYTES;
#pragma unroll
                    for (int i = 0; i < QROWS / 2; ++i) {
                        if (2 * i < rows) {
                            stream_copy16(dst + i * 512, left[i / 8] + (i % 8) * left_step);
                            stream_copy16(dst + RAW_ARRAY_BYTES + i * 512, right + i * right_step);
                        }
                    }
                    stream_copies_arrive(ptx::smem_u32(&raw_full[slot]));
                    if (++slot == RAW_SLOTS) { slot = 0; phase ^= 1u; }
                }
            }
        }
        if (SMALL) pdl_wait();
        asm volatile("cp.async.wait_all;" ::: "memory");          // no copy outlives the CTA, whatever ended the loop
    } else if (warp < CONV_WARPS) {
        // ---------------- converters ----------------
        const int group = warp / GROUP_WARPS, c = lane & 7;
        // this lane's row of a slot, and of it the words 2c, 2c+1, 16+2c, 17+2c.  Lanes c >= 4 take the row four further,
        // which keeps the plane stores free of bank conflicts.
        const int r = 4 * (2 * ((warp & 7) >> 1) + ((warp & 1) ^ (c >> 2))) + (lane >> 3);
        const uint8_t* raw_lane = sRaw + r * (KC * 8) + c * 16;
        const int cell = (r >> 3) * 256 + (c >> 2) * 128 + (r & 7) * 16 + (c & 3) * 4;
        int slot = 0;
        uint32_t phase = 0, unit_phase = 0;
        bool ok = true, planes_free = !a.sync || !stream_owns(a, u_begin, u_end) || SMALL;
        for (unsigned u = u_begin; u < u_end && ok;) {
            const StreamSegment sg = stream_segment(a, u, u_end);
            u += sg.count;
            const int quarters = stream_quarters<FEATURES>(a, sg.tn);
            for (int it = 0; it < sg.count && ok; ++it) {
                const int k0 = (sg.step + it) * KC;
                const bool kv[2] = {k0 + 2 * c < a.K, k0 + 16 + 2 * c < a.K};
                bool first = true;
                for (int q = 0; q < quarters; ++q) {
                    const int my_slot = slot;
                    const uint32_t my_phase = phase;
                    if (++slot == RAW_SLOTS) { slot = 0; phase ^= 1u; }
                    if (q % CONV_GROUPS != group) continue;
                    ok = limb_wait(ptx::smem_u32(&raw_full[my_slot]), my_phase, &abort_flag);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    const uint8_t* raw = raw_lane + my_slot * RAW_SLOT_BYTES;
                    u64 f[2][4], b[2][4];                            // per party: W_i, then the message F_i; B_i
#pragma unroll
                    for (int p = 0; p < 2; ++p)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const ulonglong2 w =
                                *reinterpret_cast<const ulonglong2*>(raw + 2 * p * RAW_ARRAY_BYTES + h * 128);
                            const ulonglong2 v =
                                *reinterpret_cast<const ulonglong2*>(raw + (2 * p + 1) * RAW_ARRAY_BYTES + h * 128);
                            f[p][2 * h] = w.x;
                            f[p][2 * h + 1] = w.y;
                            b[p][2 * h] = v.x;
                            b[p][2 * h + 1] = v.y;
                        }
                    __syncwarp();                                    // the slot has been read
                    if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&raw_empty[my_slot]));
#pragma unroll
                    for (int p = 0; p < 2; ++p)
#pragma unroll
                        for (int e = 0; e < 4; ++e) f[p][e] -= b[p][e];
                    const int row = sg.tn * FEATURES + q * QROWS + r;
                    const bool live = row < a.N;
                    if (a.blk_label && live) {                       // rows / columns outside every component stay closed
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            if (a.down ? (kv[h] && a.blk_label[(k0 + 16 * h) / a.bs] < 0)
                                       : a.blk_label[(row % a.n) / a.bs] < 0)
#pragma unroll
                                for (int p = 0; p < 2; ++p) f[p][2 * h] = f[p][2 * h + 1] = 0ull;
                    }
                    if (live && sg.tm == 0) {                        // the messages
                        const size_t at = (size_t)row * a.K + k0 + 2 * c;
#pragma unroll
                        for (int p = 0; p < 2; ++p) {
                            if (kv[0]) __stcs(reinterpret_cast<ulonglong2*>(a.F[p] + at), make_ulonglong2(f[p][0], f[p][1]));
                            if (kv[1]) __stcs(reinterpret_cast<ulonglong2*>(a.F[p] + at + 16), make_ulonglong2(f[p][2], f[p][3]));
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) f[0][e] += f[1][e];  // the exchange
                    uint8_t* to = sB + q * (QROWS / 8) * 256 + cell;
                    if (!planes_free) ok = limb_wait(ptx::smem_u32(&own_stored), 0, &abort_flag);
                    planes_free = true;
                    // a step's first planes: the MMAs of the step before must have read the old ones
                    if (first) ok = ok && limb_wait(ptx::smem_u32(&own_empty[0]), unit_phase ^ 1u, &abort_flag);
                    limb_emit4(to, W_PLANE_BYTES, b[0]);
                    if (first) ok = ok && limb_wait(ptx::smem_u32(&own_empty[1]), unit_phase ^ 1u, &abort_flag);
                    limb_emit4(to + W_SET_BYTES, W_PLANE_BYTES, b[1]);
                    if (first) ok = ok && limb_wait(ptx::smem_u32(&shared_empty), unit_phase ^ 1u, &abort_flag);
                    limb_emit4(to + 2 * W_SET_BYTES, W_PLANE_BYTES, f[0]);
                    first = false;
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                }
                // a ragged tile may leave a group without a slot: it must not arrive for a step before the last one is over
                if (ok && first) ok = __all_sync(0xffffffffu, limb_wait(ptx::smem_u32(&shared_empty), unit_phase ^ 1u, &abort_flag));
                if (!ok) break;
                ptx::fence_proxy_async_smem();                           // the planes are read by the tensor cores
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&planes_full));
                unit_phase ^= 1u;
            }
        }
        if (SMALL && ok && u_begin < u_end && (warp & 3) == 0) {         // two of three rounds of the sums are these warps'
            const StreamSegment sg = stream_segment(a, u_begin, u_end);
            const int party = warp >> 3, worker = 1 + (warp >> 2 & 1);
            if (worker * OUT_TOKENS < min(a.M - sg.tm * BT, BT) && arrived(sg, party, 0)) {
                drain_small(sg, party, worker);
                if (lane == 0) ptx::bulk_wait_group0();
            }
        }
    } else if (warp < MMA_WARP) {
        // ---------------- token side: the converters' cells, straight from L2 ----------------
        const int c = lane & 7, r = (4 * (warp - TOK_WARP0) ^ (c >= 4 ? 4 : 0)) + (lane >> 3);
        uint8_t* to = sV + (r >> 3) * 256 + (c >> 2) * 128 + (r & 7) * 16 + (c & 3) * 4;
        const int party = (warp - TOK_WARP0) / EPI_WARPS;
        u64* out = reinterpret_cast<u64*>(sOut + (size_t)(warp - TOK_WARP0) * OUT_BYTES);
        uint32_t unit_phase = 0, seg_phase = 0;
        bool ok = true;
        for (unsigned u = u_begin; u < u_end && ok;) {
            const StreamSegment sg = stream_segment(a, u, u_end);
            u += sg.count;
            const int row = sg.tm * BT + r;
            const bool live = row < a.M, closed = live && a.row_label && a.row_label[row] < 0;
            for (int it = 0; it < sg.count; ++it) {
                const int k0 = (sg.step + it) * KC;
                u64 e[2][4], v[2][4];                            // X_i, then the message E_i; A_i, then V_i
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // indices past the operand's depth and entries off the support are zero in E and in A_i
                    const int k = k0 + 16 * h + 2 * c;
                    bool has = live && k < a.K;
                    if (has && a.tmask) has = a.tmask[(size_t)row * a.tmask_ld + (k0 + 16 * h) / a.bs] != 0;
                    const size_t at = (size_t)row * a.K + k;
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        ulonglong2 x = make_ulonglong2(0ull, 0ull), m = x;
                        if (has) {
                            m = __ldg(reinterpret_cast<const ulonglong2*>(a.A[p] + at));
                            x = __ldg(reinterpret_cast<const ulonglong2*>(a.X[p] + at));
                        }
                        e[p][2 * h] = x.x;
                        e[p][2 * h + 1] = x.y;
                        v[p][2 * h] = m.x;
                        v[p][2 * h + 1] = m.y;
                    }
                }
#pragma unroll
                for (int p = 0; p < 2; ++p) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) e[p][i] = closed ? 0ull : e[p][i] - v[p][i];
                    if (live && sg.tn == 0) {                    // the message
                        u64* out = a.E[p] + (size_t)row * a.K + k0 + 2 * c;
                        if (k0 + 2 * c < a.K) *reinterpret_cast<ulonglong2*>(out) = make_ulonglong2(e[p][0], e[p][1]);
                        if (k0 + 16 + 2 * c < a.K) *reinterpret_cast<ulonglong2*>(out + 16) = make_ulonglong2(e[p][2], e[p][3]);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    e[0][i] += e[1][i];                          // the exchange
                    v[1][i] += e[0][i];                          // V_1 = A_1 + E  (V_0 = A_0)
                }
                ok = limb_wait(ptx::smem_u32(&shared_empty), unit_phase ^ 1u, &abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (live) {                                      // planes of rows past the last token are never looked at
                    limb_emit4(to, COLS * KC, v[0]);
                    limb_emit4(to + T_SET_BYTES, COLS * KC, v[1]);
                    limb_emit4(to + 2 * T_SET_BYTES, COLS * KC, e[0]);
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&planes_full));
                unit_phase ^= 1u;
            }
            if (!ok) break;
            ok = arrived(sg, party, seg_phase);
            if (!ok) break;
            const int quarter = warp & 3;        // TMEM lanes this warp may read
            if (SMALL) {
                if (quarter == 0) drain_small(sg, party, 0);
            } else {
                // A CTA's last segment stages its rows in the raw ring, which nothing uses any more, so that no round waits for the copy
                // engine to have read the one before.  (With both kinds of tile in one function, rounds and place by its arguments, every
                // layer in tiles of 128 features took 0.4 to 1 % longer: 32 tokens, 2048 x 832 54.4 -> 55.0 us, 4096 x 1312 127.5 -> 128.3.)
                ptx::fence_after_sync();
                const int tokens = min(a.M - sg.tm * BT, BT);
                const uint32_t acc = tmem_base + party * ACC_COLS + ((uint32_t)(quarter * 32) << 16);
                const bool at_end = u >= u_end;
                u64* stage = at_end ? reinterpret_cast<u64*>(sRaw + (size_t)(warp - TOK_WARP0) * (BT / OUT_TOKENS) * OUT_BYTES) : out;
#pragma unroll 1
                for (int t0 = 0; t0 < tokens; t0 += OUT_TOKENS) {
                    drain_round(party, acc, sg.tn * BW + quarter * 32, sg.tm * BT, t0, stage, !at_end);
                    if (at_end) stage += OUT_TOKENS * 32;
                }
            }
            ptx::fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&acc_empty[party]));
            seg_phase ^= 1u;
        }
        if (lane == 0) ptx::bulk_wait_group0();
    } else if (warp == MMA_WARP) {
        // ---------------- MMA issuer: weight plane q against token planes 0..7-q ----------------
        if (lane == 0) {
            constexpr uint32_t IDESC = (2u << 4) | ((uint32_t)(BW >> 4) << 24);
            const uint32_t w_lo = limb_desc_lo(ptx::smem_u32(sB)), t_lo = limb_desc_lo(ptx::smem_u32(sV));
            auto product = [&](uint32_t d, int w_set, int t_set, uint32_t acc) {
                const uint32_t w = w_lo + ((w_set * W_SET_BYTES) >> 4), t = t_lo + ((t_set * T_SET_BYTES) >> 4);
#pragma unroll
                for (int q = 0; q < PLANES; ++q)
                    ptx::mma_i8(d + COLS * q, w + ((q * W_PLANE_BYTES) >> 4), LIMB_DESC_HI, t, LIMB_DESC_HI,
                                IDESC | ((uint32_t)((COLS * (PLANES - q)) >> 3) << 17), q == 0 ? acc : 1u);
            };
            if (a.sync && ticket + 1 == gridDim.x) {
                // The last ticket is taken: no tickets of the next epoch.  Nobody reads the word before the next launch, whose
                // CTAs begin when every CTA of this one has let them or has ended; this one does so behind the fence.
                atomicAdd(reinterpret_cast<u64*>(a.sync), ((u64)(epoch + 1 ? 1u : 2u) << 32) - gridDim.x);
                __threadfence();
            }
            uint32_t unit_phase = 0, seg_phase = 0;
            bool ok = true;
            for (unsigned u = u_begin; u < u_end && ok;) {
                const StreamSegment sg = stream_segment(a, u, u_end);
                u += sg.count;
                for (int it = 0; it < sg.count; ++it) {
                    ok = limb_wait(ptx::smem_u32(&planes_full), unit_phase, &abort_flag);
                    if (!ok) break;
                    unit_phase ^= 1u;
                    ptx::fence_after_sync();
                    const bool last = it + 1 == sg.count;
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        if (it == 0) {
                            ok = ok && limb_wait(ptx::smem_u32(&acc_empty[p]), seg_phase ^ 1u, &abort_flag);
                            if (!ok) break;
                            ptx::fence_after_sync();
                        }
                        product(tmem_base + p * ACC_COLS, p, 2, it > 0 ? 1u : 0u);       // E*B_i
                        ptx::mma_commit(ptx::smem_u32(&own_empty[p]));
                    }
                    if (!ok) break;
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        product(tmem_base + p * ACC_COLS, 2, p, 1u);                      // V_i*F
                        if (last) ptx::mma_commit(ptx::smem_u32(&acc_full[p]));
                    }
                    ptx::mma_commit(ptx::smem_u32(&shared_empty));
                }
                seg_phase ^= 1u;
            }
            // the main loop is over: the next kernel of the stream may be brought in beside the last drain
            pdl_launch_dependents();
        }
    } else if (a.sync && stream_owns(a, u_begin, u_end)) {
        // ---------------- Z <- C for the tiles whose first step is in this CTA's range ----------------
        // By the copy engine, a lane per token row, through the weight planes' place before the first of them is written; the
        // loads go out before the raw ones fill the queue.  (The token warps' own loads and stores, queued behind the raw
        // copies, held the first planes back by 10000 cycles.)  Then the flag.  Whoever adds to a tile waits for its flag
        // first: a CTA with the same or an earlier ticket sets it, and a CTA that has a ticket is running, so the wait ends
        // whatever else is on the device and in whatever order the CTAs were started.
        const unsigned last = (u_end + a.kb - 1) / a.kb;
        bool ok = true;
        uint32_t phase = 0;
        for (unsigned tile = (u_begin + a.kb - 1) / a.kb; tile < last && ok; ++tile, phase ^= 1u) {
            const int tn = (int)(tile / (unsigned)a.mt), tm = (int)tile - tn * a.mt;
            const int rows = min(a.M - tm * BT, BT), bytes = min(a.N - tn * FEATURES, FEATURES) * 8;
            const size_t at = (size_t)(tm * BT + lane) * a.N + tn * FEATURES;
            if (SMALL) {                         // through registers: 3 us until the flag is up, and 4 through shared memory
                const int across = bytes / 16, pieces = rows * across;
                const size_t corner = (size_t)(tm * BT) * a.N + tn * FEATURES;
                for (int i = lane; i < pieces; i += 4 * 32) {
                    ulonglong2 v[2][4];
                    unsigned piece[4];           // a tile's rows lie within 32 N words
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int k = i + 32 * j, r = k / across;
                        piece[j] = (unsigned)(r * a.N + 2 * (k - r * across));
                        if (k < pieces)
                            for (int p = 0; p < 2; ++p) v[p][j] = __ldcs(reinterpret_cast<const ulonglong2*>(a.C[p] + corner + piece[j]));
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (i + 32 * j < pieces)
                            for (int p = 0; p < 2; ++p) *reinterpret_cast<ulonglong2*>(a.Z[p] + corner + piece[j]) = v[p][j];
                }
                asm volatile("fence.proxy.async;" ::: "memory");
                __threadfence();
                __syncwarp();
                if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.sync + SYNC_WORDS + tile), "r"(epoch) : "memory");
                continue;
            }
            const uint32_t place = ptx::smem_u32(sB) + lane * (2 * BW * 8);
            if (lane == 0) ptx::mbar_expect_tx(ptx::smem_u32(&own_landed), 2 * rows * bytes);
            __syncwarp();
            if (lane < rows)
                for (int p = 0; p < 2; ++p)
                    ptx::bulk_g2s(place + p * (BW * 8), a.C[p] + at, bytes, ptx::smem_u32(&own_landed));
            ok = limb_wait_warp(ptx::smem_u32(&own_landed), phase, &abort_flag);
            if (!ok) break;
            if (lane < rows)
                for (int p = 0; p < 2; ++p) ptx::bulk_s2g(a.Z[p] + at, place + p * (BW * 8), bytes);
            ptx::bulk_commit_group();
            ptx::bulk_wait_group_read0();
            __syncwarp();
            if (lane == 0 && tile + 1 == last) ptx::mbar_arrive(ptx::smem_u32(&own_stored));
            ptx::bulk_wait_group0();
            asm volatile("fence.proxy.async;" ::: "memory");
            __threadfence();
            __syncwarp();
            if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.sync + SYNC_WORDS + tile), "r"(epoch) : "memory");
        }
    }

    __syncwarp();
    ptx::fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) {
        *a.error_flag = 1;
        if (a.error_host) *reinterpret_cast<volatile int*>(a.error_host) = 1;
        __threadfence_system();
    }
    if (warp == MMA_WARP) {
        ptx::fence_after_sync();
        ptx::tmem_dealloc(tmem_base, 2 * ACC_COLS);
    }
}

}  // namespace comet
