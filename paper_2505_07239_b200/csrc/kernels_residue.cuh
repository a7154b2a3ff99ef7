// K4, tensor-core variant through residues: Z_i = C_i + E*B_i + V_i*F (Eq. 1; V_i = A_i + i*E) with 18 byte products per ring
// product instead of the 36 of combine_limb_kernel (kernels_limb.cuh).  residue_planes.cuh has the number system.
//
// Three launches: the exchange kernel (limb_exchange_kernel<true>) writes 17 planes of signed bytes per operand word where the
// limb path writes 8; this kernel multiplies them, a plane against a plane, and leaves one byte per byte product and result word;
// residue_recombine_kernel makes the words.  Half the multiply-adds against 99 bytes of exchange traffic per word of both
// parties instead of 72, and a launch: large products gain (comet_api.cu has the rule, with both sides' times).
//
// A job is one byte product of one output tile, both parties: E is the same for both, and so is F, so a stage of 128 contraction
// indices is three operands for two products.  A CTA pair (cta_group::2) holds 256 rows of one side against up to 256 of the
// other, a party's 32-bit sums in 256 columns of tensor memory; which side of the product the 256 rows take is the host's choice.
// The pair's CTAs each fetch half of every operand.  Bytes fetched per multiply-add are those of the limb kernel; per cycle
// they are 48 a CTA, 13 TB/s of L2 over the device, and shared memory serves 112 of its 128 bytes a cycle.
//   warps 0-7   epilogue: sums -> residues -> memory (32 x 16 results of a chunk contiguous, so that a warp stores whole lines)
//   warp 8      fetches this CTA's halves
//   warp 9      issues the MMAs, in the first CTA of the pair
// Measured, [512, 2048] x [2048, 832] (N = 224: two jobs a pair): 50 us under ncu, 44 in the step, tensor pipe active 77 % of
// the active cycles at 1.68 GHz; a stage takes 923 cycles where its MMAs take 896, the rest is the fill (3400 cycles) and some
// 2500 to 3500 cycles between jobs (combine_limb_kernel: 80 us).  [512, 832] x [832, 2048]: 51 us (82).  512 x 8192 x 2048: 390 us,
// power-capped at about 1.5 GHz (some 900).
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "kernels_limb.cuh"
#include "pdl.cuh"
#include "residue_planes.cuh"

namespace comet {

namespace residue {
constexpr int BM = 256, MAX_BN = 256;                    // a CTA pair's tile; the N side in multiples of 32
constexpr int STAGE_BLOCKS = 2;                          // blocks of an operand to a stage
constexpr int SLOT_BYTES = STAGE_BLOCKS * 128 * KC;      // 16 KiB: one CTA's half of an operand's blocks
constexpr int STAGE_BYTES = 3 * SLOT_BYTES;              // an operand pair's two and the one both parties share
constexpr int STAGES = 4, LAG = 3;
// k-blocks of 32 a CTA of the exchange kernel takes.  Its work per block is three times that for limbs, so small CTAs even out
// better than they cost: [512 | 832, 2048] 58 us with as many blocks as fill the device once, 50 with 2, 54 with 4;
// [256 | 3328, 4096] 261, 230 and 239.
constexpr int EX_KB_PER_CTA = 2;
constexpr int EPI_WARPS = 8, THREADS = 32 * (EPI_WARPS + 2);
constexpr int ACC_COLS = 256;                            // of a party
constexpr size_t SMEM_BYTES = (size_t)STAGES * STAGE_BYTES + 1024;
}  // namespace residue

struct ResidueMaps {
    // planes as [set][block][8 rows][plane][128 words of 4 bytes]; sets 0, 1: V_i / B_i, 2: E / F.  Boxes: one CTA's half tile.
    CUtensorMap m_side, n_side;
};

struct ResidueArgs {
    uint8_t* T[2];           // the products' residues: [JOBS][m_groups][n_chunks][32 on the M side][16 on the N side]
    int m_groups, n_chunks;
    int swapped;             // 0: rows of Z (token rows) on the M side, 1: columns of Z
    int mt, nt, n_tile;      // tiles
    int k32;                 // instructions of depth 32 per operand pair
    int jobs;                // JOBS * mt * nt
    int* error_flag;
    int* error_host;
};

namespace ptx {
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// On a barrier of either CTA.  It says that tensor memory has been read, nothing about global memory: a release at cluster scope
// would wait for this thread's stores (1500 to 3000 cycles).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// A box into this CTA's shared memory; the bytes are counted on a barrier of either CTA of the pair.
__device__ __forceinline__ void tensor_g2s_pair(uint32_t dst, const CUtensorMap* map, int plane, int group, int block, int set,
                                                uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
                 ::"r"(dst), "l"(map), "r"(0), "r"(plane), "r"(group), "r"(block), "r"(set), "r"(bar) : "memory");
}
__device__ __forceinline__ void mma_s8_pair(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::2.kind::i8 [%0], da, db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(acc) : "memory");
}
// Arrival on the barrier at this address in both CTAs of the pair once the MMAs issued so far are done.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* d) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
                 "[%16];"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7]), "=r"(d[8]),
                   "=r"(d[9]), "=r"(d[10]), "=r"(d[11]), "=r"(d[12]), "=r"(d[13]), "=r"(d[14]), "=r"(d[15])
                 : "r"(taddr) : "memory");
}
}  // namespace ptx

struct ResidueJob { int job, tm, tn; };
__device__ __forceinline__ ResidueJob residue_job(const ResidueArgs& a, int w) {
    const int tiles = a.mt * a.nt;
    ResidueJob r;
    r.job = w / tiles;
    const int t = w - r.job * tiles;
    r.tn = t / a.mt;
    r.tm = t - r.tn * a.mt;
    return r;
}

__global__ void __cluster_dims__(2, 1, 1) __maxnreg__(144)
combine_residue_kernel(const __grid_constant__ ResidueArgs a, const __grid_constant__ ResidueMaps maps) {
    using namespace residue;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES];
    __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_rank();
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const int kb = (a.k32 + 2 * STAGE_BLOCKS - 1) / (2 * STAGE_BLOCKS);          // stages per operand pair

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&full_bar[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&empty_bar[s]), 1);
        }
        for (int p = 0; p < 2; ++p) {
            ptx::mbar_init(ptx::smem_u32(&acc_full[p]), 1);
            ptx::mbar_init(ptx::smem_u32(&acc_empty[p]), 2 * EPI_WARPS);      // of both CTAs
        }
        abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 0) {
        ptx::tmem_alloc_pair(ptx::smem_u32(&tmem_slot), 2 * ACC_COLS);
        ptx::tmem_relinquish_pair();
    }
    ptx::fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();                     // the peer's barriers are set up too
    ptx::fence_after_sync();
    const uint32_t tmem_base = tmem_slot;
    pdl_wait();

    if (warp == EPI_WARPS) {
        // ---------------- producer: this CTA's halves of the operands ----------------
        if (ptx::elect_one()) {
            const uint32_t s0 = ptx::smem_u32(smem), empty0 = ptx::smem_u32(&empty_bar[0]), full0 = ptx::smem_u32(&full_bar[0]);
            const uint32_t full_leader = ptx::map_to_rank(full0, 0);
            const uint32_t n_bytes = (uint32_t)(a.n_tile / 2 * KC * STAGE_BLOCKS);
            const int n_groups = a.n_tile / 16;
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int w = pair; w < a.jobs && ok; w += pairs) {
                const ResidueJob jb = residue_job(a, w);
                const int left = jb.job == MODULI ? PLANES - 1 : jb.job == MODULI + 1 ? 0 : jb.job;       // planes of the job
                const int right = jb.job == MODULI + 1 ? PLANES - 1 : jb.job == MODULI ? 0 : jb.job;
                const int m_plane = a.swapped ? right : left, n_plane = a.swapped ? left : right;
                const int m_group = (jb.tm * 2 + (int)rank) * 16, n_group = (jb.tn * 2 + (int)rank) * n_groups;
                for (int second = 0; second < 2; ++second) {
                    const uint32_t bytes = 2 * (second ? 2 * SLOT_BYTES + n_bytes : SLOT_BYTES + 2 * n_bytes);
                    // the middle one is the second of the side that has two
                    const CUtensorMap* middle = second ? &maps.m_side : &maps.n_side;
                    const int middle_plane = second ? m_plane : n_plane, middle_group = second ? m_group : n_group;
                    for (int block = 0; block < kb; ++block) {
                        ok = limb_wait(empty0 + 8 * stage, phase ^ 1u, &abort_flag);
                        if (!ok) break;
                        const uint32_t dst = s0 + stage * STAGE_BYTES, bar = full_leader + 8 * stage;
                        if (rank == 0) ptx::mbar_expect_tx(full0 + 8 * stage, bytes);
                        ptx::tensor_g2s_pair(dst, &maps.m_side, m_plane, m_group, STAGE_BLOCKS * block, second ? 0 : 2, bar);
                        ptx::tensor_g2s_pair(dst + SLOT_BYTES, middle, middle_plane, middle_group, STAGE_BLOCKS * block, second ? 1 : 0, bar);
                        ptx::tensor_g2s_pair(dst + 2 * SLOT_BYTES, &maps.n_side, n_plane, n_group, STAGE_BLOCKS * block, second ? 2 : 1, bar);
                        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                    }
                    if (!ok) break;
                }
            }
            if (!ok) {                       // gave up: the copies in flight land long before this ends
                const long long t0 = clock64();
                while (clock64() - t0 < 20000000ll) {}
            }
        }
    } else if (warp == EPI_WARPS + 1) {
        // ---------------- MMA issuer of the pair ----------------
        if (rank == 0 && ptx::elect_one()) {
            // s32 accumulate, s8 x s8, both K-major, M = 256
            const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(a.n_tile >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            constexpr uint32_t DESC_HI = (uint32_t)(GROUP_BYTES >> 4) | (1u << 14);
            const uint32_t full0 = ptx::smem_u32(&full_bar[0]), empty0 = ptx::smem_u32(&empty_bar[0]);
            const uint32_t acc_full0 = ptx::smem_u32(&acc_full[0]), acc_empty0 = ptx::smem_u32(&acc_empty[0]);
            const uint32_t d0 = limb_desc_lo(ptx::smem_u32(smem));
            constexpr uint32_t SLOT = SLOT_BYTES >> 4, STEP = (8 * 32) >> 4, M_BLOCK = (128 * KC) >> 4;
            const uint32_t n_block = (uint32_t)(a.n_tile / 2 * KC) >> 4;
            uint32_t acc_phase = 0, phase = 0;
            int stage = 0;
            bool ok = true;
            // the job's `it`-th stage of operands, in stage s: what it adds to a party's accumulator
            auto party = [&](int it, int s, int p) {
                const uint32_t at = d0 + s * (STAGE_BYTES >> 4);
                const bool second = it >= kb;
                const uint32_t m = at + (second && p ? SLOT : 0u), n = at + (second || p ? 2 * SLOT : SLOT);
                const int steps = a.k32 - 2 * STAGE_BLOCKS * (second ? it - kb : it);       // left of the operand pair
#pragma unroll
                for (int k = 0; k < 2 * STAGE_BLOCKS; ++k)
                    if (k < steps)
                        ptx::mma_s8_pair(tmem_base + p * ACC_COLS, m + (k / 2) * M_BLOCK + (k & 1) * STEP,
                                         n + (k / 2) * n_block + (k & 1) * STEP, DESC_HI, idesc, it + k > 0 ? 1u : 0u);
            };
            const int total = 2 * kb, head = total < LAG ? total : LAG, tail = total - head < LAG ? total - head : LAG;
            for (int w = pair; w < a.jobs && ok; w += pairs) {
                // At both ends of a job party 0 runs LAG stages ahead of party 1, so that a party's accumulators are drained
                // while the other's are added to.
                const int stage0 = stage;
                const uint32_t phase0 = phase;
                ok = limb_wait(acc_empty0, acc_phase ^ 1u, &abort_flag);
                ptx::fence_after_sync();
                for (int it = 0; it < head && ok; ++it) {
                    ok = limb_wait(full0 + 8 * stage, phase, &abort_flag);
                    if (!ok) break;
                    ptx::fence_after_sync();
                    party(it, stage, 0);
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                ok = ok && limb_wait(acc_empty0 + 8, acc_phase ^ 1u, &abort_flag);
                if (!ok) break;
                ptx::fence_after_sync();
                stage = stage0;
                phase = phase0;
                for (int it = 0; it < head; ++it) {
                    party(it, stage, 1);
                    ptx::mma_commit_pair(empty0 + 8 * stage);
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                for (int it = head; it < total - tail; ++it) {
                    ok = limb_wait(full0 + 8 * stage, phase, &abort_flag);
                    if (!ok) break;
                    ptx::fence_after_sync();
                    party(it, stage, 0);
                    party(it, stage, 1);
                    ptx::mma_commit_pair(empty0 + 8 * stage);
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                int s = stage;
                for (int it = total - tail; it < total && ok; ++it) {
                    ok = limb_wait(full0 + 8 * stage, phase, &abort_flag);
                    if (!ok) break;
                    ptx::fence_after_sync();
                    party(it, stage, 0);
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                ptx::mma_commit_pair(acc_full0);
                for (int it = total - tail; it < total; ++it) {
                    party(it, s, 1);
                    ptx::mma_commit_pair(empty0 + 8 * s);
                    if (++s == STAGES) s = 0;
                }
                ptx::mma_commit_pair(acc_full0 + 8);
                acc_phase ^= 1u;
            }
            if (!ok) {
                const long long t0 = clock64();
                while (clock64() - t0 < 20000000ll) {}
            }
        }
        // The main loop is over: the recombination may be brought in beside the last drain, and no sooner, because its waiting
        // CTAs take the registers that an exchange beside this kernel needs (the lanes that were not elected wait here).
        __syncwarp();
        pdl_launch_dependents();
    } else {
        // ---------------- epilogue: TMEM -> residues -> memory ----------------
        // rows 32 * quarter .. of tensor memory; chunks of 16 columns: part, part + 2, ..
        const int quarter = warp & 3, part = warp >> 2, chunks = a.n_tile / 16;
        const uint32_t empty_leader = ptx::map_to_rank(ptx::smem_u32(&acc_empty[0]), 0);
        const size_t plane = (size_t)a.m_groups * a.n_chunks * 512;
        uint32_t acc_phase = 0;
        bool ok = true;
        for (int w = pair; w < a.jobs && ok; w += pairs) {
            const ResidueJob jb = residue_job(a, w);
            // the residue of a 32-bit sum, as in residue_of, from its bytes: the top one is signed
            int m = 256;
#pragma unroll
            for (int i = 1; i < MODULI; ++i)
                if (jb.job == i) m = modulus(i);
            unsigned weights = 0, start = 0;
            for (int b = 0, x = 1; b < 4; ++b, x = x * 256 % m) {
                const int c = x > m / 2 ? x - m : x;
                weights |= (unsigned)(c & 255) << (8 * b);
                start = (unsigned)(-128 * c);
            }
            const int base = 12582912 / (256 * m) * (256 * m);
            start += 0x4B000000u + (unsigned)(base - 8388608);
            const float share = 1.0f / (float)m, zero = (float)(12582912 - base / m);
            const int m0 = jb.tm * (BM / 32) + (int)rank * 4 + quarter, n0 = jb.tn * chunks;
            for (int p = 0; p < 2 && ok; ++p) {
                ok = limb_wait_warp(ptx::smem_u32(&acc_full[p]), acc_phase, &abort_flag);
                if (!ok) break;
                ptx::fence_after_sync();
                uint8_t* out = (p ? a.T[1] : a.T[0]) + (size_t)jb.job * plane + ((size_t)m0 * a.n_chunks + n0) * 512 + lane * 16;
                const uint32_t from = tmem_base + ((uint32_t)(quarter * 32) << 16) + p * ACC_COLS;
                // A lane holds sixteen columns of its row per chunk, HELD of the warp's chunks at a time, so that the issuer, which
                // waits for the reads only, gets tensor memory back before most of them are reduced (after 1100 cycles, of which
                // the other party's MMAs hide 1300 to 1500).  Registers: an exchange CTA has to fit beside this one, 72 a thread.
                constexpr int MINE = MAX_BN / 32, HELD = 5;
                uint32_t d[HELD][16];
                auto read = [&](int k) {
                    if (part + 2 * k < chunks) ptx::tmem_ld16(from + (part + 2 * k) * 16, d[k % HELD]);
                };
                auto give_back = [&] {
                    ptx::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive_cluster(empty_leader + 8 * p);
                };
                auto reduce = [&](int k) {
                    const int c = part + 2 * k;
                    uint32_t* v = d[k % HELD];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const unsigned t = residue_dot(v[j] ^ 0x80000000u, weights, start);
                        v[j] = t - __float_as_uint(__fmaf_rn(__uint_as_float(t), share, zero)) * (unsigned)m;
                    }
                    if (m0 < a.m_groups && c < chunks && n0 + c < a.n_chunks)
                        *reinterpret_cast<uint4*>(out + (size_t)c * 512) =
                            make_uint4(residue_pack(v[0], v[1], v[2], v[3]), residue_pack(v[4], v[5], v[6], v[7]),
                                       residue_pack(v[8], v[9], v[10], v[11]), residue_pack(v[12], v[13], v[14], v[15]));
                };
#pragma unroll
                for (int k = 0; k < HELD; ++k) read(k);
                ptx::tmem_wait_ld();
                const bool more = part + 2 * HELD < chunks;
                if (!more) give_back();
#pragma unroll
                for (int k = 0; k < MINE - HELD; ++k) reduce(k);
                if (more) {
#pragma unroll
                    for (int k = HELD; k < MINE; ++k) read(k);
                    ptx::tmem_wait_ld();
                    give_back();
                }
#pragma unroll
                for (int k = MINE - HELD; k < MINE; ++k) {
                    if (part + 2 * k >= chunks) break;
                    reduce(k);
                }
            }
            acc_phase ^= 1u;
        }
    }

    __syncwarp();
    ptx::fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) {
        *a.error_flag = 1;
        *reinterpret_cast<volatile int*>(a.error_host) = 1;
        __threadfence_system();
    }
    ptx::cluster_sync();                     // the peer no longer reads this CTA's operands or arrives on its barriers
    if (warp == 0) {
        ptx::fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, 2 * ACC_COLS);
    }
}

// ---------------------------------------------------------------------------
// Z_i = C_i + S + 2^56 (the two cross products), S from its residues: S = sum_i t_i (M / m_i) - k M, k the nearest whole number
// to sum_i t_i / m_i, which 24 bits after the point tell (MAX_DEPTH keeps |S| below M / 2 by more than their error).
// 18 bytes in, mostly from L2, C in and Z out, 34 bytes a word: 512 x 832 both parties 9.0 us under ncu, 512 x 2048 15.8, which
// is 3.2 and 4.5 TB/s and so not memory's bound.  A scheduler issues in 49 and 61 % of its cycles; of its 9 and 13 warps 6.5 and
// 6.1 wait for loads, 3.5 and 4.9 for the integer multiply pipe: a thread has only its eighteen 4-byte loads and C in flight and
// nothing to do beside them.  (Two moduli at a time, with a third fewer integer instructions, took the same time.)
// ---------------------------------------------------------------------------
struct RecombineArgs {
    const uint8_t* T[2];     // see ResidueArgs
    const u64* C[2];
    u64* Z[2];
    int rows, cols;          // of Z, or of a band of its rows (SWAPPED: of its columns); cols a multiple of 16
    int m_groups, n_chunks;
    int ld;                  // SWAPPED: columns of Z
};

// Residues are signed bytes; as r + 128 they are not.
template <int I>
__device__ __forceinline__ void residue_gather(const uint8_t* t, size_t plane, unsigned* quotient, u64* sum) {
    if constexpr (I < residue::MODULI) {
        unsigned v = __ldcs(reinterpret_cast<const unsigned*>(t + I * plane));
        constexpr u64 cof = residue::cofactor(I);
        constexpr unsigned share = ((1u << 25) / (unsigned)residue::modulus(I) + 1) / 2;
        if (I > 0) v ^= 0x80808080u;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            unsigned r = v >> (8 * e) & 255u;
            if (I == 0) r = r * (unsigned)residue::inverse(0) & 255u;
            quotient[e] += r * share;
            sum[e] += (u64)r * cof;
        }
        residue_gather<I + 1>(t, plane, quotient, sum);
    }
}

// What the 128s of all residues but the first add.
__device__ constexpr u64 RESIDUE_BIAS = [] {
    u64 s = 0;
    for (int i = 1; i < residue::MODULI; ++i) s += 128ull * residue::cofactor(i);
    return s;
}();
__device__ constexpr unsigned RESIDUE_QUOTIENT_BIAS = [] {
    unsigned s = 0;
    for (int i = 1; i < residue::MODULI; ++i) s += 128u * (((1u << 25) / (unsigned)residue::modulus(i) + 1) / 2);
    return s;
}();

// A thread makes four words: of a row (SWAPPED = 0) or of a column of Z.
template <bool SWAPPED>
__global__ void __launch_bounds__(256)
residue_recombine_kernel(const __grid_constant__ RecombineArgs a) {
    pdl_wait();
    pdl_launch_dependents();
    const uint8_t* T = blockIdx.y ? a.T[1] : a.T[0];
    const u64* C = blockIdx.y ? a.C[1] : a.C[0];
    u64* Z = blockIdx.y ? a.Z[1] : a.Z[0];
    const size_t plane = (size_t)a.m_groups * a.n_chunks * 512;
    const unsigned pieces = (unsigned)a.m_groups * a.n_chunks * 128;
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < pieces; q += gridDim.x * blockDim.x) {
        // 32 on the M side x 16 on the N side make 128 pieces; a warp takes whole lines of Z
        const unsigned cell = q >> 7, mg = cell / (unsigned)a.n_chunks, nc = cell - mg * a.n_chunks;
        const unsigned m = SWAPPED ? q & 31 : q >> 2 & 31, n = SWAPPED ? q >> 5 & 3 : q & 3;
        const unsigned row = SWAPPED ? nc * 16 + n * 4 : mg * 32 + m, col = SWAPPED ? mg * 32 + m : nc * 16 + n * 4;
        if (row >= (unsigned)a.rows || col >= (unsigned)a.cols) continue;
        const size_t at = (size_t)row * (SWAPPED ? a.ld : a.cols) + col;
        u64 sum[4];
        unsigned quotient[4];
        if (!SWAPPED) {
            const ulonglong2 c0 = __ldcs(reinterpret_cast<const ulonglong2*>(C + at)), c1 = __ldcs(reinterpret_cast<const ulonglong2*>(C + at + 2));
            sum[0] = c0.x; sum[1] = c0.y; sum[2] = c1.x; sum[3] = c1.y;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) sum[e] = row + e < (unsigned)a.rows ? __ldcs(C + at + (size_t)e * a.ld) : 0ull;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) quotient[e] = (1u << 23) + (8u << 24) - RESIDUE_QUOTIENT_BIAS;
        const uint8_t* t = T + (size_t)cell * 512 + m * 16 + n * 4;
        residue_gather<0>(t, plane, quotient, sum);
        const unsigned x = __ldcs(reinterpret_cast<const unsigned*>(t + residue::MODULI * plane));
        const unsigned y = __ldcs(reinterpret_cast<const unsigned*>(t + (residue::MODULI + 1) * plane));
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            sum[e] -= RESIDUE_BIAS + (u64)(long long)((int)(quotient[e] >> 24) - 8) * residue::product();
            sum[e] += (u64)((x >> (8 * e)) + (y >> (8 * e))) << 56;
        }
        if (!SWAPPED) {
            *reinterpret_cast<ulonglong2*>(Z + at) = make_ulonglong2(sum[0], sum[1]);
            *reinterpret_cast<ulonglong2*>(Z + at + 2) = make_ulonglong2(sum[2], sum[3]);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (row + e < (unsigned)a.rows) Z[at + (size_t)e * a.ld] = sum[e];
        }
    }
}

}  // namespace comet
