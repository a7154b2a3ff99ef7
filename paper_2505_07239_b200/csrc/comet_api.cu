// C ABI of the library: context, host-side validation and kernel launches.
// Every argument is checked on the host before anything is enqueued; device
// code never traps.  See include/comet.h for the contract of each call.
#include "../../include/comet.h"

#include <chrono>
#include <cstdio>
#include <cstring>
#include <algorithm>
#include <atomic>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

#include "kernels_limb.cuh"
#include "kernels_mul.cuh"
#include "kernels_open.cuh"
#include "kernels_peak.cuh"
#include "kernels_residue.cuh"
#include "kernels_shuffle.cuh"
#include "kernels_simt.cuh"
#include "kernels_stream.cuh"

using comet::u64;

struct comet_ctx {
    comet_config cfg;
    cudaStream_t stream;
    int groups;                   // 1, 2 or 3 weight matrices stacked in the up-projection
    int64_t cap_T, cap_n;         // capacities
    int sm_count;
    u64* buf[2][COMET_NUM_TENSORS];   // where each tensor is read / written: the library's own buffer, or a bound one
    u64* own[2][COMET_NUM_TENSORS];   // the library's own buffers
    void* device_memory;              // one allocation each, made in comet_init and cut into every buffer below and above
    void* pinned_memory;
    int64_t cap_words[COMET_NUM_TENSORS];
    bool loaded[2][COMET_NUM_TENSORS];
    // limb path: operand planes, of limbs or of residues (left: V_i per party and E; right: B_i per party and F), and the device
    // error flag
    int path;                     // COMET_PATH_SIMT or COMET_PATH_LIMB
    struct Planes {
        uint8_t* at;              // three sets, one behind the other
        size_t bytes;             // room
    };
    Planes planes_left;           // V_0, V_1, E; shared by the two projections
    Planes planes_right_up;       // B_0, B_1, F of the up-projection
    Planes planes_right_dn;       // B'_0, B'_1, F' of the down-projection
    Planes residues;              // of one product: what the kernel on residues hands to the recombination
    int* d_error;                     // = d_count + 1
    // the weight side of the down-projection is opened on a second stream while the up-projection's
    // tensor-core kernel runs (it only needs the mask, W2 and B'_i)
    cudaStream_t side;
    cudaEvent_t ev_fork, ev_join;
    bool side_pending;                // ev_join not yet waited for on the main stream
    bool dn_right_ready;              // F'_i and the right planes of the down-projection are current
    bool dn_right_residue;            // ... and they are planes of residues
    bool dn_copy_ready;               // Y_i already holds C'_i (copied beside the up-projection)
    int32_t dn_copy_tokens;           // ... for this many token rows
    uint8_t* d_mask;
    // a block mask given in host memory is counted on the host and copied from a pinned staging slot of the
    // library's own, so that comet_set_mask need not wait for the device
    uint8_t* h_mask_stage;            // pinned: kMaskSlots x n_blocks bytes
    cudaEvent_t stage_done[4];        // recorded after the copy out of each slot
    bool stage_used[4];
    int stage_next;
    uint8_t* d_tmask;             // per-token mask over the active blocks, [cap_T, d_ff / block] capacity
    bool tmask_set;
    int32_t tmask_tokens;
    int64_t tmask_masked;         // non-zero entries of the hidden state under the token mask (neurons, not blocks)
    unsigned long long* h_masked; // pinned and mapped: token_plan_kernel's report
    unsigned long long plan_ticket;   // of its last launch
    uint32_t* d_plan_scratch;     // its working storage when that does not fit into shared memory
    unsigned long long* h_masked_dev;
    int32_t* d_row_label;         // component label per token row / per active block under the token mask
    int32_t* d_blk_label;
    int32_t n_components, live_rows, live_blocks;
    // one multiplication per component on the tensor-core path: component-sorted order and the tiles with work
    int32_t* d_row_map;
    int32_t* d_col_map;
    int32_t* d_kmap;
    comet::LimbGroupRow* d_group_up;
    comet::LimbGroupRow* d_group_dn;
    bool grouped;                 // the products under the current token mask run over the component rectangles only
    int32_t group_units_up, group_units_dn;   // k-block units per party of the two grouped launches
    int64_t component_pairs;      // sum over components of token rows x active blocks
    int32_t* d_ids;
    comet::BlockIds held;         // the ids of a mask the host held, when there are few enough blocks (ids_held)
    bool ids_held;
    uint32_t* d_stream_sync;      // StreamArgs::sync: epoch and tickets, a flag per tile of the streaming kernel
    size_t stream_sync_words;
    int32_t* d_count;             // {count, error flag of the bounded waits}
    int32_t* h_count;             // pinned and mapped: {count, error flag as the compaction kernel saw it, ticket,
                                  // error word written by a kernel whose bounded wait ran out}
    int32_t* h_count_dev;         // device-side address of h_count
    int top_priority;             // the device's highest stream / launch priority (numerically lowest)
    int32_t ticket;               // sequence number of the last compaction launch (echoed in h_count[2])
    bool mask_set;
    int32_t n_active, n_active_blocks;
    int32_t tokens;               // T fixed by the last load of X / A_UP / H
    bool up_done, down_done;
    int32_t up_tokens, down_tokens;
    comet_stats_t stats;
    int last_cuda_error;
    // per-phase timers: pairs of events recorded around each phase while profiling is on
    bool profiling;
    struct Pending { cudaEvent_t start, stop; int phase, launches; };
    std::vector<Pending>* pending;
    std::vector<cudaEvent_t>* free_events;
};

namespace {

#define COMET_CUDA(ctx, call)                                  \
    do {                                                       \
        cudaError_t err__ = (call);                            \
        if (err__ != cudaSuccess) {                            \
            (ctx)->last_cuda_error = (int)err__;               \
            return COMET_ERR_CUDA;                             \
        }                                                      \
    } while (0)

// Brackets the launches of one phase with two events when profiling is on.
struct PhaseTimer {
    comet_ctx* c;
    comet_ctx::Pending p;
    bool on;
    static cudaEvent_t take(comet_ctx* c) {
        if (!c->free_events->empty()) {
            cudaEvent_t e = c->free_events->back();
            c->free_events->pop_back();
            return e;
        }
        cudaEvent_t e = nullptr;
        cudaEventCreate(&e);
        return e;
    }
    PhaseTimer(comet_ctx* ctx, int phase, int launches) : c(ctx), on(ctx->profiling) {
        if (!on) return;
        p.phase = phase;
        p.launches = launches;
        p.start = take(c);
        p.stop = take(c);
        cudaEventRecord(p.start, c->stream);
    }
    ~PhaseTimer() {
        if (!on) return;
        cudaEventRecord(p.stop, c->stream);
        c->pending->push_back(p);
    }
};

inline int is_input(int id) { return (id >= COMET_X && id <= COMET_C_DN) || id == COMET_W3; }

// current shape of a tensor as stored; rows = cols = 0 when not defined yet
void tensor_shape(const comet_ctx* c, int id, int64_t T, int64_t* rows, int64_t* cols) {
    const int64_t d = c->cfg.d_model, D = c->cfg.d_ff, n = c->n_active, gn = (int64_t)c->groups * n;
    switch (id) {
        case COMET_X: case COMET_A_UP: case COMET_E_UP: case COMET_C_DN: case COMET_Y: *rows = T; *cols = d; break;
        case COMET_W1: case COMET_WG: case COMET_W3: *rows = D; *cols = d; break;
        case COMET_W2: *rows = d; *cols = D; break;
        case COMET_B_UP: case COMET_F_UP: *rows = gn; *cols = d; break;
        case COMET_C_UP: case COMET_Z_UP: *rows = T; *cols = gn; break;
        case COMET_H: case COMET_A_DN: case COMET_E_DN: *rows = T; *cols = n; break;
        case COMET_B_DN: case COMET_F_DN: *rows = d; *cols = n; break;
        default: *rows = 0; *cols = 0;
    }
}

int64_t tensor_capacity(const comet_ctx* c, int id) {
    const int64_t d = c->cfg.d_model, D = c->cfg.d_ff, T = c->cap_T, n = c->cap_n, gn = c->groups * n;
    switch (id) {
        case COMET_X: case COMET_A_UP: case COMET_E_UP: case COMET_C_DN: case COMET_Y: return T * d;
        case COMET_W1: return D * d;
        case COMET_WG: return c->groups >= 2 ? D * d : 0;
        case COMET_W3: return c->groups == 3 ? D * d : 0;
        case COMET_W2: return d * D;
        case COMET_B_UP: case COMET_F_UP: return gn * d;
        case COMET_C_UP: case COMET_Z_UP: return T * gn;
        case COMET_H: case COMET_A_DN: case COMET_E_DN: return T * n;
        case COMET_B_DN: case COMET_F_DN: return d * n;
        default: return 0;
    }
}

inline int ew_grid(const comet_ctx* c, int64_t items, int threads) {
    int64_t want = (items + threads - 1) / threads;
    int64_t cap = (int64_t)c->sm_count * 8;
    if (want < 1) want = 1;
    return (int)(want < cap ? want : cap);
}

cudaMemcpyKind copy_kind(int location, bool to_library) {
    if (location == COMET_DEVICE) return cudaMemcpyDeviceToDevice;
    return to_library ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost;
}

inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Launch of a kernel of the step's chain: programmatic stream serialisation (the kernel may begin while its
// predecessor on the stream is finishing; it calls pdl_wait() before it touches global memory) and, for the
// tensor-core kernels, the device's highest scheduling priority.
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                           const int* priority, Args&&... args) {
    cudaLaunchConfig_t lc;
    std::memset(&lc, 0, sizeof(lc));
    lc.gridDim = grid;
    lc.blockDim = block;
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.numAttrs = 1;
    if (priority) {
        attr[1].id = cudaLaunchAttributePriority;
        attr[1].val.priority = *priority;
        lc.numAttrs = 2;
    }
    lc.attrs = attr;
    return cudaLaunchKernelEx(&lc, kernel, std::forward<Args>(args)...);
}

// True once a kernel of this context gave up on a bounded wait (the word is written by the kernel itself, in
// mapped host memory, and never cleared: the context's results are not to be trusted from then on).
inline bool timed_out(const comet_ctx* c) {
    return *reinterpret_cast<volatile int32_t*>(c->h_count + 3) != 0 ||
           *reinterpret_cast<volatile int32_t*>(c->h_count + 1) != 0;
}

// One Pi_MatMul of the path: sizes and tensor ids.
struct Proj {
    int M, N, K;
    int idX, idA, idE, idB, idF, idC, idZ;
    bool down;
};

Proj proj_up(const comet_ctx* c, int tokens) {
    return Proj{tokens, c->groups * c->n_active, c->cfg.d_model, COMET_X, COMET_A_UP, COMET_E_UP, COMET_B_UP,
                COMET_F_UP, COMET_C_UP, COMET_Z_UP, false};
}
Proj proj_down(const comet_ctx* c, int tokens) {
    return Proj{tokens, c->cfg.d_model, c->n_active, COMET_H, COMET_A_DN, COMET_E_DN, COMET_B_DN, COMET_F_DN,
                COMET_C_DN, COMET_Y, true};
}

// An input may be bound to memory of the library's own: a layer's X to the result of the one before it, say.  The kernels of the
// tensor-core path write Z <- C in the launch that reads the operands, so an operand that lies on the result is moved to its own
// buffer for the length of the call.
struct OperandsOffResult {
    comet_ctx* c;
    const Proj& pr;
    int ids[7], count = 0;
    u64* bound[2][7];
    OperandsOffResult(comet_ctx* ctx, const Proj& proj) : c(ctx), pr(proj) {
        for (int id : {pr.idX, pr.idA, pr.idB, pr.idC}) ids[count++] = id;
        if (pr.down) ids[count++] = COMET_W2;
        else for (int id : {COMET_W1, COMET_WG, COMET_W3}) ids[count++] = id;
        for (int p = 0; p < 2; ++p)
            for (int k = 0; k < count; ++k) bound[p][k] = c->buf[p][ids[k]];
    }
    // Whether operand `id` of a party lies on a result buffer of either party; *bytes becomes its size.
    bool on(int party, int id, int result, size_t* bytes) const {
        if (c->buf[party][id] == c->own[party][id]) return false;
        int64_t rows, cols;
        tensor_shape(c, id, pr.M, &rows, &cols);
        *bytes = (size_t)(rows * cols) * sizeof(u64);
        const uintptr_t at = reinterpret_cast<uintptr_t>(c->buf[party][id]);
        for (int q = 0; q < 2; ++q) {
            const uintptr_t z = reinterpret_cast<uintptr_t>(c->own[q][result]);
            if (at < z + (uintptr_t)c->cap_words[result] * sizeof(u64) && z < at + *bytes) return true;
        }
        return false;
    }
    bool any_on(int result) const {
        for (int k = 0; k < count; ++k)
            if (on(ids[k], result)) return true;
        return false;
    }
    bool on(int id, int result) const {
        size_t bytes;
        return on(0, id, result, &bytes) || on(1, id, result, &bytes);
    }
    int move() {
        size_t bytes;
        for (int p = 0; p < 2; ++p)
            for (int k = 0; k < count; ++k) {
                const int id = ids[k];
                if (!on(p, id, pr.idZ, &bytes) || (id == pr.idC && c->buf[p][id] == c->own[p][pr.idZ])) continue;
                COMET_CUDA(c, cudaMemcpyAsync(c->own[p][id], c->buf[p][id], bytes, cudaMemcpyDeviceToDevice, c->stream));
                c->buf[p][id] = c->own[p][id];
            }
        return COMET_OK;
    }
    ~OperandsOffResult() {
        for (int p = 0; p < 2; ++p)
            for (int k = 0; k < count; ++k) c->buf[p][ids[k]] = bound[p][k];
    }
};

// The streaming kernel (one kernel per product, operand roles exchanged) serves layers with at most 32 token rows: its planes
// live in shared memory, so every further 32 rows convert the weights once more.  Up to 64 rows that still beats writing the
// planes to memory and reading them back where the weights are many (without a token mask, whose components only the other
// kernel separates).  Both products of a step, 48 rows, streaming / planes: 448 x 320 32.8 / 25.9 us, 1024 x 320 38.4 / 35.1, 1024 x 768 51.9 / 50.9,
// 2048 x 512 56.7 / 61.6, 2048 x 832 77.3 / 88.3, 4096 x 1312 207 / 249; 33 rows, 1024 x 768 52.1 / 49.5, 2048 x 512 56.7 / 60.6; 64 rows, 1536 x 512 51.6 / 51.2,
// 2048 x 512 59.6 / 62.8; 96 rows of 4096 x 1312 took 329 / 263.  Very small layers would gain too, in tiles of 32 features: 48 rows, 256 x 96
// 22.2 / 26.1; they are left to the planes.
constexpr int STREAM_TOKENS = 2 * comet::limb_stream::BT;
constexpr int64_t STREAM_WORDS = 3 << 19;          // of the layer's active weights, from which on 33..64 rows are streamed
bool few_tokens(const comet_ctx* c, int tokens) {
    if (tokens <= comet::limb_stream::BT) return true;
    return tokens <= STREAM_TOKENS && !c->tmask_set && (int64_t)(c->groups + 1) * c->cfg.d_model * c->n_active >= STREAM_WORDS;
}

cudaError_t tensor_map(CUtensorMap* map, CUtensorMapDataType type, int rank, void* base, const cuuint64_t* size, const cuuint64_t* pitch,
                       const cuuint32_t* box, const cuuint32_t* step, CUtensorMapSwizzle swizzle) {
    typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                               const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {                    // a driver function: the library does not link to the driver
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            fn = nullptr;
        }
        return reinterpret_cast<Encode>(fn);
    }();
    if (!encode) return cudaErrorSymbolNotFound;
    return encode(map, type, (cuuint32_t)rank, base, size, pitch, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                  CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? cudaSuccess : cudaErrorInvalidValue;
}

// Tensor map of a result matrix for the tensor-core kernel's reductions (see LimbMaps).
cudaError_t result_map(CUtensorMap* map, u64* z, int rows, int cols, int box_rows, int box_cols, CUtensorMapSwizzle swizzle) {
    const cuuint64_t size[2] = {(cuuint64_t)cols, (cuuint64_t)rows}, pitch[1] = {(cuuint64_t)cols * sizeof(u64)};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows}, step[2] = {1, 1};
    return tensor_map(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, z, size, pitch, box, step, swizzle);
}

// Features of a tile of the streaming kernel: 32 where the device has room for a CTA per step of such tiles.  Beyond that a CTA would
// have several such steps, and the MMAs of each take as long as those of a step of 128.
int stream_features(int M, int N, int K, int sm_count) {
    namespace ls = comet::limb_stream;
    return (long long)ceil_div(M, ls::BT) * ceil_div(N, ls::QROWS) * ceil_div(K, ls::KC) <= sm_count ? ls::QROWS : ls::BW;
}

// The streaming kernel.  Without `sync` words (they belong to one stream's order, so a call without a context has none) Z <- C
// is a launch of its own before it; the product's CTAs are set up while the copy runs.
int launch_stream(comet::StreamArgs& args, const comet::BlockIds& held, int sm_count, cudaStream_t stream,
                  const int* priority, cudaError_t* err) {
    namespace ls = comet::limb_stream;
    *err = cudaSuccess;
    args.mt = ceil_div(args.M, ls::BT);
    args.kb = ceil_div(args.K, ls::KC);
    const int features = stream_features(args.M, args.N, args.K, sm_count);
    const bool small = features < ls::BW;
    args.nt = ceil_div(args.N, features);
    const long long steps = (long long)args.mt * args.nt * args.kb;
    const unsigned grid = (unsigned)(steps < sm_count ? steps : sm_count);
    args.last_cost = ceil_div(args.N - (args.nt - 1) * features, ls::QROWS) + ls::STEP_SLOTS;
    args.own_cost = args.sync ? (unsigned)ceil_div(ls::OWN_SIXTEENTHS * (args.M < ls::BT ? args.M : ls::BT), 16) : 0u;
    const long long cost = (((long long)(ls::QUARTERS + ls::STEP_SLOTS) * (args.nt - 1) + args.last_cost) * args.kb +
                            (long long)args.own_cost * args.nt) * args.mt;
    if (cost > 0x7fffffffll) return COMET_ERR_SHAPE;                   // the kernel counts in 32 bits
    args.cta_cost = steps > sm_count ? (unsigned)(cost / grid) : 0u;
    args.cta_extra = (unsigned)(cost % grid);
    comet::LimbMaps maps;
    for (int p = 0; p < 2; ++p) {
        *err = result_map(&maps.z[p], args.Z[p], args.M, args.N, ls::OUT_TOKENS, 32, CU_TENSOR_MAP_SWIZZLE_NONE);
        if (*err != cudaSuccess) return COMET_ERR_CUDA;
    }
    if (!args.sync) {
        const long long pairs = (long long)args.M * args.N / 2, want = (pairs + 255) / 256, most = (long long)sm_count * 8;
        *err = launch_chained(comet::result_init_kernel, dim3((unsigned)(want < most ? want : most), 2), dim3(256), 0, stream,
                              nullptr, args.C[0], args.C[1], args.Z[0], args.Z[1], pairs);
        if (*err != cudaSuccess) return COMET_ERR_CUDA;
    }
    auto* const kernel = small ? (args.M <= 16 ? comet::combine_stream_kernel<16, ls::QROWS> : comet::combine_stream_kernel<32, ls::QROWS>)
                               : (args.M <= 16 ? comet::combine_stream_kernel<16, ls::BW> : comet::combine_stream_kernel<32, ls::BW>);
    *err = launch_chained(kernel, dim3(grid), dim3(ls::THREADS), ls::SMEM_BYTES, stream, priority, args, maps, held);
    return *err == cudaSuccess ? COMET_OK : COMET_ERR_CUDA;
}

// Tensor-core path with few token rows: the whole Pi_MatMul.
int stream_product(comet_ctx* c, const Proj& pr) {
    namespace ls = comet::limb_stream;
    comet::StreamArgs a;
    std::memset(&a, 0, sizeof(a));
    for (int p = 0; p < 2; ++p) {
        a.X[p] = c->buf[p][pr.idX];
        a.A[p] = c->buf[p][pr.idA];
        a.E[p] = c->buf[p][pr.idE];
        a.W0[p] = pr.down ? c->buf[p][COMET_W2] : (c->groups >= 2 ? c->buf[p][COMET_WG] : c->buf[p][COMET_W1]);
        a.W1[p] = c->buf[p][COMET_W1];
        a.W2[p] = c->buf[p][COMET_W3];
        a.B[p] = c->buf[p][pr.idB];
        a.F[p] = c->buf[p][pr.idF];
        a.Z[p] = c->buf[p][pr.idZ];
        a.C[p] = c->buf[p][pr.idC];
    }
    if (ls::SYNC_WORDS + (size_t)ceil_div(pr.M, ls::BT) * ceil_div(pr.N, ls::QROWS) > c->stream_sync_words) return COMET_ERR_SHAPE;
    a.sync = c->d_stream_sync;
    a.gather = 1;
    a.ids = c->ids_held ? nullptr : c->d_ids;
    a.n = c->n_active;
    a.bs = c->cfg.block;
    a.M = pr.M; a.N = pr.N; a.K = pr.K;
    a.ldw = pr.down ? c->cfg.d_ff : c->cfg.d_model;
    a.down = pr.down ? 1 : 0;
    if (c->tmask_set) {
        a.tmask = pr.down ? c->d_tmask : nullptr;
        a.tmask_ld = c->n_active_blocks;
        a.row_label = pr.down ? nullptr : c->d_row_label;
        a.blk_label = c->d_blk_label;
    }
    a.error_flag = c->d_error;
    a.error_host = c->h_count_dev + 3;
    cudaError_t err;
    {
        PhaseTimer timer(c, COMET_PHASE_COMBINE, 1);
        const int rc = launch_stream(a, c->held, c->sm_count, c->stream, &c->top_priority, &err);
        if (rc == COMET_ERR_CUDA) c->last_cuda_error = (int)err;
        if (rc != COMET_OK) return rc;
    }
    c->stats.kernel_launches += 1;
    c->stats.tensor_tile_macs = 2ll * 2 * a.mt * a.nt * a.kb * ls::KC * stream_features(a.M, a.N, a.K, c->sm_count) * ls::BT;
    c->stats.matmul_path = COMET_PATH_LIMB;
    c->stats.product_kernel = COMET_KERNEL_STREAM;
    return COMET_OK;
}

// Waits for a kernel's report: it is the last thing on the stream and reports through mapped memory, with a ticket.  Watching
// for the ticket for a short while is quicker than a stream synchronise; after that, synchronise as usual.
template <typename Arrived>
int wait_for_report(comet_ctx* c, Arrived report) {
    const auto t0 = std::chrono::steady_clock::now();
    bool arrived = false;
    while (!(arrived = report()))
        if (std::chrono::steady_clock::now() - t0 > std::chrono::microseconds(300)) break;
    if (!arrived) COMET_CUDA(c, cudaStreamSynchronize(c->stream));
    std::atomic_thread_fence(std::memory_order_acquire);
    return COMET_OK;
}

// Makes the main stream wait for the side stream's outstanding work (if any).
int join_side(comet_ctx* c) {
    if (c->side_pending) {
        COMET_CUDA(c, cudaStreamWaitEvent(c->stream, c->ev_join, 0));
        c->side_pending = false;
    }
    return COMET_OK;
}

// Bytes of one set of operand planes: of limbs (tiles of `tile` rows), of residues.
size_t limb_set(int rows, int K, int tile) {
    return (size_t)ceil_div(rows, tile) * ceil_div(K, comet::limb::KC) * tile * comet::limb::KC * comet::limb::PLANES;
}
size_t residue_set(int rows, int K) {
    return (size_t)ceil_div(rows, 8) * ceil_div(K, comet::residue::KC) * comet::residue::CELL_BYTES;
}

// Arguments of the exchange kernel for the left and / or right side of one product, and / or Z <- C.  Returns its CTAs.
int exchange_args(comet_ctx* c, const Proj& pr, bool residue, bool left, bool right, bool copy, comet::LimbExchangeArgs& a) {
    namespace lb = comet::limb;
    std::memset(&a, 0, sizeof(a));
    uint8_t* const lpl = c->planes_left.at;
    uint8_t* const rpl = (pr.down ? c->planes_right_dn : c->planes_right_up).at;
    const size_t lset = residue ? residue_set(pr.M, pr.K) : limb_set(pr.M, pr.K, lb::BM);
    const size_t rset = residue ? residue_set(pr.N, pr.K) : limb_set(pr.N, pr.K, lb::BN);
    for (int p = 0; p < 2; ++p) {
        a.X[p] = c->buf[p][pr.idX];
        a.A[p] = c->buf[p][pr.idA];
        a.E[p] = c->buf[p][pr.idE];
        a.Vpl[p] = lpl + p * lset;
        a.W0[p] = pr.down ? c->buf[p][COMET_W2] : (c->groups >= 2 ? c->buf[p][COMET_WG] : c->buf[p][COMET_W1]);
        a.W1[p] = c->buf[p][COMET_W1];
        a.W2[p] = c->buf[p][COMET_W3];
        a.B[p] = c->buf[p][pr.idB];
        a.F[p] = c->buf[p][pr.idF];
        a.Bpl[p] = rpl + p * rset;
        a.C[p] = c->buf[p][pr.idC];
        a.Z[p] = c->buf[p][pr.idZ];
    }
    a.Epl = lpl + 2 * lset;
    a.Fpl = rpl + 2 * rset;
    a.ids = c->ids_held ? nullptr : c->d_ids;
    a.n = c->n_active;
    a.bs = c->cfg.block;
    a.M = pr.M; a.N = pr.N; a.K = pr.K;
    a.ldw = pr.down ? c->cfg.d_ff : c->cfg.d_model;
    a.down = pr.down ? 1 : 0;
    if (c->tmask_set) {
        a.tmask = pr.down ? c->d_tmask : nullptr;
        a.tmask_ld = c->n_active_blocks;
        a.row_label = pr.down ? nullptr : c->d_row_label;
        a.blk_label = c->d_blk_label;
    }
    if (c->grouped) {                       // component-sorted planes
        a.row_map = c->d_row_map;
        a.col_map = pr.down ? nullptr : c->d_col_map;
        a.kmap = pr.down ? c->d_kmap : nullptr;
    }
    a.kblocks = ceil_div(pr.K, lb::KC);
    const int left_rows = left ? ceil_div(pr.M, lb::EX_ROWS) : 0, right_rows = right ? ceil_div(pr.N, lb::EX_ROWS) : 0;
    // enough CTAs to fill the device once, else as many k-blocks per CTA as spread the row set-up
    const long long fill = (long long)c->sm_count * 7;
    const long long per = (long long)(left_rows + right_rows) * a.kblocks / fill;
    a.kb_per_cta = residue ? comet::residue::EX_KB_PER_CTA : (int)(per < 1 ? 1 : per > lb::EX_MAX_KB_PER_CTA ? lb::EX_MAX_KB_PER_CTA : per);
    a.kchunks = ceil_div(a.kblocks, a.kb_per_cta);
    a.left_blocks = left_rows * a.kchunks;
    a.right_blocks = right_rows * a.kchunks;
    a.copy_pairs = copy ? (long long)pr.M * pr.N / 2 : 0;
    a.copy_blocks = copy ? 2 * ew_grid(c, a.copy_pairs, lb::EX_THREADS) : 0;
    return a.left_blocks + a.right_blocks + a.copy_blocks;
}

// Tensor-core path: messages, exchange and operand planes of one product, in one launch; `also`, if given, are the arguments
// of a second product's for the same launch.
int limb_exchange(comet_ctx* c, const Proj& pr, bool residue, bool left, bool right, bool copy, cudaStream_t stream,
                  const comet::LimbExchangeArgs* also = nullptr, int also_blocks = 0) {
    namespace lb = comet::limb;
    comet::LimbExchangeArgs a;
    const int blocks = exchange_args(c, pr, residue, left, right, copy, a);
    if (blocks + also_blocks == 0) return COMET_OK;
    // A CTA of one k-block uses one stage, and more of them fit on an SM: 500 tokens, 512 x 256 40.7 -> 39.7 us a layer, 156 tokens,
    // 2304 x 384 78.7 -> 77.0.
    const size_t stages = std::min(std::max(left || right ? a.kb_per_cta : 0, also_blocks ? also->kb_per_cta : 0), (int)lb::EX_STAGES);
    COMET_CUDA(c, launch_chained(residue ? comet::limb_exchange_kernel<true> : comet::limb_exchange_kernel<false>, dim3(blocks + also_blocks), dim3(lb::EX_THREADS),
                                 stages * lb::EX_STAGE_BYTES, stream, nullptr, a, also ? *also : a, blocks, c->held));
    c->stats.kernel_launches += 1;
    COMET_CUDA(c, cudaGetLastError());
    return COMET_OK;
}

// How the limb kernel's work is cut.  Equal ranges of all tiles' blocks (0) balance the blocks, but a range that crosses from one tile
// into the next drains two, 1.9 us each, where a block takes 0.7.  So where that is less a tile is cut into as many parts as keep
// its longest as short as the SMs allow, and no more.  Layers, ranges and parts: 128 tokens, 768 x 320 33.4 and 31.4 us; 500 tokens,
// 512 x 256 42.7 and 40.7; 156 tokens, 2304 x 384 80.3 and 78.7; 90 tokens, 1536 x 768 69.8 and 67.7; 203 tokens, QKV of 8 heads, where
// the down-projection is just on this side of the line, the same.
int limb_parts(int sm_count, int tiles, int tile_blocks) {
    constexpr int DRAIN_TENTHS = 27;             // a drain in tenths of a block
    const int64_t all = (int64_t)tiles * tile_blocks;
    if (tiles > sm_count || all <= sm_count) return 0;
    const int blocks = ceil_div(tile_blocks, sm_count / tiles);
    if ((int64_t)blocks * sm_count * 10 >= all * 10 + (int64_t)sm_count * DRAIN_TENTHS) return 0;
    return ceil_div(tile_blocks, blocks);
}

// Tensor-core path: the persistent stream-K kernel over both parties' tiles.
int limb_combine(comet_ctx* c, const Proj& pr) {
    namespace lb = comet::limb;
    const int kb = ceil_div(pr.K, lb::KC), mt = ceil_div(pr.M, lb::BM), nt = ceil_div(pr.N, lb::BN);
    uint8_t* const lpl = c->planes_left.at;
    uint8_t* const rpl = (pr.down ? c->planes_right_dn : c->planes_right_up).at;
    const size_t lset = limb_set(pr.M, pr.K, lb::BM), rset = limb_set(pr.N, pr.K, lb::BN);
    comet::LimbArgs a;
    for (int p = 0; p < 2; ++p) {
        a.Vpl[p] = lpl + p * lset;
        a.Bpl[p] = rpl + p * rset;
        a.Z[p] = c->buf[p][pr.idZ];
    }
    a.Epl = lpl + 2 * lset;
    a.Fpl = rpl + 2 * rset;
    a.M = pr.M; a.N = pr.N; a.mt = mt; a.nt = nt; a.kb = kb;
    a.parts = c->grouped ? 0 : limb_parts(c->sm_count, 2 * mt * nt, 2 * kb);
    a.error_flag = c->d_error;
    a.error_host = c->h_count_dev + 3;
    a.ldz = pr.N; a.bs = c->cfg.block; a.group_units = 0;
    a.groups = nullptr; a.row_map = nullptr; a.col_map = nullptr;
    a.row_label = nullptr; a.blk_label = nullptr; a.blocks = 1;
    if (c->grouped) {
        a.M = c->live_rows;
        a.mt = ceil_div(a.M, lb::BM);
        a.row_map = c->d_row_map;
        if (pr.down) {
            a.groups = c->d_group_dn;
            a.group_units = c->group_units_dn;
        } else {
            a.N = c->groups * c->live_blocks * c->cfg.block;
            a.nt = ceil_div(a.N, lb::BN);
            a.col_map = c->d_col_map;
            a.row_label = c->d_row_label;
            a.blk_label = c->d_blk_label;
            a.blocks = c->n_active_blocks;
            a.groups = c->d_group_up;
            a.group_units = c->group_units_up;
        }
    }
    const long long total_units = c->grouped ? 2ll * a.group_units : 2ll * mt * nt * 2 * kb;
    c->stats.tensor_tile_macs = total_units * lb::KC * lb::BM * lb::BN;
    const int grid = a.parts ? 2 * mt * nt * a.parts : (int)(total_units < c->sm_count ? total_units : c->sm_count);
    {
        PhaseTimer timer(c, COMET_PHASE_COMBINE, 1);
        // The persistent kernel needs a slot on every SM.  With the device's highest scheduling priority its CTAs
        // get the slots that free up before the memory-side CTAs of other contexts queued beside it do, so the
        // tensor cores do not wait behind work that could as well run under them.
        if (c->grouped) {
            COMET_CUDA(c, launch_chained(comet::combine_limb_grouped_kernel, dim3(grid), dim3(lb::THREADS), lb::SMEM_BYTES,
                                         c->stream, &c->top_priority, a));
        } else {
            comet::LimbMaps maps;
            for (int p = 0; p < 2; ++p)
                COMET_CUDA(c, result_map(&maps.z[p], a.Z[p], a.M, a.N, 32, lb::OUT_COLS, CU_TENSOR_MAP_SWIZZLE_128B));
            COMET_CUDA(c, launch_chained(comet::combine_limb_kernel, dim3(grid), dim3(lb::THREADS), lb::SMEM_BYTES, c->stream,
                                         &c->top_priority, a, maps));
        }
    }
    c->stats.kernel_launches += 1;
    c->stats.matmul_path = COMET_PATH_LIMB;
    c->stats.product_kernel = c->grouped ? COMET_KERNEL_GROUPED : COMET_KERNEL_LIMB;
    COMET_CUDA(c, cudaGetLastError());
    return COMET_OK;
}

// Words of the down-projection's weight side from which on it is opened apart from the up-projection's exchange, and whether fewer are for
// the multiply-adds of the up-projection's product: see comet_ffn_up.
constexpr int64_t EXCHANGE_APART = 1 << 18;
bool long_product(int64_t words, int64_t macs) { return words >= 1 << 16 && macs >= (words >= 1 << 17 ? 45000000 : 52000000); }

bool limb_fits(const comet_ctx* c, const Proj& pr) {
    namespace lb = comet::limb;
    return 3 * limb_set(pr.M, pr.K, lb::BM) <= c->planes_left.bytes &&
           3 * limb_set(pr.N, pr.K, lb::BN) <= (pr.down ? c->planes_right_dn : c->planes_right_up).bytes;
}

// Tiles of the kernel on residues for a product: which side of it the MMAs' 256 rows take, and how many of the other side their
// columns.  The jobs (JOBS per tile, all alike) are dealt to the CTA pairs in rounds.  A block of 64 takes the four MMAs'
// 2 * n_tile cycles, or 380 to issue them and to fetch its operands; a job 2000 more to fill and to drain.
struct ResidueTiles {
    int swapped, n_tile, mt, nt;
    int64_t cycles;
};
ResidueTiles residue_tiles(int sm_count, int M, int N, int K) {
    namespace rs = comet::residue;
    ResidueTiles best{};
    const int64_t blocks = 2 * ceil_div(K, rs::KC), pairs = sm_count / 2;
    for (int swapped = 0; swapped < 2; ++swapped)
        for (int n_tile = rs::MAX_BN; n_tile >= 32; n_tile -= 32) {
            const int mt = ceil_div(swapped ? N : M, rs::BM), nt = ceil_div(swapped ? M : N, n_tile);
            const int64_t rounds = ((int64_t)rs::JOBS * mt * nt + pairs - 1) / pairs;
            const int64_t cycles = rounds * (blocks * (n_tile > 190 ? 2 * n_tile : 380) + 2000);
            if (best.n_tile == 0 || cycles < best.cycles) best = ResidueTiles{swapped, n_tile, mt, nt, cycles};
        }
    return best;
}
// What the kernel on residues leaves for the recombination, of both parties: a byte per byte product and result word, 2.25 times
// both parties' Z.  It has RESIDUE_ROOM at most, or one band of 256 rows where that is more; a product that leaves more goes band
// by band over the M side, each band's recombination before the next one's product.  512 tokens fit up to 58 thousand columns.
constexpr size_t RESIDUE_ROOM = (size_t)1 << 30;
size_t residue_bytes(int m_rows, int n_rows) {
    return 2 * (size_t)comet::residue::JOBS * (ceil_div(m_rows, 32) * 32) * (size_t)(ceil_div(n_rows, 32) * 32);
}
size_t residue_room(int rows, int cols) {
    return std::min(residue_bytes(rows, cols),
                    std::max(RESIDUE_ROOM, residue_bytes(comet::residue::BM, std::max(rows, cols))));
}

// Whether a product is quicker through residues than through limbs.
// Either way's time in ns, exchange included, is a constant, a share per step of a CTA, per operand word and per result word,
// fitted to timings of 65 to 512 rows, 256 to 4096 columns and depths: 512 x 256 x 256 19 us through limbs, 31 through residues;
// 512 x 1024 x 1024 67 and 65; 512 x 2048 x 2048 235 and 197; 512 x 4096 x 4096 966 and 726; 256 x 4096 x 4096 546 and 516;
// 128 x 4096 x 4096 376 and 452.  Over 136 such products either time is at most 28 % too short (512 x 256 x 256) and 19 % too long.
// With the 5 % asked for, none of the 19 that go through residues is slower for it; of the 117 others three lose 5 % or more, the
// wide and shallow ones, whose time per result word through limbs is understated: 512 x 4096 columns x 512 deep 152 and 130 us,
// 384 x 4096 x 512 123 and 117, 256 x 2048 x 4096 278 and 264.
bool residues_pay(int sm_count, int M, int N, int K) {
    namespace lb = comet::limb;
    const int64_t operands = (int64_t)(M + N) * K, results = (int64_t)M * N;
    const int64_t steps = 4ll * ceil_div(M, lb::BM) * ceil_div(N, lb::BN) * ceil_div(K, lb::KC) / sm_count;
    const int64_t limbs = 8900 + steps * 825 + (operands * 86 + results * 50) / 10000;
    const int64_t residues = 16300 + residue_tiles(sm_count, M, N, K).cycles * 344 / 1000 + (operands * 202 + results * 169) / 10000;
    return residues * 21 < limbs * 20;
}

// Whether this product goes through residues.
bool through_residues(const comet_ctx* c, const Proj& pr) {
    return c->residues.bytes >= residue_room(pr.M, pr.N) && !c->grouped && pr.K <= comet::residue::MAX_DEPTH &&
           3 * residue_set(pr.M, pr.K) <= c->planes_left.bytes &&
           3 * residue_set(pr.N, pr.K) <= (pr.down ? c->planes_right_dn : c->planes_right_up).bytes &&
           residues_pay(c->sm_count, pr.M, pr.N, pr.K);
}

// Tensor map of one side's residue planes (ResidueMaps), `take` rows from row `first` (a multiple of 8) on, in boxes of `rows`.
cudaError_t residue_map(CUtensorMap* map, uint8_t* planes, int operand_rows, int first, int take, int K, int rows) {
    namespace rs = comet::residue;
    const cuuint64_t groups = ceil_div(operand_rows, 8), blocks = ceil_div(K, rs::KC);
    const cuuint64_t size[5] = {rs::GROUP_BYTES / 4, rs::PLANES, (cuuint64_t)ceil_div(take, 8), blocks, 3};
    const cuuint64_t pitch[4] = {rs::GROUP_BYTES, rs::CELL_BYTES, groups * rs::CELL_BYTES, blocks * groups * rs::CELL_BYTES};
    const cuuint32_t box[5] = {rs::GROUP_BYTES / 4, 1, (cuuint32_t)rows / 8, rs::STAGE_BLOCKS, 1}, step[5] = {1, 1, 1, 1, 1};
    return tensor_map(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 5, planes + (size_t)(first / 8) * rs::CELL_BYTES, size, pitch, box, step,
                      CU_TENSOR_MAP_SWIZZLE_NONE);
}

// Tensor-core path: both parties' product through residues, from the planes to Z.
int residue_combine(comet_ctx* c, const Proj& pr) {
    namespace rs = comet::residue;
    const ResidueTiles t = residue_tiles(c->sm_count, pr.M, pr.N, pr.K);
    const int m_rows = t.swapped ? pr.N : pr.M, n_rows = t.swapped ? pr.M : pr.N;
    const bool whole = residue_bytes(m_rows, n_rows) <= c->residues.bytes;
    const int fit = whole ? t.mt : (int)(c->residues.bytes / residue_bytes(rs::BM, n_rows));      // tile rows that the room holds
    const int bands = ceil_div(t.mt, fit), band_tiles = ceil_div(t.mt, bands);
    comet::ResidueArgs a;
    comet::RecombineArgs r;
    r.ld = pr.N;
    r.n_chunks = a.n_chunks = ceil_div(n_rows, 16);
    a.swapped = t.swapped;
    a.nt = t.nt; a.n_tile = t.n_tile;
    a.k32 = ceil_div(pr.K, 32);
    a.error_flag = c->d_error;
    a.error_host = c->h_count_dev + 3;
    uint8_t* const left = c->planes_left.at;
    uint8_t* const right = (pr.down ? c->planes_right_dn : c->planes_right_up).at;
    comet::ResidueMaps maps;
    COMET_CUDA(c, residue_map(&maps.n_side, t.swapped ? left : right, n_rows, 0, n_rows, pr.K, t.n_tile / 2));
    PhaseTimer timer(c, COMET_PHASE_COMBINE, 2 * ceil_div(t.mt, band_tiles));
    for (int tile = 0; tile < t.mt; tile += band_tiles) {
        const int first = tile * rs::BM, rows = std::min(m_rows - first, band_tiles * rs::BM);
        a.mt = ceil_div(rows, rs::BM);
        a.jobs = rs::JOBS * a.mt * t.nt;
        r.m_groups = a.m_groups = ceil_div(rows, 32);
        r.rows = t.swapped ? pr.M : rows;
        r.cols = t.swapped ? rows : pr.N;
        const size_t at = (size_t)first * (t.swapped ? 1 : pr.N);
        for (int p = 0; p < 2; ++p) {
            r.T[p] = a.T[p] = c->residues.at + p * (residue_bytes(rows, n_rows) / 2);
            r.C[p] = c->buf[p][pr.idC] + at;
            r.Z[p] = c->buf[p][pr.idZ] + at;
        }
        COMET_CUDA(c, residue_map(&maps.m_side, t.swapped ? right : left, m_rows, first, rows, pr.K, rs::BM / 2));
        // no more pairs than the rounds need: what is left serves the kernels beside this one
        const int most = c->sm_count / 2, pairs = ceil_div(a.jobs, ceil_div(a.jobs, most));
        COMET_CUDA(c, launch_chained(comet::combine_residue_kernel, dim3(2 * pairs), dim3(rs::THREADS), rs::SMEM_BYTES, c->stream,
                                     &c->top_priority, a, maps));
        COMET_CUDA(c, launch_chained(t.swapped ? comet::residue_recombine_kernel<true> : comet::residue_recombine_kernel<false>,
                                     dim3(ew_grid(c, (int64_t)a.m_groups * a.n_chunks * 128, 256), 2), dim3(256), 0, c->stream,
                                     nullptr, r));
        c->stats.kernel_launches += 2;
    }
    c->stats.tensor_tile_macs = 2ll * 2 * t.mt * rs::BM * t.nt * t.n_tile * a.k32 * 32;
    c->stats.matmul_path = COMET_PATH_LIMB;
    c->stats.product_kernel = COMET_KERNEL_RESIDUE;
    COMET_CUDA(c, cudaGetLastError());
    return COMET_OK;
}

int launch_combine(comet_ctx* c, int M, int N, int K, int idE, int idF, int idA, int idB, int idC, int idZ) {
    comet::CombineArgs a;
    for (int p = 0; p < 2; ++p) {
        a.E[p] = c->buf[p][idE];
        a.F[p] = c->buf[p][idF];
        a.A[p] = c->buf[p][idA];
        a.B[p] = c->buf[p][idB];
        a.C[p] = c->buf[p][idC];
        a.Z[p] = c->buf[p][idZ];
    }
    a.M = M; a.N = N; a.K = K;
    a.tmask = (idZ == COMET_Y && c->tmask_set) ? c->d_tmask : nullptr;
    a.tmask_ld = c->n_active_blocks;
    a.bs = c->cfg.block;
    dim3 grid((N + comet::simt::BN - 1) / comet::simt::BN, (M + comet::simt::BM - 1) / comet::simt::BM, 2);
    PhaseTimer timer(c, COMET_PHASE_COMBINE, 1);
    comet::combine_simt_kernel<<<grid, comet::simt::THREADS, 0, c->stream>>>(a);
    c->stats.kernel_launches += 1;
    c->stats.matmul_path = COMET_PATH_SIMT;
    c->stats.product_kernel = COMET_KERNEL_SIMT;
    COMET_CUDA(c, cudaGetLastError());
    return COMET_OK;
}

// The Merge step of Protocol 2 under a token mask: entries of the compact result outside the component blocks become zero.
// The grouped launch does that itself.
int somm_merge(comet_ctx* c, int tokens) {
    if (!c->tmask_set || c->grouped) return COMET_OK;
    const int cols = c->groups * c->n_active;
    const int64_t pairs = (int64_t)tokens * cols / 2;
    if (pairs == 0) return COMET_OK;
    comet::PartyOut Z;
    for (int p = 0; p < 2; ++p) Z.p[p] = c->buf[p][COMET_Z_UP];
    COMET_CUDA(c, launch_chained(comet::somm_merge_kernel, dim3(ew_grid(c, pairs, 256), 2), dim3(256), 0, c->stream,
                                 nullptr, Z, pairs, cols, (int)c->n_active, (int)c->cfg.block,
                                 (const int32_t*)c->d_row_label, (const int32_t*)c->d_blk_label));
    c->stats.kernel_launches += 1;
    COMET_CUDA(c, cudaGetLastError());
    return COMET_OK;
}

}  // namespace

extern "C" {

const char* comet_strerror(int code) {
    switch (code) {
        case COMET_OK: return "ok";
        case COMET_ERR_INVALID_ARG: return "invalid argument";
        case COMET_ERR_SHAPE: return "shape disagrees with the configuration or the current mask";
        case COMET_ERR_STATE: return "call out of order: a required input has not been loaded";
        case COMET_ERR_OOM: return "device memory allocation failed";
        case COMET_ERR_CUDA: return "a CUDA runtime call failed";
        case COMET_ERR_TIMEOUT: return "a bounded device-side wait ran out";
        case COMET_ERR_SCRATCH_LIMIT:
            return "problem exceeds the library's static scratch array (COMET_STATIC_SCRATCH_WORDS)";
        default: return "unknown error code";
    }
}

int comet_last_cuda_error(comet_ctx* ctx) { return ctx ? ctx->last_cuda_error : 0; }

int comet_init(const comet_config* cfg, void* cuda_stream, comet_ctx** out) {
    if (!cfg || !out) return COMET_ERR_INVALID_ARG;
    *out = nullptr;
    if (cfg->gated < 0 || cfg->gated > 2) return COMET_ERR_INVALID_ARG;
    if (cfg->matmul_path < COMET_PATH_AUTO || cfg->matmul_path > COMET_PATH_LIMB) return COMET_ERR_INVALID_ARG;
    if (cfg->device < 0) return COMET_ERR_INVALID_ARG;
    if (cfg->max_tokens < 1 || cfg->d_model < 16 || cfg->d_ff < 16 || cfg->block < 16) return COMET_ERR_SHAPE;
    if (cfg->d_model % 16 || cfg->block % 16 || cfg->d_ff % cfg->block) return COMET_ERR_SHAPE;
    if (cfg->frac_bits < 1 || cfg->frac_bits > 31) return COMET_ERR_SHAPE;
    if (cfg->max_active < 0 || cfg->max_active > cfg->d_ff || cfg->max_active % cfg->block) return COMET_ERR_SHAPE;

    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || cfg->device >= ndev) {
        cudaGetLastError();
        return COMET_ERR_CUDA;
    }
    comet_ctx* c = new (std::nothrow) comet_ctx;
    if (!c) return COMET_ERR_OOM;
    std::memset(c, 0, sizeof(*c));
    c->pending = new (std::nothrow) std::vector<comet_ctx::Pending>();
    c->free_events = new (std::nothrow) std::vector<cudaEvent_t>();
    if (!c->pending || !c->free_events) {
        delete c->pending;
        delete c->free_events;
        delete c;
        return COMET_ERR_OOM;
    }
    c->cfg = *cfg;
    c->stream = (cudaStream_t)cuda_stream;
    c->groups = cfg->gated + 1;
    c->cap_T = cfg->max_tokens;
    c->cap_n = cfg->max_active ? cfg->max_active : cfg->d_ff;
    if (cudaSetDevice(cfg->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, cfg->device) != cudaSuccess) {
        cudaGetLastError();
        delete c->pending;
        delete c->free_events;
        delete c;
        return COMET_ERR_CUDA;
    }
    {
        int least = 0, greatest = 0;
        if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess) cudaGetLastError();
        c->top_priority = greatest;
    }
    bool ok = true;
    // Every buffer is a piece of one allocation (and of one pinned allocation): an allocation costs about as much whatever
    // its size, and this many of them one by one took 9 of the 11 ms in which a context came up.
    constexpr int MAX_PIECES = 2 * COMET_NUM_TENSORS + 32;
    struct Pieces {                     // fixed in size: nothing here may throw
        void** where[MAX_PIECES];
        size_t bytes[MAX_PIECES];
        int count = 0;
    } device, pinned;
    auto reserve = [](Pieces& list, auto** where, size_t bytes) {
        list.where[list.count] = reinterpret_cast<void**>(where);
        list.bytes[list.count++] = bytes;
    };
    for (int id = 0; id < COMET_NUM_TENSORS; ++id) {
        c->cap_words[id] = tensor_capacity(c, id);
        for (int p = 0; p < 2; ++p)
            if (c->cap_words[id] > 0) reserve(device, &c->own[p][id], (size_t)c->cap_words[id] * sizeof(u64));
    }
    c->path = cfg->matmul_path == COMET_PATH_AUTO ? COMET_PATH_LIMB : cfg->matmul_path;
    int planes_piece = 0, planes_pieces = 0;
    size_t planes_of_limbs[3];
    if (c->path == COMET_PATH_LIMB) {
        namespace lb = comet::limb;
        const int d = cfg->d_model;
        const int64_t n = c->cap_n, gn = c->groups * n;
        const int T = (int)c->cap_T, deepest = d > n ? d : (int)n;
        // a context for few tokens only never builds planes in memory
        planes_piece = device.count;
        if (T > comet::limb_stream::BT) {
            // room for planes of residues where a product of the full size would go through them
            const int up_depth = std::min(d, comet::residue::MAX_DEPTH), dn_depth = std::min((int)n, comet::residue::MAX_DEPTH);
            const bool up = residues_pay(c->sm_count, T, (int)gn, up_depth), dn = residues_pay(c->sm_count, T, d, dn_depth);
            auto planes = [&](comet_ctx::Planes& p, size_t limbs, size_t residues) {
                p.bytes = 3 * std::max(limbs, residues);
                planes_of_limbs[planes_pieces++] = 3 * limbs;
                reserve(device, &p.at, p.bytes);
            };
            planes(c->planes_left, limb_set(T, deepest, lb::BM),
                   std::max(up ? residue_set(T, up_depth) : 0, dn ? residue_set(T, dn_depth) : 0));
            planes(c->planes_right_up, limb_set((int)gn, d, lb::BN), up ? residue_set((int)gn, up_depth) : 0);
            planes(c->planes_right_dn, limb_set(d, (int)n, lb::BN), dn ? residue_set(d, dn_depth) : 0);
            c->residues.bytes = std::max(up ? residue_room(T, (int)gn) : 0, dn ? residue_room(T, d) : 0);
            reserve(device, &c->residues.at, c->residues.bytes);
        }
        ok = ok && cudaFuncSetAttribute(comet::combine_limb_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)lb::SMEM_BYTES) == cudaSuccess;
        // the memory-side kernels may share an SM with a resident tensor-core CTA (which forces the largest
        // shared-memory carve-out), so they ask for the same carve-out
        for (auto* kernel : {comet::combine_stream_kernel<16, comet::limb_stream::BW>, comet::combine_stream_kernel<32, comet::limb_stream::BW>,
                             comet::combine_stream_kernel<16, comet::limb_stream::QROWS>, comet::combine_stream_kernel<32, comet::limb_stream::QROWS>})
            ok = ok && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)comet::limb_stream::SMEM_BYTES) == cudaSuccess;
        ok = ok && cudaFuncSetAttribute(comet::combine_limb_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                        (int)cudaSharedmemCarveoutMaxShared) == cudaSuccess;
        ok = ok && cudaFuncSetAttribute(comet::combine_limb_grouped_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)lb::SMEM_BYTES) == cudaSuccess;
        ok = ok && cudaFuncSetAttribute(comet::combine_limb_grouped_kernel,
                                        cudaFuncAttributePreferredSharedMemoryCarveout,
                                        (int)cudaSharedmemCarveoutMaxShared) == cudaSuccess;
        ok = ok && cudaFuncSetAttribute(comet::combine_residue_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)comet::residue::SMEM_BYTES) == cudaSuccess;
        for (auto* kernel : {comet::limb_exchange_kernel<false>, comet::limb_exchange_kernel<true>}) {
            ok = ok && cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                            (int)cudaSharedmemCarveoutMaxShared) == cudaSuccess;
            ok = ok && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)lb::EX_SMEM_BYTES) == cudaSuccess;
        }
        ok = ok && cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking) == cudaSuccess;
        ok = ok && cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming) == cudaSuccess;
        ok = ok && cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming) == cudaSuccess;
    }
    const int nb = cfg->d_ff / cfg->block;
    for (int k = 0; k < 4 && ok; ++k)
        ok = cudaEventCreateWithFlags(&c->stage_done[k], cudaEventDisableTiming) == cudaSuccess;
    const size_t row_tiles = ceil_div((int)c->cap_T, comet::limb::BM);
    reserve(device, &c->d_mask, (size_t)nb);
    reserve(device, &c->d_tmask, (size_t)nb * (size_t)c->cap_T);
    reserve(device, &c->d_row_map, (size_t)c->cap_T * sizeof(int32_t));
    reserve(device, &c->d_col_map, (size_t)c->groups * nb * sizeof(int32_t));
    reserve(device, &c->d_kmap, (size_t)nb * sizeof(int32_t));
    reserve(device, &c->d_plan_scratch, comet::token_plan_words(c->cap_T, nb, ceil_div(nb, 32), c->groups) * sizeof(uint32_t));
    reserve(device, &c->d_group_up, row_tiles * sizeof(comet::LimbGroupRow));
    reserve(device, &c->d_group_dn, row_tiles * sizeof(comet::LimbGroupRow));
    reserve(device, &c->d_row_label, (size_t)c->cap_T * sizeof(int32_t));
    reserve(device, &c->d_blk_label, (size_t)nb * sizeof(int32_t));
    reserve(device, &c->d_ids, (size_t)nb * sizeof(int32_t));
    reserve(device, &c->d_count, 2 * sizeof(int32_t));              // {count, error flag}
    {
        namespace ls = comet::limb_stream;
        const int64_t widest = c->groups * c->cap_n > cfg->d_model ? c->groups * c->cap_n : cfg->d_model;
        c->stream_sync_words = ls::SYNC_WORDS + (STREAM_TOKENS / ls::BT) * (size_t)((widest + ls::QROWS - 1) / ls::QROWS);
        reserve(device, &c->d_stream_sync, c->stream_sync_words * sizeof(uint32_t));
    }
    reserve(pinned, &c->h_masked, comet::PLAN_WORDS * sizeof(long long));
    reserve(pinned, &c->h_count, 4 * sizeof(int32_t));
    reserve(pinned, &c->h_mask_stage, (size_t)nb * 4);
    constexpr size_t ALIGN = 256;
    auto total = [](const Pieces& list) {
        size_t bytes = 0;
        for (int k = 0; k < list.count; ++k) bytes += (list.bytes[k] + ALIGN - 1) / ALIGN * ALIGN;
        return bytes;
    };
    auto hand_out = [](const Pieces& list, void* base) {
        uint8_t* at = static_cast<uint8_t*>(base);
        for (int k = 0; k < list.count; ++k) {
            *list.where[k] = at;
            at += (list.bytes[k] + ALIGN - 1) / ALIGN * ALIGN;
        }
    };
    // Room for residues adds up to a half to a context (27 bytes an operand word, 36 a result word).  It is for speed alone, so
    // it is taken only where a quarter of the device's memory stays free for what else the caller has to place there.
    size_t free_bytes = 0, all_bytes = 0;
    if (ok && c->residues.bytes &&
        (cudaMemGetInfo(&free_bytes, &all_bytes) != cudaSuccess || total(device) + all_bytes / 4 > free_bytes)) {
        cudaGetLastError();
        for (int k = 0; k < planes_pieces; ++k) device.bytes[planes_piece + k] = planes_of_limbs[k];
        device.bytes[planes_piece + planes_pieces] = 0;
        c->planes_left.bytes = planes_of_limbs[0];
        c->planes_right_up.bytes = planes_of_limbs[1];
        c->planes_right_dn.bytes = planes_of_limbs[2];
        c->residues.bytes = 0;
    }
    ok = ok && cudaMalloc(&c->device_memory, total(device)) == cudaSuccess;
    ok = ok && cudaHostAlloc(&c->pinned_memory, total(pinned), cudaHostAllocMapped) == cudaSuccess;
    if (ok) {
        hand_out(device, c->device_memory);
        hand_out(pinned, c->pinned_memory);
        for (int p = 0; p < 2; ++p)
            for (int id = 0; id < COMET_NUM_TENSORS; ++id) c->buf[p][id] = c->own[p][id];
        c->d_error = c->d_count + 1;
        c->h_count[0] = c->h_count[1] = c->h_count[2] = c->h_count[3] = 0;     // pinned memory is not zeroed
        for (int k = 0; k < comet::PLAN_WORDS; ++k) c->h_masked[k] = 0;
    }
    // on the context's own stream: every kernel that uses these words is ordered behind it, whatever the default stream does
    ok = ok && cudaMemsetAsync(c->d_count, 0, 2 * sizeof(int32_t), c->stream) == cudaSuccess;
    ok = ok && cudaMemsetAsync(c->d_stream_sync, 0, c->stream_sync_words * sizeof(uint32_t), c->stream) == cudaSuccess;
    ok = ok && cudaHostGetDevicePointer((void**)&c->h_masked_dev, c->h_masked, 0) == cudaSuccess;
    ok = ok && cudaHostGetDevicePointer((void**)&c->h_count_dev, c->h_count, 0) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        comet_destroy(c);
        return COMET_ERR_OOM;
    }
    *out = c;
    return COMET_OK;
}

void comet_destroy(comet_ctx* c) {
    if (!c) return;
    cudaSetDevice(c->cfg.device);
    cudaStreamSynchronize(c->stream);
    if (c->side) cudaStreamSynchronize(c->side);
    if (c->ev_fork) cudaEventDestroy(c->ev_fork);
    if (c->ev_join) cudaEventDestroy(c->ev_join);
    if (c->side) cudaStreamDestroy(c->side);
    for (int k = 0; k < 4; ++k)
        if (c->stage_done[k]) cudaEventDestroy(c->stage_done[k]);
    if (c->device_memory) cudaFree(c->device_memory);
    if (c->pinned_memory) cudaFreeHost(c->pinned_memory);
    for (auto& p : *c->pending) {
        cudaEventDestroy(p.start);
        cudaEventDestroy(p.stop);
    }
    for (auto e : *c->free_events) cudaEventDestroy(e);
    delete c->pending;
    delete c->free_events;
    cudaGetLastError();
    delete c;
}

// Shared by comet_load_shares (copy) and comet_bind_shares (use in place).
static int set_shares(comet_ctx* c, int party, int tensor_id, const uint64_t* ptr, int location, int64_t rows,
                      int64_t cols, bool bind) {
    if (!c || (party != 0 && party != 1) || !is_input(tensor_id)) return COMET_ERR_INVALID_ARG;
    if (!ptr && rows * cols != 0) return COMET_ERR_INVALID_ARG;      // an empty tensor may come with a null pointer
    if (location != COMET_DEVICE && location != COMET_HOST) return COMET_ERR_INVALID_ARG;
    if (bind && (location != COMET_DEVICE || (reinterpret_cast<uintptr_t>(ptr) & 15u) != 0)) return COMET_ERR_INVALID_ARG;
    if (tensor_id == COMET_WG && c->groups < 2) return COMET_ERR_INVALID_ARG;
    if (tensor_id == COMET_W3 && c->groups != 3) return COMET_ERR_INVALID_ARG;
    const bool needs_mask = tensor_id == COMET_B_UP || tensor_id == COMET_C_UP || tensor_id == COMET_H ||
                            tensor_id == COMET_A_DN || tensor_id == COMET_B_DN;
    if (needs_mask && !c->mask_set) return COMET_ERR_STATE;
    const bool token_rows = tensor_id == COMET_X || tensor_id == COMET_A_UP || tensor_id == COMET_C_UP ||
                            tensor_id == COMET_H || tensor_id == COMET_A_DN || tensor_id == COMET_C_DN;
    if (token_rows && (rows < 1 || rows > c->cap_T)) return COMET_ERR_SHAPE;
    int64_t er, ec;
    tensor_shape(c, tensor_id, rows, &er, &ec);
    if (rows != er || cols != ec) return COMET_ERR_SHAPE;
    if (rows * cols > c->cap_words[tensor_id]) return COMET_ERR_SHAPE;
    if (tensor_id == COMET_W2 || tensor_id == COMET_B_DN || tensor_id == COMET_C_DN) {
        const int rc = join_side(c);       // the side stream may still be reading the old contents
        if (rc != COMET_OK) return rc;
        if (tensor_id == COMET_C_DN) c->dn_copy_ready = false;
        else c->dn_right_ready = false;
    }
    if (bind && rows * cols > 0) {
        c->buf[party][tensor_id] = const_cast<u64*>(reinterpret_cast<const u64*>(ptr));   // only ever read
    } else {
        c->buf[party][tensor_id] = c->own[party][tensor_id];
        if (rows * cols > 0)
            COMET_CUDA(c, cudaMemcpyAsync(c->buf[party][tensor_id], ptr, (size_t)(rows * cols) * sizeof(u64),
                                          copy_kind(location, true), c->stream));
    }
    c->loaded[party][tensor_id] = true;
    if (token_rows) c->tokens = (int32_t)rows;
    return COMET_OK;
}

int comet_load_shares(comet_ctx* c, int party, int tensor_id, const uint64_t* ptr, int location, int64_t rows,
                      int64_t cols) {
    return set_shares(c, party, tensor_id, ptr, location, rows, cols, false);
}

int comet_bind_shares(comet_ctx* c, int party, int tensor_id, const uint64_t* dev_ptr, int64_t rows, int64_t cols) {
    return set_shares(c, party, tensor_id, dev_ptr, COMET_DEVICE, rows, cols, true);
}

int comet_set_mask(comet_ctx* c, const uint8_t* block_mask, int location, int32_t n_blocks, int32_t* n_active_out) {
    if (!c || !block_mask || !n_active_out) return COMET_ERR_INVALID_ARG;
    if (location != COMET_DEVICE && location != COMET_HOST) return COMET_ERR_INVALID_ARG;
    if (n_blocks != c->cfg.d_ff / c->cfg.block) return COMET_ERR_SHAPE;
    {
        const int rc = join_side(c);           // the side stream reads the index list
        if (rc != COMET_OK) return rc;
    }
    c->dn_right_ready = false;
    const uint8_t* dmask = block_mask;         // a device mask is read in place
    int32_t host_count = -1;                   // number of active blocks when the host could count them itself
    bool launched = false;
    c->ids_held = location == COMET_HOST && n_blocks <= comet::BlockIds::CAPACITY && c->path == COMET_PATH_LIMB;
    if (location == COMET_HOST) {
        // The count is public (Section 3.2) and the mask is in host memory: count here and do not wait for the
        // device.  The index list of a mask of up to 1024 blocks is made here and travels with the launches that gather; a
        // mask that fits into a kernel's parameter block travels with the compaction's launch; a larger one is handed
        // to the copy engine from a pinned slot of our own (the caller's buffer is free again on return either way).
        host_count = 0;
        if (c->ids_held) {
            for (int32_t b = 0; b < n_blocks; ++b)
                if (block_mask[b]) c->held.id[host_count++] = (uint16_t)b;
            launched = true;
        } else {
            for (int32_t b = 0; b < n_blocks; ++b) host_count += block_mask[b] != 0;
        }
        if (launched) {
            // nothing to launch
        } else if (n_blocks <= comet::MaskBytes::CAPACITY) {
            comet::MaskBytes arg;
            std::memcpy(arg.bytes, block_mask, (size_t)n_blocks);
            PhaseTimer timer(c, COMET_PHASE_COMPACT, 1);
            c->ticket += 1;
            COMET_CUDA(c, launch_chained(comet::compact_mask_arg_kernel, dim3(1), dim3(1024), 0, c->stream, nullptr, arg,
                                         (int)n_blocks, c->d_ids, c->d_count, (int32_t*)nullptr, c->ticket));
            c->stats.kernel_launches += 1;
            launched = true;
        } else {
            const int slot = c->stage_next;
            c->stage_next = (slot + 1) % 4;
            if (c->stage_used[slot]) COMET_CUDA(c, cudaEventSynchronize(c->stage_done[slot]));
            uint8_t* stage = c->h_mask_stage + (size_t)slot * n_blocks;
            std::memcpy(stage, block_mask, (size_t)n_blocks);
            COMET_CUDA(c, cudaMemcpyAsync(c->d_mask, stage, (size_t)n_blocks, cudaMemcpyHostToDevice, c->stream));
            COMET_CUDA(c, cudaEventRecord(c->stage_done[slot], c->stream));
            c->stage_used[slot] = true;
            dmask = c->d_mask;
        }
    }
    if (!launched) {
        PhaseTimer timer(c, COMET_PHASE_COMPACT, 1);
        // the kernel reports {count, error flag} straight into mapped host memory: no copy to enqueue
        c->ticket += 1;
        COMET_CUDA(c, launch_chained(comet::compact_mask_kernel, dim3(1), dim3(1024), 0, c->stream, nullptr, dmask,
                                     (int)n_blocks, c->d_ids, c->d_count, host_count < 0 ? c->h_count_dev : (int32_t*)nullptr,
                                     c->ticket));
        c->stats.kernel_launches += 1;
    }
    COMET_CUDA(c, cudaGetLastError());
    if (host_count < 0) {
        const volatile int32_t* seen = c->h_count + 2;
        const int32_t ticket = c->ticket;
        const int rc = wait_for_report(c, [=] { return *seen == ticket; });
        if (rc != COMET_OK) return rc;
    }
    if (timed_out(c)) return COMET_ERR_TIMEOUT;           // an earlier kernel gave up on a bounded wait
    const int32_t blocks = host_count >= 0 ? host_count : *c->h_count;
    const int64_t n = (int64_t)blocks * c->cfg.block;
    if (n > c->cap_n) {            // more active neurons than the context was sized for
        c->mask_set = false;
        return COMET_ERR_SHAPE;
    }
    c->n_active_blocks = blocks;
    c->n_active = (int32_t)n;
    c->mask_set = true;
    c->tmask_set = false;             // a token mask refines one block mask
    c->grouped = false;
    c->up_done = c->down_done = false;
    for (int p = 0; p < 2; ++p)
        for (int id = COMET_A_UP; id <= COMET_C_DN; ++id) {
            c->loaded[p][id] = false;
            c->buf[p][id] = c->own[p][id];          // a binding ends with the mask it was made under
        }
    c->stats.n_active = c->n_active;
    c->stats.n_active_blocks = blocks;
    *n_active_out = c->n_active;
    return COMET_OK;
}

int comet_set_token_mask(comet_ctx* c, const uint8_t* token_mask, int location, int32_t tokens,
                         int32_t n_active_blocks, int64_t* masked_out) {
    if (!c) return COMET_ERR_INVALID_ARG;
    if (!c->mask_set) return COMET_ERR_STATE;
    if (!token_mask) {                         // back to "every token uses every active neuron"
        if (tokens != 0 || n_active_blocks != 0) return COMET_ERR_INVALID_ARG;
        // the weight side of the down-projection may have been opened early under the mask that is going away
        // (its unused blocks zeroed, its contraction index in component order): it is opened again
        if (c->tmask_set) c->dn_right_ready = false;
        c->tmask_set = false;
        c->grouped = false;
        if (masked_out) *masked_out = 0;
        return COMET_OK;
    }
    if (location != COMET_DEVICE && location != COMET_HOST) return COMET_ERR_INVALID_ARG;
    if (tokens < 1 || tokens > c->cap_T || n_active_blocks != c->n_active_blocks || n_active_blocks < 1)
        return COMET_ERR_SHAPE;
    if ((int64_t)tokens * c->n_active < 0 || (int64_t)tokens * c->n_active > 0x7fffffffll) return COMET_ERR_SHAPE;
    const size_t bytes = (size_t)tokens * (size_t)n_active_blocks;
    if (location == COMET_HOST)
        COMET_CUDA(c, cudaMemcpyAsync(c->d_tmask, token_mask, bytes, cudaMemcpyHostToDevice, c->stream));
    // Protocol 2, first step: the connected components the up-projection is partitioned into, the number of
    // non-zero entries (Theorem 2's count) and, for the tensor-core path, the component-sorted order and the work
    // of every row tile, in one launch
    const bool plan = c->path == COMET_PATH_LIMB && tokens > comet::limb_stream::BT && tokens <= 32768;
    {
        comet::TokenPlanArgs a;
        std::memset(&a, 0, sizeof(a));
        a.S = location == COMET_HOST ? c->d_tmask : token_mask;
        a.copy = location == COMET_HOST ? nullptr : c->d_tmask;
        a.T = tokens; a.nab = n_active_blocks; a.wpr = ceil_div(n_active_blocks, 32);
        a.row_label = c->d_row_label; a.blk_label = c->d_blk_label;
        a.report = c->h_masked_dev;
        c->plan_ticket = c->plan_ticket % ((1ull << (64 - comet::PLAN_VALUE_BITS)) - 1) + 1;      // never 0
        a.ticket = c->plan_ticket;
        a.scratch = c->d_plan_scratch;
        a.plan = plan ? 1 : 0;
        a.groups = c->groups; a.bs = c->cfg.block;
        a.kb_up = ceil_div(c->cfg.d_model, comet::limb::KC);
        a.nt_dn = ceil_div(c->cfg.d_model, comet::limb::BN);
        a.row_map = c->d_row_map; a.col_map = c->d_col_map; a.kmap = c->d_kmap;
        a.up = c->d_group_up; a.dn = c->d_group_dn;
        const size_t words = comet::token_plan_words(tokens, n_active_blocks, a.wpr, c->groups);
        a.in_smem = words * sizeof(uint32_t) <= 36 * 1024 ? 1 : 0;
        COMET_CUDA(c, launch_chained(comet::token_plan_kernel, dim3(1), dim3(1024), a.in_smem ? words * sizeof(uint32_t) : 0,
                                     c->stream, nullptr, a));
    }
    c->stats.kernel_launches += 1;
    {
        const volatile unsigned long long* words = c->h_masked;
        const unsigned long long ticket = c->plan_ticket;
        const int rc = wait_for_report(c, [=] {
            for (int k = 0; k < comet::PLAN_WORDS; ++k)
                if (words[k] >> comet::PLAN_VALUE_BITS != ticket) return false;
            return true;
        });
        if (rc != COMET_OK) return rc;
    }
    auto reported = [c](int k) { return (int64_t)(c->h_masked[k] & ((1ull << comet::PLAN_VALUE_BITS) - 1)); };
    c->tmask_masked = reported(0) * c->cfg.block;
    c->n_components = (int32_t)reported(1);
    c->live_rows = (int32_t)reported(2);
    c->live_blocks = (int32_t)reported(3);
    c->group_units_up = plan ? (int32_t)reported(4) : 0;
    c->component_pairs = plan ? reported(5) : -1;
    c->group_units_dn = plan ? (int32_t)reported(6) : 0;
    // several components, or rows / blocks in none: compute the component rectangles only
    c->grouped = plan && c->group_units_up > 0 && c->group_units_dn > 0 &&
                 (c->n_components > 1 || c->live_rows < tokens || c->live_blocks < n_active_blocks);
    c->dn_right_ready = false;    // the order of the contraction index in the down-projection's planes may change
    c->stats.n_components = c->n_components;
    c->tmask_tokens = tokens;
    c->tmask_set = true;
    if (masked_out) *masked_out = c->tmask_masked;
    return COMET_OK;
}

int comet_ffn_up(comet_ctx* c, int32_t tokens) {
    if (!c) return COMET_ERR_INVALID_ARG;
    if (tokens < 1 || tokens > c->cap_T) return COMET_ERR_SHAPE;
    if (!c->mask_set) return COMET_ERR_STATE;
    const int need[] = {COMET_X, COMET_W1, COMET_A_UP, COMET_B_UP, COMET_C_UP};
    for (int p = 0; p < 2; ++p) {
        for (int id : need)
            if (!c->loaded[p][id]) return COMET_ERR_STATE;
        if (c->groups >= 2 && !c->loaded[p][COMET_WG]) return COMET_ERR_STATE;
        if (c->groups == 3 && !c->loaded[p][COMET_W3]) return COMET_ERR_STATE;
    }
    const int d = c->cfg.d_model, n = c->n_active, g = c->groups, bs = c->cfg.block;
    if (c->tmask_set && c->tmask_tokens != tokens) return COMET_ERR_SHAPE;   // the token mask was given for another T
    c->stats.tokens = tokens;
    // under a token mask only the rows and columns of the connected components are opened (Theorem 1)
    c->stats.message_bytes = c->tmask_set
        ? 2ll * 8 * ((int64_t)c->live_rows * d + (int64_t)d * g * c->live_blocks * bs)
        : 2ll * 8 * ((int64_t)tokens * d + (int64_t)d * g * n);
    // Theorem 1's multiplication count when the components are known (one product per component), else the
    // product over the union of the supports
    c->stats.ring_macs = (c->tmask_set && c->component_pairs >= 0)
        ? 2ll * 2 * d * g * bs * c->component_pairs : 2ll * 2 * tokens * (int64_t)d * g * n;
    c->stats.tensor_tile_macs = 0;
    c->up_tokens = tokens;
    c->up_done = true;
    if (n == 0) return COMET_OK;

    if (c->path == COMET_PATH_LIMB) {
        const Proj up = proj_up(c, tokens), dn = proj_down(c, tokens);
        int rc = join_side(c);
        if (rc != COMET_OK) return rc;
        OperandsOffResult operands(c, up);
        rc = operands.move();
        if (rc != COMET_OK) return rc;
        if (few_tokens(c, tokens)) {
            rc = stream_product(c, up);
            return rc != COMET_OK ? rc : somm_merge(c, tokens);
        }
        if (!limb_fits(c, up)) return COMET_ERR_SHAPE;
        const bool residue = through_residues(c, up), dn_residue = through_residues(c, dn);
        // The weight side of the down-projection depends only on the mask, W2 and B'_i: if those are loaded already, it is
        // opened now, and if the triple's C' share is there too, Y_i <- C'_i, the value the down-projection's sums are added
        // to, is copied with it.  Where: a small one in the same launch as this product's exchange, which costs nothing but
        // its traffic; from EXCHANGE_APART words on, on the side stream beside the tensor-core kernel (not beside the
        // exchange before it, which is bound by the same memory), which hides about half of it but takes two events, a
        // launch and the programmatic start of the tensor-core kernel.  A step with 0.03 million such words takes 25 us in
        // one launch and 34 apart, with 0.52 million 97 and 94, with 1.7 million 249 and 237.  Fewer words are
        // worth that where the product is long enough to hide them all (long_product).  The stream then waits for them
        // behind the product: what such a call has enqueued is over when the stream is, so it can be captured without the
        // down-projection, and the down-projection without it.  In one launch, apart, and apart without that wait: 0.25 million words and
        // 49 million multiply-adds 40.9, 40.8 and 39.8 us, 0.23 million and 117 million 57.0, 55.1 and 55.2; 0.16 million and 65 million 48.1, 46.6
        // and 46.9; 0.13 million and 52 million 40.5, 38.8 and 39.0, 65 million 41.0, 40.4 and 40.1; 0.11 million and 59 million 41.0, 39.7 and 39.8
        // as 256 x 448, 39.2, 39.5 and 39.2 as 512 x 224.  In one launch and apart: 0.1 million and 50 million 36.6 and 36.9 as 512 x 192, 36.6 and
        // 36.2 as 384 x 256; 0.09 million and 46 million 36.2 and 36.7; 0.08 million and 82 million 50.1 and 49.0; 0.07 million and 67 million
        // 42.5 either way.  Under a token mask of several components the product works through fewer, but drains longer, so the count is
        // the same: 0.25 million words in four groups 76.0 and 75.2 (768 x 320), 81.2 and 77.8 (1024 x 240), in sixteen 74.4 and 73.3, in eight
        // 75.6 either way; 0.13 million in sixteen 59.0 and 59.1.
        // A launch writes planes of one kind, so a weight side of the other kind goes apart whatever its size.  The kernel on
        // residues reads C' when it makes Y: nothing is copied for it.
        // An operand of this product may lie on Y: C' is then not copied there before it has been read.  The exchange reads
        // all operands, so a copy that waits for it (on the side stream) is safe, one in the same launch is not; C is read
        // after the product where that goes through residues, and a copy beside the product would be too early for it.
        const bool early = !c->dn_right_ready && limb_fits(c, dn) && c->loaded[0][COMET_W2] &&
                           c->loaded[1][COMET_W2] && c->loaded[0][COMET_B_DN] && c->loaded[1][COMET_B_DN];
        const bool few_words = residue == dn_residue && (int64_t)dn.N * dn.K < EXCHANGE_APART;
        const bool apart = early && (!few_words || long_product((int64_t)dn.N * dn.K, (int64_t)up.M * up.N * up.K));
        const bool y_in_use = !apart ? operands.any_on(COMET_Y) : residue && operands.on(up.idC, COMET_Y);
        const bool early_copy = early && !dn_residue && !y_in_use && c->loaded[0][COMET_C_DN] && c->loaded[1][COMET_C_DN];
        comet::LimbExchangeArgs also;
        const int also_blocks = early && !apart ? exchange_args(c, dn, dn_residue, false, true, early_copy, also) : 0;
        {
            PhaseTimer timer(c, COMET_PHASE_OPEN, 1);
            rc = limb_exchange(c, up, residue, true, true, !residue, c->stream, also_blocks ? &also : nullptr, also_blocks);
        }
        if (rc != COMET_OK) return rc;
        if (apart) COMET_CUDA(c, cudaEventRecord(c->ev_fork, c->stream));
        rc = residue ? residue_combine(c, up) : limb_combine(c, up);
        if (rc != COMET_OK) return rc;
        if (apart) {
            COMET_CUDA(c, cudaStreamWaitEvent(c->side, c->ev_fork, 0));
            rc = limb_exchange(c, dn, dn_residue, false, true, early_copy, c->side);
            if (rc != COMET_OK) return rc;
            COMET_CUDA(c, cudaEventRecord(c->ev_join, c->side));
            c->side_pending = true;
            rc = few_words ? join_side(c) : COMET_OK;
            if (rc != COMET_OK) return rc;
        }
        if (early) {
            c->dn_right_ready = true;
            c->dn_right_residue = dn_residue;
            c->dn_copy_ready = early_copy;
            c->dn_copy_tokens = tokens;
        }
        return somm_merge(c, tokens);
    }

    comet::PartyPtrs X, A, W0, W1, W3, B;
    comet::PartyOut E, F;
    for (int p = 0; p < 2; ++p) {
        X.p[p] = c->buf[p][COMET_X];
        A.p[p] = c->buf[p][COMET_A_UP];
        E.p[p] = c->buf[p][COMET_E_UP];
        W0.p[p] = (g >= 2) ? c->buf[p][COMET_WG] : c->buf[p][COMET_W1];
        W3.p[p] = c->buf[p][COMET_W3];
        W1.p[p] = c->buf[p][COMET_W1];
        B.p[p] = c->buf[p][COMET_B_UP];
        F.p[p] = c->buf[p][COMET_F_UP];
    }
    const int64_t pairs = (int64_t)tokens * d / 2;
    {
        PhaseTimer timer(c, COMET_PHASE_OPEN, 2);
        comet::open_activation_kernel<<<dim3(ew_grid(c, pairs, 256), 2), 256, 0, c->stream>>>(
            X, A, E, pairs, nullptr, 0, d, bs, c->tmask_set ? c->d_row_label : nullptr);
        int rows_grid = g * n < c->sm_count * 8 ? g * n : c->sm_count * 8;
        comet::open_weight_rows_kernel<<<dim3(rows_grid, 2), 256, 0, c->stream>>>(
            W0, W1, W3, B, F, c->d_ids, n, g, bs, d, c->tmask_set ? c->d_blk_label : nullptr);
    }
    c->stats.kernel_launches += 2;
    COMET_CUDA(c, cudaGetLastError());
    const int rc = launch_combine(c, tokens, g * n, d, COMET_E_UP, COMET_F_UP, COMET_A_UP, COMET_B_UP, COMET_C_UP,
                                  COMET_Z_UP);
    if (rc != COMET_OK) return rc;
    return somm_merge(c, tokens);
}

int comet_ffn_down(comet_ctx* c, int32_t tokens) {
    if (!c) return COMET_ERR_INVALID_ARG;
    if (tokens < 1 || tokens > c->cap_T) return COMET_ERR_SHAPE;
    if (!c->mask_set) return COMET_ERR_STATE;
    const int d = c->cfg.d_model, n = c->n_active, bs = c->cfg.block, D = c->cfg.d_ff;
    for (int p = 0; p < 2; ++p) {
        if (!c->loaded[p][COMET_W2] || !c->loaded[p][COMET_C_DN]) return COMET_ERR_STATE;
        if (n > 0 && (!c->loaded[p][COMET_H] || !c->loaded[p][COMET_A_DN] || !c->loaded[p][COMET_B_DN]))
            return COMET_ERR_STATE;
    }
    if (c->tmask_set && c->tmask_tokens != tokens) return COMET_ERR_SHAPE;   // the token mask was given for another T
    c->stats.tokens = tokens;
    // with a token mask only the non-zero entries of the hidden state and the rows of the weight matrix that meet
    // a non-zero column are opened (Theorem 2's communication)
    c->stats.message_bytes = c->tmask_set
        ? 2ll * 8 * (c->tmask_masked + (int64_t)c->live_blocks * bs * d)
        : 2ll * 8 * ((int64_t)tokens * n + (int64_t)n * d);
    // Theorem 2's multiplication count under a token mask (one product row per non-zero entry), else the full product
    c->stats.ring_macs = 2ll * 2 * (c->tmask_set ? c->tmask_masked : (int64_t)tokens * n) * d;
    c->stats.tensor_tile_macs = 0;
    c->down_tokens = tokens;
    c->down_done = true;
    if (n == 0) {
        // no active neuron: the product is empty and both result shares are zero
        for (int p = 0; p < 2; ++p)
            COMET_CUDA(c, cudaMemsetAsync(c->buf[p][COMET_Y], 0, (size_t)tokens * d * sizeof(u64), c->stream));
        return COMET_OK;
    }
    if (c->path == COMET_PATH_LIMB) {
        const Proj dn = proj_down(c, tokens);
        int rc = join_side(c);
        if (rc != COMET_OK) return rc;
        OperandsOffResult operands(c, dn);
        rc = operands.move();
        if (rc != COMET_OK) return rc;
        if (few_tokens(c, tokens)) {
            c->dn_right_ready = false;
            c->dn_copy_ready = false;
            return stream_product(c, dn);
        }
        if (!limb_fits(c, dn)) return COMET_ERR_SHAPE;
        // opened early, during the up-projection
        const bool residue = through_residues(c, dn);
        const bool have_right = c->dn_right_ready && c->dn_right_residue == residue;
        const bool have_copy = residue || (c->dn_right_ready && c->dn_copy_ready && c->dn_copy_tokens == tokens);
        {
            PhaseTimer timer(c, COMET_PHASE_OPEN, 1);
            rc = limb_exchange(c, dn, residue, true, !have_right, !have_copy, c->stream);
        }
        if (rc != COMET_OK) return rc;
        c->dn_right_ready = false;                     // a triple serves one product
        c->dn_copy_ready = false;
        return residue ? residue_combine(c, dn) : limb_combine(c, dn);
    }

    comet::PartyPtrs H, A, W, B;
    comet::PartyOut E, F;
    for (int p = 0; p < 2; ++p) {
        H.p[p] = c->buf[p][COMET_H];
        A.p[p] = c->buf[p][COMET_A_DN];
        E.p[p] = c->buf[p][COMET_E_DN];
        W.p[p] = c->buf[p][COMET_W2];
        B.p[p] = c->buf[p][COMET_B_DN];
        F.p[p] = c->buf[p][COMET_F_DN];
    }
    const int64_t pairs = (int64_t)tokens * n / 2;
    {
        PhaseTimer timer(c, COMET_PHASE_OPEN, 2);
        comet::open_activation_kernel<<<dim3(ew_grid(c, pairs, 256), 2), 256, 0, c->stream>>>(
            H, A, E, pairs, c->tmask_set ? c->d_tmask : nullptr, c->n_active_blocks, n, bs);
        const int64_t wpairs = (int64_t)d * n / 2;
        comet::open_weight_strips_kernel<<<dim3(ew_grid(c, wpairs, 256), 2), 256, 0, c->stream>>>(
            W, B, F, c->d_ids, n, bs, d, D, c->tmask_set ? c->d_blk_label : nullptr);
    }
    c->stats.kernel_launches += 2;
    COMET_CUDA(c, cudaGetLastError());
    return launch_combine(c, tokens, d, n, COMET_E_DN, COMET_F_DN, COMET_A_DN, COMET_B_DN, COMET_C_DN, COMET_Y);
}

int comet_truncate(comet_ctx* c, int tensor_id) {
    if (!c || (tensor_id != COMET_Z_UP && tensor_id != COMET_Y)) return COMET_ERR_INVALID_ARG;
    const bool up = tensor_id == COMET_Z_UP;
    if (up ? !c->up_done : !c->down_done) return COMET_ERR_STATE;
    int64_t rows, cols;
    tensor_shape(c, tensor_id, up ? c->up_tokens : c->down_tokens, &rows, &cols);
    const int64_t pairs = rows * cols / 2;
    if (pairs == 0) return COMET_OK;
    comet::PartyOut Z;
    for (int p = 0; p < 2; ++p) Z.p[p] = c->buf[p][tensor_id];
    {
        PhaseTimer timer(c, COMET_PHASE_TRUNCATE, 1);
        COMET_CUDA(c, launch_chained(comet::truncate_kernel, dim3(ew_grid(c, pairs, 256), 2), dim3(256), 0, c->stream,
                                     nullptr, Z, pairs, (int)c->cfg.frac_bits));
    }
    c->stats.kernel_launches += 1;
    COMET_CUDA(c, cudaGetLastError());
    return COMET_OK;
}

int comet_get(comet_ctx* c, int party, int tensor_id, uint64_t* out, int location, int64_t capacity,
              int64_t* written) {
    if (!c || !out || (party != 0 && party != 1) || tensor_id < 0 || tensor_id >= COMET_NUM_TENSORS)
        return COMET_ERR_INVALID_ARG;
    if (location != COMET_DEVICE && location != COMET_HOST) return COMET_ERR_INVALID_ARG;
    if (tensor_id == COMET_WG && c->groups < 2) return COMET_ERR_INVALID_ARG;
    if (tensor_id == COMET_W3 && c->groups != 3) return COMET_ERR_INVALID_ARG;
    int64_t T = c->tokens;
    if (tensor_id == COMET_E_UP || tensor_id == COMET_Z_UP) T = c->up_tokens;
    if (tensor_id == COMET_E_DN || tensor_id == COMET_Y) T = c->down_tokens;
    int64_t rows, cols;
    tensor_shape(c, tensor_id, T, &rows, &cols);
    const int64_t words = rows * cols;
    if (is_input(tensor_id) ? !c->loaded[party][tensor_id]
                            : !((tensor_id == COMET_E_UP || tensor_id == COMET_F_UP || tensor_id == COMET_Z_UP)
                                    ? c->up_done : c->down_done))
        return COMET_ERR_STATE;
    if (capacity < words) return COMET_ERR_SHAPE;
    if (words > 0)
        COMET_CUDA(c, cudaMemcpyAsync(out, c->buf[party][tensor_id], (size_t)words * sizeof(u64),
                                      copy_kind(location, false), c->stream));
    if (written) *written = words;
    if (timed_out(c)) return COMET_ERR_TIMEOUT;    // what has been handed out is not the result
    return COMET_OK;
}

int comet_synchronize(comet_ctx* c) {
    if (!c) return COMET_ERR_INVALID_ARG;
    COMET_CUDA(c, cudaStreamSynchronize(c->stream));
    if (c->side) COMET_CUDA(c, cudaStreamSynchronize(c->side));
    std::atomic_thread_fence(std::memory_order_acquire);
    return timed_out(c) ? COMET_ERR_TIMEOUT : COMET_OK;
}

int comet_inject_timeout(comet_ctx* c) {
    if (!c) return COMET_ERR_INVALID_ARG;
    COMET_CUDA(c, cudaStreamSynchronize(c->stream));
    const int32_t one = 1;
    COMET_CUDA(c, cudaMemcpy(c->d_error, &one, sizeof(one), cudaMemcpyHostToDevice));
    c->h_count[3] = 1;
    return COMET_OK;
}

int comet_device_pointer(comet_ctx* c, int party, int tensor_id, uint64_t** out) {
    if (!c || !out || (party != 0 && party != 1)) return COMET_ERR_INVALID_ARG;
    if (tensor_id != COMET_Z_UP && tensor_id != COMET_Y) return COMET_ERR_INVALID_ARG;
    *out = reinterpret_cast<uint64_t*>(c->own[party][tensor_id]);
    return COMET_OK;
}

int comet_get_index(comet_ctx* c, int32_t* out, int location, int32_t capacity, int32_t* n_active_blocks_out) {
    if (!c || !out || !n_active_blocks_out) return COMET_ERR_INVALID_ARG;
    if (location != COMET_DEVICE && location != COMET_HOST) return COMET_ERR_INVALID_ARG;
    if (!c->mask_set) return COMET_ERR_STATE;
    if (capacity < c->n_active_blocks) return COMET_ERR_SHAPE;
    if (c->ids_held) {
        if (location == COMET_HOST) std::copy(c->held.id, c->held.id + c->n_active_blocks, out);
        else if (c->n_active_blocks > 0) {
            COMET_CUDA(c, launch_chained(comet::held_ids_kernel, dim3(1), dim3(comet::BlockIds::CAPACITY), 0, c->stream, nullptr,
                                         c->held, (int)c->n_active_blocks, out));
            c->stats.kernel_launches += 1;
        }
    } else if (c->n_active_blocks > 0)
        COMET_CUDA(c, cudaMemcpyAsync(out, c->d_ids, (size_t)c->n_active_blocks * sizeof(int32_t),
                                      copy_kind(location, false), c->stream));
    *n_active_blocks_out = c->n_active_blocks;
    return COMET_OK;
}

int comet_get_components(comet_ctx* c, int32_t* row_label, int32_t* blk_label, int location,
                         int32_t* n_components_out) {
    if (!c || !row_label || !blk_label || !n_components_out) return COMET_ERR_INVALID_ARG;
    if (location != COMET_DEVICE && location != COMET_HOST) return COMET_ERR_INVALID_ARG;
    if (!c->mask_set || !c->tmask_set) return COMET_ERR_STATE;
    COMET_CUDA(c, cudaMemcpyAsync(row_label, c->d_row_label, (size_t)c->tmask_tokens * sizeof(int32_t),
                                  copy_kind(location, false), c->stream));
    COMET_CUDA(c, cudaMemcpyAsync(blk_label, c->d_blk_label, (size_t)c->n_active_blocks * sizeof(int32_t),
                                  copy_kind(location, false), c->stream));
    *n_components_out = c->n_components;
    return COMET_OK;
}

int comet_stats(comet_ctx* c, comet_stats_t* out) {
    if (!c || !out) return COMET_ERR_INVALID_ARG;
    if (!c->pending->empty()) {
        COMET_CUDA(c, cudaStreamSynchronize(c->stream));
        for (auto& p : *c->pending) {
            float ms = 0.f;
            if (cudaEventElapsedTime(&ms, p.start, p.stop) == cudaSuccess) {
                c->stats.phase_ms[p.phase] += ms;
                c->stats.phase_launches[p.phase] += p.launches;
            }
            c->free_events->push_back(p.start);
            c->free_events->push_back(p.stop);
        }
        c->pending->clear();
        cudaGetLastError();
    }
    *out = c->stats;
    return COMET_OK;
}

int comet_set_profiling(comet_ctx* c, int on) {
    if (!c) return COMET_ERR_INVALID_ARG;
    comet_stats_t tmp;
    const int rc = comet_stats(c, &tmp);      // drain what is pending
    if (rc != COMET_OK) return rc;
    c->profiling = on != 0;
    if (c->profiling)
        for (int k = 0; k < COMET_NUM_PHASES; ++k) {
            c->stats.phase_ms[k] = 0.0;
            c->stats.phase_launches[k] = 0;
        }
    return COMET_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free Pi_MatMul: the message buffers live in the library image.
// ---------------------------------------------------------------------------
namespace {

// Scratch for E_0, E_1, F_0, F_1 of comet_beaver_matmul_static.  In host code
// this name is only a handle for cudaGetSymbolAddress, never an address to hand
// to a kernel; each GPU that loads the library carries its own 8 MiB copy.
static __device__ __align__(256) unsigned long long g_static_scratch[COMET_STATIC_SCRATCH_WORDS];
// Set by a kernel of such a call that gave up on a bounded wait; comet_static_status reads and clears it.
static __device__ int g_static_error;

constexpr int kMaxDevices = 64;
struct StaticDevice {
    u64* scratch;      // device address of the array
    int* error;        // and of the error word
    int sm_count;
};
std::mutex g_static_mutex;
StaticDevice g_static_device[kMaxDevices] = {};    // per device ordinal

// The scratch array on the current device and what launching there needs (looked up once per device).
cudaError_t static_device(StaticDevice* out) {
    int dev = -1;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    StaticDevice& d = g_static_device[dev];
    if (!d.scratch) {
        void *p = nullptr, *e = nullptr;
        err = cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, dev);
        for (auto* kernel : {comet::combine_stream_kernel<16, comet::limb_stream::BW>, comet::combine_stream_kernel<32, comet::limb_stream::BW>,
                             comet::combine_stream_kernel<16, comet::limb_stream::QROWS>, comet::combine_stream_kernel<32, comet::limb_stream::QROWS>})
            if (err == cudaSuccess)
                err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)comet::limb_stream::SMEM_BYTES);
        if (err == cudaSuccess) err = cudaGetSymbolAddress(&p, g_static_scratch);
        if (err == cudaSuccess) err = cudaGetSymbolAddress(&e, g_static_error);
        if (err != cudaSuccess) return err;
        d.error = static_cast<int*>(e);
        d.scratch = static_cast<u64*>(p);
    }
    *out = d;
    return cudaSuccess;
}

// Products a quarter of a step deep with very many token rows and few features run on the CUDA cores: the streaming kernel fills
// up every step and walks the features again for each of its 32-row tiles, where the other kernel takes 128 x 64 results at a
// time.  The line is the fourth round of tiles over the SMs.  CUDA cores / streaming, K = 8: 14000 x 4 25 / 22 us, 16384 x 4
// 25 / 28, 64000 x 4 66 / 86, 16384 x 64 28 / 32, 64000 x 64 101 / 113, but 64000 x 68 177 / 120, and K = 16: 16384 x 4 37 / 28.
// (20000 .. 50000 x 4000 .. 8000, 3 to 7 % slower streaming, are left there.)
bool static_on_alus(int T, int K, int N, int sm_count) {
    return K < 16 && N <= comet::simt::BN && T > 3 * comet::limb_stream::BT * sm_count;
}

// Whether the result lies on an operand other than its own C (an in-place product).  The streaming kernel writes Z before it
// has read every operand; the kernels of the other path read X and Y in a launch of their own before the first word of Z.
bool static_in_place(const uint64_t* const X[2], const uint64_t* const A[2], const uint64_t* const Y[2],
                     const uint64_t* const B[2], const uint64_t* const C[2], uint64_t* const Z[2], int64_t T, int64_t K,
                     int64_t N) {
    for (int q = 0; q < 2; ++q) {
        const uintptr_t z = reinterpret_cast<uintptr_t>(Z[q]), z_end = z + (uintptr_t)(T * N) * sizeof(u64);
        auto on = [&](const uint64_t* p, int64_t words) {
            const uintptr_t at = reinterpret_cast<uintptr_t>(p);
            return at < z_end && z < at + (uintptr_t)words * sizeof(u64);
        };
        for (int p = 0; p < 2; ++p)
            if (on(X[p], T * K) || on(A[p], T * K) || on(Y[p], N * K) || on(B[p], N * K) || (on(C[p], T * N) && (p != q || C[p] != Z[q])))
                return true;
    }
    return false;
}

}  // namespace

extern "C" int comet_beaver_matmul_static(void* cuda_stream, const uint64_t* const X[2], const uint64_t* const A[2],
                                          const uint64_t* const Y[2], const uint64_t* const B[2],
                                          const uint64_t* const C[2], uint64_t* const Z[2], int32_t T, int32_t K,
                                          int32_t N) {
    if (!X || !A || !Y || !B || !C || !Z) return COMET_ERR_INVALID_ARG;
    for (int p = 0; p < 2; ++p)
        if (!X[p] || !A[p] || !Y[p] || !B[p] || !C[p] || !Z[p]) return COMET_ERR_INVALID_ARG;
    // the kernels below read and write every operand 16 bytes at a time
    for (int p = 0; p < 2; ++p) {
        const void* ptrs[6] = {X[p], A[p], Y[p], B[p], C[p], Z[p]};
        for (const void* q : ptrs)
            if ((reinterpret_cast<uintptr_t>(q) & 15u) != 0) return COMET_ERR_INVALID_ARG;
    }
    if (T < 1 || K < 8 || N < 4 || K % 8 || N % 4) return COMET_ERR_SHAPE;
    const int64_t left = (int64_t)T * K, right = (int64_t)N * K;
    if (2 * (left + right) > (int64_t)COMET_STATIC_SCRATCH_WORDS) return COMET_ERR_SCRATCH_LIMIT;

    StaticDevice dev;
    if (static_device(&dev) != cudaSuccess) {
        cudaGetLastError();
        return COMET_ERR_CUDA;
    }
    // the array is carved into E_0 | E_1 | F_0 | F_1 (every word used is written before anything reads it)
    u64* const E[2] = {dev.scratch, dev.scratch + left};
    u64* const F[2] = {dev.scratch + 2 * left, dev.scratch + 2 * left + right};
    if (static_on_alus(T, K, N, dev.sm_count) || static_in_place(X, A, Y, B, C, Z, T, K, N)) {
        comet::PartyPtrs x, a, y, b;
        comet::PartyOut e, f;
        comet::CombineArgs args;
        std::memset(&args, 0, sizeof(args));
        for (int p = 0; p < 2; ++p) {
            x.p[p] = reinterpret_cast<const u64*>(X[p]);
            y.p[p] = reinterpret_cast<const u64*>(Y[p]);
            args.A[p] = a.p[p] = reinterpret_cast<const u64*>(A[p]);
            args.B[p] = b.p[p] = reinterpret_cast<const u64*>(B[p]);
            args.C[p] = reinterpret_cast<const u64*>(C[p]);
            args.Z[p] = reinterpret_cast<u64*>(Z[p]);
            args.E[p] = e.p[p] = E[p];
            args.F[p] = f.p[p] = F[p];
        }
        args.M = T; args.N = N; args.K = K;
        args.bs = 1;
        cudaStream_t stream = (cudaStream_t)cuda_stream;
        auto grid = [&](int64_t pairs) {
            const int64_t want = (pairs + 255) / 256, most = (int64_t)dev.sm_count * 8;
            return dim3((unsigned)(want < most ? want : most), 2);
        };
        comet::open_activation_kernel<<<grid(left / 2), 256, 0, stream>>>(x, a, e, left / 2, nullptr, 0, K, 1);
        comet::open_activation_kernel<<<grid(right / 2), 256, 0, stream>>>(y, b, f, right / 2, nullptr, 0, K, 1);
        comet::combine_simt_kernel<<<dim3(ceil_div(N, comet::simt::BN), ceil_div(T, comet::simt::BM), 2), comet::simt::THREADS, 0,
                                     stream>>>(args);
        return cudaGetLastError() == cudaSuccess ? COMET_OK : COMET_ERR_CUDA;
    }
    // the streaming kernel over [N, K] right operands without a gather
    comet::StreamArgs a;
    std::memset(&a, 0, sizeof(a));
    for (int p = 0; p < 2; ++p) {
        a.X[p] = reinterpret_cast<const u64*>(X[p]);
        a.A[p] = reinterpret_cast<const u64*>(A[p]);
        a.E[p] = E[p];
        a.W0[p] = reinterpret_cast<const u64*>(Y[p]);
        a.B[p] = reinterpret_cast<const u64*>(B[p]);
        a.F[p] = F[p];
        a.Z[p] = reinterpret_cast<u64*>(Z[p]);
        a.C[p] = reinterpret_cast<const u64*>(C[p]);
    }
    a.n = N; a.bs = 1;
    a.M = T; a.N = N; a.K = K;
    a.ldw = K;
    a.error_flag = dev.error;
    cudaError_t err;
    static const comet::BlockIds none = {};
    const int rc = launch_stream(a, none, dev.sm_count, (cudaStream_t)cuda_stream, nullptr, &err);
    if (err != cudaSuccess) cudaGetLastError();
    return rc;
}

extern "C" int comet_static_status(void* cuda_stream) {
    StaticDevice dev;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    int seen = 0;
    cudaError_t err = static_device(&dev);
    if (err == cudaSuccess) err = cudaMemcpyAsync(&seen, dev.error, sizeof(seen), cudaMemcpyDeviceToHost, stream);
    if (err == cudaSuccess) err = cudaStreamSynchronize(stream);
    if (err == cudaSuccess && seen) err = cudaMemsetAsync(dev.error, 0, sizeof(seen), stream);
    if (err != cudaSuccess) {
        cudaGetLastError();
        return COMET_ERR_CUDA;
    }
    return seen ? COMET_ERR_TIMEOUT : COMET_OK;
}

extern "C" int comet_static_inject_timeout(void* cuda_stream) {
    StaticDevice dev;
    if (static_device(&dev) != cudaSuccess || cudaMemsetAsync(dev.error, 1, sizeof(int), (cudaStream_t)cuda_stream) != cudaSuccess) {
        cudaGetLastError();
        return COMET_ERR_CUDA;
    }
    return COMET_OK;
}

// ---------------------------------------------------------------------------
// Oblivious shuffle (Protocol 1), online stage.  Stateless: no context, no
// memory of its own.
// ---------------------------------------------------------------------------
namespace {

int shuffle_grid(long long items) {
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long want = (items + 255) / 256, cap = (long long)sms * 16;
    if (want < 1) want = 1;
    return (int)(want < cap ? want : cap);
}

// A kernel of a call without a context, 256 threads per CTA, chained to the one before it.  Started after its end, the six kernels
// of a shuffle and its way back (512 x 2048) take 51.7 us, chained 36.7.
template <typename... KArgs, typename... Args>
int launch_pass(void (*kernel)(KArgs...), dim3 grid, cudaStream_t stream, Args&&... args) {
    const cudaError_t err = launch_chained(kernel, grid, dim3(256), 0, stream, nullptr, std::forward<Args>(args)...);
    if (err != cudaSuccess) cudaGetLastError();
    return err == cudaSuccess ? COMET_OK : COMET_ERR_CUDA;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// One pass over both steps reads X and a twice, the second time from L2 if they stay there: up to 2^21 words per matrix, when
// the four matrices take half of it.  One pass against two at 512 x 2048: 24 and 30 us, 512 x 4096 (2^21 words): 34 and 37 us,
// 768 x 4096: 52 and 52 us, 1024 x 4096: 70 and 66 us.  A row of one or two words is less than the 32 bytes that a random fetch
// moves, and one pass makes three of those per row instead of two: as long as one round of resident threads covers the rows of
// one word (148 SMs x 1024), and up to 3 x 2^16 rows of two.  151552 x 1: 6.5 and 9.0 us, 156000 x 1 11.5 and 9.1, 2^21 x 1 100 and
// 59; 188000 x 2 8.8 and 9.0, 196608 x 2 10.1 and 9.2, 2^20 x 2 54 and 41.  Rows of three words on: one pass (2^21 words: 46 and 48).
bool shuffle_in_one_pass(int64_t rows, int64_t cols) {
    return rows <= (cols == 1 ? 148 << 10 : cols == 2 ? 3 << 16 : (int64_t)(1 << 21) / cols);
}

// out_i = in_i[perm_i] +/- mask_i for both parties, one launch
int launch_shuffle_step(cudaStream_t stream, const uint64_t* const in[2], const int32_t* const perm[2],
                        const uint64_t* const mask[2], uint64_t* const out[2], int64_t rows, int64_t cols,
                        int subtract, int32_t* bad) {
    comet::ShuffleArgs a;
    bool vec = (cols % 2) == 0;
    for (int p = 0; p < 2; ++p) {
        a.in[p] = reinterpret_cast<const u64*>(in[p]);
        a.perm[p] = perm[p];
        a.mask[p] = reinterpret_cast<const u64*>(mask[p]);
        a.out[p] = reinterpret_cast<u64*>(out[p]);
        vec = vec && aligned16(in[p]) && aligned16(mask[p]) && aligned16(out[p]);
    }
    a.rows = rows;
    a.pieces = (int)(vec ? cols / 2 : cols);
    a.subtract = subtract;
    a.bad_index = bad;
    const int grid = shuffle_grid(rows * a.pieces);
    const long long stride = (long long)grid * 256;
    a.stride_rows = stride / a.pieces;
    a.stride_pieces = (int)(stride % a.pieces);
    return launch_pass(vec ? comet::shuffle_rows_kernel<ulonglong2> : comet::shuffle_rows_kernel<u64>, dim3(grid, 2), stream, a);
}

}  // namespace

extern "C" int comet_shuffle(void* cuda_stream, const uint64_t* const X[2], const int32_t* const tau[2],
                             const int32_t* const rho[2], const uint64_t* const a[2], const uint64_t* const b[2],
                             uint64_t* const Y[2], uint64_t* const Z[2], int64_t rows, int64_t cols,
                             int32_t* bad_index_flag) {
    if (!X || !tau || !rho || !a || !b || !Y || !Z) return COMET_ERR_INVALID_ARG;
    for (int p = 0; p < 2; ++p)
        if (!X[p] || !tau[p] || !rho[p] || !a[p] || !b[p] || !Y[p] || !Z[p]) return COMET_ERR_INVALID_ARG;
    if (rows < 1 || cols < 1 || rows > 0x7fffffffll || cols > 0x7fffffffll) return COMET_ERR_SHAPE;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    if (shuffle_in_one_pass(rows, cols)) {
        comet::ShuffleBothArgs g;
        bool vec = (cols % 2) == 0;
        for (int p = 0; p < 2; ++p) {
            g.x[p] = reinterpret_cast<const u64*>(X[p]);
            g.a[p] = reinterpret_cast<const u64*>(a[p]);
            g.b[p] = reinterpret_cast<const u64*>(b[p]);
            g.y[p] = reinterpret_cast<u64*>(Y[p]);
            g.z[p] = reinterpret_cast<u64*>(Z[p]);
            g.tau[p] = tau[p];
            g.rho[p] = rho[p];
            vec = vec && aligned16(X[p]) && aligned16(a[p]) && aligned16(b[p]) && aligned16(Y[p]) && aligned16(Z[p]);
        }
        g.rows = rows;
        g.pieces = (int)(vec ? cols / 2 : cols);
        g.bad_index = bad_index_flag;
        const int grid = shuffle_grid(rows * g.pieces);
        g.stride_rows = (long long)grid * 256 / g.pieces;
        g.stride_pieces = (int)((long long)grid * 256 % g.pieces);
        auto* kernel = vec ? comet::shuffle_both_kernel<ulonglong2> : comet::shuffle_both_kernel<u64>;
        return launch_pass(kernel, dim3(grid), stream, g);
    }
    // [y]_i = tau_i([x]_i) + a_i
    int rc = launch_shuffle_step(stream, X, tau, a, Y, rows, cols, 0, bad_index_flag);
    if (rc != COMET_OK) return rc;
    // the exchange: party i reads what the other party wrote.  [z]_i = rho_i([y]_other) - b_i
    const uint64_t* const received[2] = {Y[1], Y[0]};
    return launch_shuffle_step(stream, received, rho, b, Z, rows, cols, 1, bad_index_flag);
}

extern "C" int comet_invert_permutation(void* cuda_stream, const int32_t* perm, int32_t* inverse, int64_t rows,
                                        int32_t* bad_index_flag) {
    if (!perm || !inverse) return COMET_ERR_INVALID_ARG;
    if (rows < 1 || rows > 0x7fffffffll) return COMET_ERR_SHAPE;
    return launch_pass(comet::invert_permutation_kernel, dim3(shuffle_grid(rows)), (cudaStream_t)cuda_stream, perm, inverse,
                       (long long)rows, bad_index_flag);
}

// ---------------------------------------------------------------------------
// Element-wise Beaver product (Eq. 1 element by element).  Stateless.
// ---------------------------------------------------------------------------
extern "C" int comet_beaver_mul(void* cuda_stream, const uint64_t* const X[2], const uint64_t* const Y[2],
                                const uint64_t* const A[2], const uint64_t* const B[2], const uint64_t* const C[2],
                                uint64_t* const D[2], uint64_t* const E[2], uint64_t* const Z[2], int64_t count) {
    if (!X || !Y || !A || !B || !C || !D || !E || !Z) return COMET_ERR_INVALID_ARG;
    for (int p = 0; p < 2; ++p)
        if (!X[p] || !Y[p] || !A[p] || !B[p] || !C[p] || !D[p] || !E[p] || !Z[p]) return COMET_ERR_INVALID_ARG;
    if (count < 1) return COMET_ERR_SHAPE;
    comet::MulArgs g;
    bool vec = (count % 2) == 0;
    for (int p = 0; p < 2; ++p) {
        g.x[p] = reinterpret_cast<const u64*>(X[p]); g.y[p] = reinterpret_cast<const u64*>(Y[p]);
        g.a[p] = reinterpret_cast<const u64*>(A[p]); g.b[p] = reinterpret_cast<const u64*>(B[p]);
        g.c[p] = reinterpret_cast<const u64*>(C[p]);
        g.d[p] = reinterpret_cast<u64*>(D[p]); g.e[p] = reinterpret_cast<u64*>(E[p]);
        g.z[p] = reinterpret_cast<u64*>(Z[p]);
        vec = vec && aligned16(X[p]) && aligned16(Y[p]) && aligned16(A[p]) && aligned16(B[p]) && aligned16(C[p]) &&
              aligned16(D[p]) && aligned16(E[p]) && aligned16(Z[p]);
    }
    g.pieces = vec ? count / 2 : count;
    auto* kernel = vec ? comet::beaver_mul_kernel<ulonglong2> : comet::beaver_mul_kernel<u64>;
    return launch_pass(kernel, dim3(shuffle_grid(g.pieces)), (cudaStream_t)cuda_stream, g);
}

// ---------------------------------------------------------------------------
// Truncation with a dealer's pair: Section 2.1's Reconstruction and Addition.
// ---------------------------------------------------------------------------
extern "C" int comet_truncate_pair(void* cuda_stream, uint64_t* const Z[2], const uint64_t* const R[2],
                                   const uint64_t* const RP[2], uint64_t* const M[2], int64_t count,
                                   int32_t frac_bits) {
    if (!Z || !R || !RP || !M) return COMET_ERR_INVALID_ARG;
    for (int p = 0; p < 2; ++p)
        if (!Z[p] || !R[p] || !RP[p] || !M[p]) return COMET_ERR_INVALID_ARG;
    if (count < 1) return COMET_ERR_SHAPE;
    if (frac_bits < 1 || frac_bits > 31) return COMET_ERR_SHAPE;
    comet::TruncPairArgs g;
    bool vec = (count % 2) == 0;
    for (int p = 0; p < 2; ++p) {
        g.z[p] = reinterpret_cast<u64*>(Z[p]); g.m[p] = reinterpret_cast<u64*>(M[p]);
        g.r[p] = reinterpret_cast<const u64*>(R[p]); g.rp[p] = reinterpret_cast<const u64*>(RP[p]);
        vec = vec && aligned16(Z[p]) && aligned16(R[p]) && aligned16(RP[p]) && aligned16(M[p]);
    }
    g.pieces = vec ? count / 2 : count;
    g.f = frac_bits;
    auto* kernel = vec ? comet::trunc_pair_kernel<ulonglong2> : comet::trunc_pair_kernel<u64>;
    return launch_pass(kernel, dim3(shuffle_grid(g.pieces)), (cudaStream_t)cuda_stream, g);
}

// ---------------------------------------------------------------------------
// KV-cache manager (Section 6): request merging and the prefetch rule.  Host logic.
// ---------------------------------------------------------------------------
extern "C" int comet_kv_plan(const uint8_t* present, const uint8_t* active, int32_t tokens, int32_t heads, int64_t x,
                             int64_t w, uint8_t* request, uint8_t* prefetch, int32_t* l1_out) {
    if (!present || !active || !request || !prefetch) return COMET_ERR_INVALID_ARG;
    if (tokens < 1 || heads < 1 || x < 1 || w < 1) return COMET_ERR_SHAPE;
    std::vector<int64_t> missing(heads, 0);
    int32_t l1 = 0;
    for (int32_t t = 0; t < tokens; ++t) {
        bool in_batch = false;
        for (int32_t h = 0; h < heads; ++h) {
            const bool miss = present[(size_t)t * heads + h] == 0;
            missing[h] += miss;
            const bool want = miss && active[h] != 0;
            request[(size_t)t * heads + h] = want ? 1 : 0;
            in_batch = in_batch || want;
        }
        l1 += in_batch;
    }
    for (int32_t h = 0; h < heads; ++h) {
        prefetch[h] = 0;
        if (active[h] != 0) continue;
        const int64_t l2 = missing[h], beyond = l2 > l1 ? l2 - l1 : 0;
        // saved 2*L2*x against spent 2*(w + x*max(0, L2 - L1)), in integers: L2 > w/x + max(0, L2 - L1)
        if (l2 * x > w + x * beyond) {
            prefetch[h] = 1;
            for (int32_t t = 0; t < tokens; ++t)
                if (present[(size_t)t * heads + h] == 0) request[(size_t)t * heads + h] = 1;
        }
    }
    if (l1_out) *l1_out = l1;
    return COMET_OK;
}

extern "C" int comet_add_bias(void* cuda_stream, uint64_t* const Z[2], const uint64_t* const bias[2], int64_t rows,
                              int64_t cols) {
    if (!Z || !bias || !Z[0] || !Z[1] || !bias[0] || !bias[1]) return COMET_ERR_INVALID_ARG;
    if (rows < 1 || cols < 1 || cols > 0x7fffffffll) return COMET_ERR_SHAPE;
    comet::BiasArgs g;
    bool vec = (cols % 2) == 0;
    for (int p = 0; p < 2; ++p) {
        g.z[p] = reinterpret_cast<u64*>(Z[p]);
        g.bias[p] = reinterpret_cast<const u64*>(bias[p]);
        vec = vec && aligned16(Z[p]) && aligned16(bias[p]);
    }
    g.pieces = (int)(vec ? cols / 2 : cols);
    g.total = rows * g.pieces;
    const int grid = shuffle_grid(g.total);
    g.stride_pieces = (int)((long long)grid * 256 % g.pieces);
    auto* kernel = vec ? comet::add_bias_kernel<ulonglong2> : comet::add_bias_kernel<u64>;
    return launch_pass(kernel, dim3(grid), (cudaStream_t)cuda_stream, g);
}

// ---------------------------------------------------------------------------
// Measured peak of a multiply pipe (support for the roofline; not a step of the path).
// ---------------------------------------------------------------------------
extern "C" int comet_pipe_probe(void* cuda_stream, int pipe, int32_t launches, int32_t work, float* ms_out,
                                double* macs_per_launch_out) {
    namespace pk = comet::peak;
    if (!ms_out || !macs_per_launch_out) return COMET_ERR_INVALID_ARG;
    if (pipe != COMET_PIPE_TENSOR_I8 && pipe != COMET_PIPE_ALU_U64) return COMET_ERR_INVALID_ARG;
    if (launches < 1 || launches > 4096 || work < 1 || work > (1 << 24)) return COMET_ERR_SHAPE;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return COMET_ERR_CUDA;
    }
    const int alu_blocks = sms * 2;
    const size_t sink_bytes = pipe == COMET_PIPE_TENSOR_I8 ? (size_t)sms * 32 * sizeof(unsigned) + sizeof(int)
                                                           : (size_t)alu_blocks * pk::ALU_THREADS * sizeof(u64);
    void* sink = nullptr;
    if (cudaMalloc(&sink, sink_bytes) != cudaSuccess) {
        cudaGetLastError();
        return COMET_ERR_OOM;
    }
    std::vector<cudaEvent_t> ev((size_t)launches + 1, nullptr);
    int rc = COMET_OK;
    for (auto& e : ev)
        if (cudaEventCreate(&e) != cudaSuccess) rc = COMET_ERR_CUDA;
    int* flag = reinterpret_cast<int*>(static_cast<char*>(sink) + (size_t)sms * 32 * sizeof(unsigned));
    if (rc == COMET_OK && cudaMemsetAsync(sink, 0, sink_bytes, stream) != cudaSuccess) rc = COMET_ERR_CUDA;
    if (rc == COMET_OK) {
        for (int i = 0; i < launches; ++i) {
            cudaEventRecord(ev[i], stream);
            if (pipe == COMET_PIPE_TENSOR_I8)
                comet::tensor_i8_probe_kernel<<<sms, pk::THREADS, 0, stream>>>(work, 0x9E3779B9u + i, flag,
                                                                                static_cast<unsigned*>(sink));
            else
                comet::alu_u64_probe_kernel<<<alu_blocks, pk::ALU_THREADS, 0, stream>>>(work, 0x9E3779B97F4A7C15ull + i,
                                                                                         static_cast<u64*>(sink));
        }
        cudaEventRecord(ev[launches], stream);
        if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(stream) != cudaSuccess) rc = COMET_ERR_CUDA;
    }
    if (rc == COMET_OK) {
        for (int i = 0; i < launches; ++i)
            if (cudaEventElapsedTime(&ms_out[i], ev[i], ev[i + 1]) != cudaSuccess) rc = COMET_ERR_CUDA;
        if (pipe == COMET_PIPE_TENSOR_I8) {
            int h_flag = 0;
            if (cudaMemcpy(&h_flag, flag, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) rc = COMET_ERR_CUDA;
            else if (h_flag) rc = COMET_ERR_TIMEOUT;
            *macs_per_launch_out = (double)sms * work * pk::BATCH * ((double)pk::M * pk::N * pk::KC);
        } else {
            *macs_per_launch_out = (double)alu_blocks * pk::ALU_THREADS * pk::ALU_CHAINS * (double)work;
        }
    }
    for (auto e : ev)
        if (e) cudaEventDestroy(e);
    cudaFree(sink);
    if (rc == COMET_ERR_CUDA) cudaGetLastError();
    return rc;
}
