// Shared declarations of the cb-DyBW round library: the handle and the host-side launchers
// each translation unit provides.  No device code crosses translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <functional>
#include <mutex>
#include <utility>
#include <vector>

#include "dbw.h"

namespace dbw {

extern std::atomic<long long> g_launches;
extern std::atomic<int> g_last_cuda_error;

inline bool cuda_ok(cudaError_t e) {
    if (e != cudaSuccess) {
        g_last_cuda_error.store((int)e);
        return false;
    }
    return true;
}

#define DBW_CUDA(call)                                  \
    do {                                                \
        if (!::dbw::cuda_ok((call))) return DBW_ERR_CUDA; \
    } while (0)

// Counts a kernel launch and reports a launch-configuration failure.
#define DBW_LAUNCHED()                                         \
    do {                                                       \
        ::dbw::g_launches.fetch_add(1);                        \
        if (!::dbw::cuda_ok(cudaGetLastError())) return DBW_ERR_CUDA; \
    } while (0)

// Launches `kernel`.  EARLY: its blocks may take their places while the kernel before it in the stream is still running
// (programmatic dependent launch), which saves the launch latency between dependent kernels of a few microseconds each; such a
// kernel begins with dependent_begin(), which waits until that kernel has completed and its writes are visible, and then lets
// the next one take its places.  Not for kernels whose blocks are few and long: placed among the blocks of the kernel before,
// they end up several to an SM (32 workers, 784-200-10: the forward GEMM's 256 blocks took 73 us instead of 38).
template <bool EARLY = true, typename... P, typename... A>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = EARLY ? 1 : 0;
    (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(std::forward<A>(args))...);  // an error is the last error, which DBW_LAUNCHED reads
}
__device__ __forceinline__ void dependent_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// One-time set-up per device (kernel attributes, symbol addresses), safe when several host threads
// make the first call at once: `f` runs under the lock until it has succeeded once on that device.
struct PerDeviceOnce {
    std::mutex mu;
    bool done[64] = {};
    template <class F>
    int run(int dev, F&& f) {
        if (dev < 0 || dev >= 64) return DBW_ERR_BAD_SHAPE;
        std::lock_guard<std::mutex> lock(mu);
        if (done[dev]) return DBW_OK;
        const int rc = f();
        if (rc == DBW_OK) done[dev] = true;
        return rc;
    }
};

// Per-round mixing plan (built on the device from kept and b): for each worker the compacted
// list of kept neighbours with their weights, padded to `stride` entries with (self, 0).
struct MixPlan {
    int* idx = nullptr;      // [N][stride]
    float* w = nullptr;      // [N][stride]
    float* w_self = nullptr; // [N]
    int* cnt = nullptr;      // [N]
    int stride = 0;
    int n = 0;                   // N (0 in a default-constructed plan: nothing to check against)
    uint32_t* status = nullptr;  // the handle's status word, for the index checks of the bounds-checked build
};

// Index check of the bounds-checked build (-DDBW_BOUNDS, libdbw_dbg.so): an index outside [0, limit) that a
// kernel read from its own data sets DBW_STATUS_BOUNDS and is replaced by 0, so that the access which follows
// stays inside its array (nothing traps).  The regular build compiles the check away.
__device__ __forceinline__ int checked(int idx, int limit, uint32_t* status) {
#ifdef DBW_BOUNDS
    if (limit > 0 && (idx < 0 || idx >= limit)) {
        if (status) atomicOr(status, DBW_STATUS_BOUNDS);
        return 0;
    }
#endif
    return idx;
}

// Which workers take part in a round (they keep a neighbour or are kept by one), as the selection kernel leaves it on
// the device.  The rows of the others are mixed with nothing: x' = x - lr g is all that happens to them.
struct ActiveRows {
    int* list = nullptr;   // [N] the participants in ascending order
    int* pos = nullptr;    // [N] position of a participant in the list, -1 for the others
    int* slot = nullptr;   // [N][plan.stride] the mixing plan's entries of the participants as list positions
    int* count = nullptr;  // [1]
};
// Up to this many participants the dW GEMMs take the others' step and the mix works on the participants alone; above it
// the round is mixed as a whole.  (Half: x and g of the participants then fit the panel buffer of all rows.)
__host__ __device__ inline int active_limit(int N) { return N / 2; }

struct BF16State;  // tensor-core gradient path (grad_bf16.cu)
struct TcMixState;  // tensor-core mix (mix_tc.cu)
struct SpMixState;  // tensor-core mix with 2:4 structured sparsity (mix_sp.cu)
struct FusedState;  // single-launch round for small networks (round_fused.cu)

}  // namespace dbw

struct dbw_handle {
    int N = 0;
    int64_t d = 0, ld = 0;
    int nnz = 0;
    int maxdeg = 0;
    uint32_t flags = 0;
    int device = 0;
    int sm_count = 0;
    int smem_optin = 0;  // max dynamic shared memory per block

    std::vector<int32_t> h_rowptr, h_col, h_links;  // host copies; links = (u,v) pairs of P
    int32_t* d_rowptr = nullptr;
    int32_t* d_col = nullptr;
    int32_t* d_links = nullptr;  // [2*(N-1)]

    // Algorithm 2 state, device resident: covered[N-1] flags then step counter
    int32_t* d_covered = nullptr;  // [N-1]
    int32_t* d_epoch = nullptr;    // [2]: links covered in this epoch, position of last credited link

    uint32_t* d_status = nullptr;    // [1]
    uint32_t* d_waited = nullptr;    // [N] scratch flags of the selection kernel (kept zero between calls)
    uint32_t* d_ticket = nullptr;    // [1] block ticket of the selection kernel (kept zero between calls)
    int* d_panel_rows = nullptr;     // [1] behind the ticket: rows that mix_pipe_kernel leaves to mix_panel_kernel in this round, all or none
    double* d_Tnbr_ws = nullptr;     // [N]
    dbw::ActiveRows active;          // participants of the round (tensor-core rounds only, allocated with that path)

    const double* t_edge = nullptr;  // optional per-link arrival times (caller-owned, DEVICE, aligned with col)

    dbw::MixPlan plan;
    int mix_panel_cols = 0;  // 0 = automatic
    int panel_per_sm[5] = {}, active_per_sm[5] = {};  // blocks per SM of the panel mix kernels, by panel width; 0 = not asked yet
    dbw::TcMixState* mix_tc = nullptr;  // selection matrix and tensor map of the tensor-core mix (lazy)
    dbw::SpMixState* mix_sp = nullptr;  // 2:4 order, compressed selection matrix and tensor maps of the sparse tensor-core mix (dbw_init)

    dbw::FusedState* fused = nullptr;   // single-launch round (dbw_init)
    int fused_mode = -1;                // -1 = where it is the faster path, 0 = never, 1 = wherever it applies

    // model / gradient path
    bool has_model = false;
    dbw_model_desc model{};
    const float* feat = nullptr;
    const int32_t* labels = nullptr;
    int32_t S = 0;
    float* d_act[DBW_MAX_LAYERS + 1] = {};  // fp32 path: A_0 (gathered batch) .. A_L (logits), [N][B][dims[l]]
    float* d_dz[DBW_MAX_LAYERS + 1] = {};   // fp32 path: dZ_l for l = 1..L, [N][B][dims[l]]
    int32_t* d_ylab = nullptr;              // [N][B] gathered labels
    float* d_head_part = nullptr;           // fp32 path, batches of several parts: [parts][N][fp32_head_partial]
    float* d_G = nullptr;                   // [N][ld] gradient workspace of dbw_round (lazy)
    dbw::BF16State* bf16 = nullptr;
    // bf16 shadow of the parameter matrix, [N][ld], same layout as X (tensor-core path only).  The
    // mix writes it next to X' when parameter tracking is on; the next gradient call then skips the
    // weight cast if it is handed that very X'.
    uint16_t* d_shadow = nullptr;
    bool track_params = false;
    bool shadow_valid = false;
    const float* shadow_of = nullptr;

    // selection of dbw_round runs beside the gradient kernels on this stream (forked from and joined back
    // into the caller's stream by the two events)
    cudaStream_t side = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    cudaEvent_t ev_dz = nullptr, ev_tail = nullptr;  // bf16 gradients: every dZ is there; the batch reductions beside the last GEMM are done
    cudaEvent_t ev_loss = nullptr, ev_read = nullptr;  // dbw_round_host: the losses are there; every result has been copied out

    // stage timing (dbw_profile): events[round][0..5] = start / end of the gradient, selection and mix stages
    bool profiling = false;
    std::vector<cudaEvent_t> prof_events;
    std::vector<cudaEvent_t> prof_gemm_events;  // pairs around every tensor-core GEMM launch while profiling
    int prof_gemm_used = 0;
    std::vector<char> prof_single;  // per recorded round: 1 = single-launch round (events 0 and 1 only)
    int prof_rounds = 0;

    // device staging of dbw_round_host
    double* s_t = nullptr;
    int32_t* s_b = nullptr;
    int32_t* s_bidx = nullptr;
    uint8_t* s_kept = nullptr;
    double* s_Tw = nullptr;
    double* s_Tr = nullptr;
    float* s_loss = nullptr;
};

namespace dbw {

// select.cu
int launch_select(dbw_handle* h, const double* t, const int32_t* b, uint8_t* kept, double* T_worker,
                  double* T_nbr, double* T_round, bool build_plan, cudaStream_t s, bool list_active = false);
int launch_plan_from_kept(dbw_handle* h, const uint8_t* kept, const int32_t* b, cudaStream_t s);

// mix.cu
int launch_mix(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out,
               cudaStream_t s);
// Asks L2 for the line of `p`: nothing waits for it and no register is held; a later load then comes from L2.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// device helper shared by the mix kernels: four floats -> four bf16 (round to nearest even)
__device__ __forceinline__ uint2 pack_bf16x4_rn(float a, float b, float c, float d) {
    uint32_t lo, hi;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(b), "f"(a));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(d), "f"(c));
    return make_uint2(lo, hi);
}
bool mix_panel_fits(const dbw_handle* h);
bool mix_in_place_advised(const dbw_handle* h);
// The mix of a round whose dW GEMMs may already have taken the step x' = x - lr g of every worker that takes no part.
bool mix_active_usable(const dbw_handle* h);
int launch_mix_active(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out, cudaStream_t s);
int mix_kernel_kind(const dbw_handle* h);

// mix_pipe.cu: the panel mix as a pipeline, where that is the faster one
bool mix_pipe_usable(const dbw_handle* h, bool gradient);
long long mix_pipe_kept_limit(const dbw_handle* h, bool gradient);  // 0, or the neighbours kept in all below which the plain one is faster
int launch_mix_pipe(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out, uint16_t* shadow, cudaStream_t s,
                    const int* active_count = nullptr, long long kept_limit = 0);

// mix_staged.cu
bool mix_staged_usable(const dbw_handle* h);
size_t mix_staged_smem(const dbw_handle* h);  // of one block, without the row weights and list lengths it can do without
int launch_mix_staged(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out,
                      uint16_t* shadow, long long kept_limit, cudaStream_t s);

// mix_tc.cu
bool mix_tc_usable(const dbw_handle* h);
bool mix_tc_in_place_ok(const dbw_handle* h);
void mix_tc_free(dbw_handle* h);
int launch_mix_tc(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out,
                  uint16_t* shadow, cudaStream_t s);

// mix_sp.cu
void mix_sp_prepare(dbw_handle* h);
bool mix_sp_usable(const dbw_handle* h);
bool mix_sp_in_place_ok(const dbw_handle* h);
void mix_sp_free(dbw_handle* h);
int launch_mix_sp(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out,
                  uint16_t* shadow, cudaStream_t s);
int mix_sp_order_host(int N, const int32_t* rowptr, const int32_t* col, int32_t* order, int capacity);

// round_fused.cu
void round_fused_prepare(dbw_handle* h);
bool round_fused_usable(const dbw_handle* h);
void round_fused_free(dbw_handle* h);
int launch_round_fused(dbw_handle* h, const float* X, const double* t, const int32_t* b, const int32_t* batch_idx, float lr,
                       const float* lr_pw, float* X_out, uint8_t* kept, double* T_worker, double* T_nbr, double* T_round,
                       float* loss, cudaStream_t s);

// dtur.cu
int launch_update_backups(dbw_handle* h, const double* t, int32_t* b_out, double* theta_out, cudaStream_t s);

// grad_fp32.cu
// fp32 gradient path: the last layer's backward step works on parts of at most kHeadPart samples (a worker's dZ of a part,
// its row offsets and losses lie in shared memory); more than one part leave partial sums that are added in a fixed order.
// Bound by the latency of a block's serial passes, so the part length sets the time: 256 samples give ten workers x batch 1024
// x 256 features 80 blocks and 45 us, or with sixteen lanes to a feature group (fp32_head_slices) 160 and 32 (with the whole batch
// in one block the layer fell back to GEMMs, a loss kernel of a block per worker and a column sum: 230 us).
constexpr int kHeadPart = 256;
__host__ __device__ inline int fp32_head_parts(int B) { return (B + kHeadPart - 1) / kHeadPart; }
inline size_t fp32_head_smem_bytes(int B, int C) {
    const int s = B < kHeadPart ? B : kHeadPart;
    return (size_t)((s * C + 1) & ~1) * 4 + (size_t)s * 12;
}
// floats of one worker's partial sums: dW, db, the bias gradient of the layer before, the loss
__host__ __device__ inline long long fp32_head_partial(int in, int C) { return (long long)C * in + (C + in + 1 + 3) / 4 * 4; }
// Whether the last layer takes the small-output path (at most 32 classes), and whether its rows are 16-byte aligned there.
inline bool fp32_head_usable(const dbw_handle* h) { return h->model.dims[h->model.n_layers] <= 32; }
inline bool fp32_head_aligned(const dbw_handle* h) {
    const dbw_model_desc& m = h->model;
    const int L = m.n_layers;
    return (m.dims[L - 1] & 3) == 0 && (m.w_off[L - 1] & 3) == 0 && (h->ld & 3) == 0 && ((uintptr_t)h->feat & 15) == 0;
}
// Networks that the single launch takes unasked, with a last layer in its two steps (round_fused.cu): samples of all workers in networks of
// one layer (fewer in deeper ones), workers in deeper ones.
constexpr int kSingleLaunchSamples = 2560, kSingleLaunchWorkers = 20;
// Lanes that share a feature group's samples in the last layer's backward step, and the feature groups of a block.  Sixteen instead of
// eight make twice the blocks, each half as long, which pays where the blocks are few and their samples many (us, 8 / 16: 10 workers
// x batch 1024, 256 features 46 / 32, 32 x 64, 200 features 13.4 / 10.3), not where a lane is left with a few samples for as many
// shuffles, nor in the networks that the single launch takes unasked, where its blocks then have a second turn (21 x 57, 784 features, a
// round 31 / 37).  The same for the per-step kernels and the single launch, which sum in this order.
__host__ __device__ constexpr int head_chunk4(int slices) { return 8 * 32 / slices; }
inline int fp32_head_slices(const dbw_handle* h) {
    const int B = h->model.batch, in4 = (h->model.dims[h->model.n_layers - 1] + 3) / 4;
    const long long blocks = (long long)h->N * ((in4 + head_chunk4(8) - 1) / head_chunk4(8)) * fp32_head_parts(B);
    const bool large = (long long)h->N * B > kSingleLaunchSamples || (h->model.n_layers > 1 && h->N > kSingleLaunchWorkers);
    return large && B >= 64 && 2 * blocks <= h->sm_count + h->sm_count / 4 ? 16 : 8;
}
// Slices over k of an fp32 backward GEMM of `batch` problems M x N x K (GemmArgs::slice), the same for the per-step kernels and
// the single launch, which sum in this order.  Forward GEMMs are not sliced: whether a pre-activation of zero up to rounding
// passes its ReLU follows from the order of its sum, which stays ascending in k for every shape.
int fp32_gemm_slice(int M, int N, int K, int batch, bool is_dw, int sm_count);
// Whether a backward fp32 GEMM runs on the tensor cores, each operand value as three bf16 pieces (gemm_split.cuh): the same for both again.
bool fp32_gemm_split(int M, int N, int K, int batch, bool is_dw);
int grad_fp32_alloc(dbw_handle* h);
void grad_fp32_free(dbw_handle* h);
// `beside` (of both gradient paths): queues what runs beside the gradients on another stream; called once the forward pass is
// queued, so that the GPU has work while the host makes those calls.
int launch_grad_fp32(dbw_handle* h, const float* X, const int32_t* batch_idx, float* G, float* loss,
                     cudaStream_t s, const std::function<int()>* beside = nullptr);

// grad_bf16.cu
int grad_bf16_alloc(dbw_handle* h);
void grad_bf16_free(dbw_handle* h);
// The SGD step of the workers that take no part in the round, taken in the epilogue of the dW GEMMs.
struct StepArgs {
    float lr;
    const float* lr_pw;
    float* X_out;
    cudaEvent_t selected;  // the selection (and with it the list of participants) is complete after this event
};
int launch_grad_bf16(dbw_handle* h, const float* X, const int32_t* batch_idx, float* G, float* loss, cudaStream_t s,
                     const StepArgs* step = nullptr, const std::function<int()>* beside = nullptr);

}  // namespace dbw
