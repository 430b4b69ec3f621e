// Masked consensus mix fused with the SGD step (Eqs. 4-5, or Eq. 3 over the kept set).
//
// Panel kernel: a CTA owns a panel of `4*GS` consecutive columns of ALL N rows.  It streams the
// panel of X and G from HBM once (128-bit loads), forms the locally updated rows x - lr*g on
// the fly and parks them in shared memory; then every output row of the panel is a weighted sum
// of shared-memory rows, written once with 128-bit stores.  Each element of X and G is read from
// HBM once and each element of X' is written once (12 bytes per parameter element).  A panel is
// fully staged before any of it is written and panels are disjoint, so X' may overwrite X.
// G == nullptr in any of the kernels means G = 0 (a consensus-only round): nothing of G is read, 8 bytes
// per element.
#include <algorithm>
#include <utility>

#include "common.cuh"
#include "round_dev.cuh"

namespace dbw {

namespace {

constexpr int kMixThreads = 512;

using namespace dev;

template <int GS, bool LOCAL>
__global__ void __launch_bounds__(kMixThreads, 3)
mix_panel_kernel(int N, long long ld, const float* X, const float* __restrict__ G, float lr,
                 const float* __restrict__ lr_pw, float* Xout, uint16_t* __restrict__ shadow, MixPlan plan,
                 int mix_then_correct, int n_panels, const int* active_count) {
    dependent_begin();
    extern __shared__ float4 sm[];  // [N][GS]
    if (active_count && *active_count <= active_limit(N)) return;  // mix_active_kernel's round (mix_pipe_kernel's: no rows left)
    for (int panel = blockIdx.x; panel < n_panels; panel += gridDim.x) {
        mix_panel_body<GS, kMixThreads, true, LOCAL>(panel, sm, N, ld, X, G, lr, lr_pw, Xout, shadow, plan, mix_then_correct);
        __syncthreads();
    }
}

// Fallback for graphs too large for a shared-memory panel: neighbour rows are re-read through L2.
// A work item is one output row of one column panel; a block computes it with consecutive lanes on
// consecutive columns (every neighbour read of a warp is one contiguous 512-byte segment).  Items are
// numbered row-fastest inside a panel and handed out in order, so the blocks that run at the same
// time work on the same column panel, whose X and G segments (N x panel_cols x 8 bytes, sized to a
// small share of L2) are fetched from HBM once and re-read out of L2 by the rows that keep them.  Out of place only.
__global__ void __launch_bounds__(256)
mix_direct_kernel(int N, long long ld, const float* __restrict__ X, const float* __restrict__ G, float lr,
                  const float* __restrict__ lr_pw, float* __restrict__ Xout, uint16_t* __restrict__ shadow,
                  MixPlan plan, int mix_then_correct, int panel_cols, long long n_items, long long kept_limit) {
    if (kept_limit > 0 && keeps_at_least(plan, N, kept_limit)) return;  // mix_staged_kernel's round
    for (long long item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int i = (int)(item % N);
        const long long c = (item / N) * panel_cols + 4 * (long long)threadIdx.x;
        if (c >= ld) continue;
        auto stepped = [&](int r) {
            float4 v = ldg4(X + (size_t)r * ld + c);
            if (G && !mix_then_correct) v = fma4(-(lr_pw ? lr_pw[r] : lr), ldg4(G + (size_t)r * ld + c), v);
            return v;
        };
        const float ws = plan.w_self[i];
        const float4 self = stepped(i);
        float4 acc = make_float4(ws * self.x, ws * self.y, ws * self.z, ws * self.w);
        const int cnt = plan.cnt[i];
        const int* pi = plan.idx + (size_t)i * plan.stride;
        const float* pw = plan.w + (size_t)i * plan.stride;
        int k = 0;
        for (; k + 4 <= cnt; k += 4) {  // four neighbour rows in flight, added in list order
            const float4 v0 = stepped(checked(pi[k], N, plan.status)), v1 = stepped(checked(pi[k + 1], N, plan.status)),
                         v2 = stepped(checked(pi[k + 2], N, plan.status)), v3 = stepped(checked(pi[k + 3], N, plan.status));
            acc = fma4(pw[k], v0, acc);
            acc = fma4(pw[k + 1], v1, acc);
            acc = fma4(pw[k + 2], v2, acc);
            acc = fma4(pw[k + 3], v3, acc);
        }
        for (; k < cnt; ++k) acc = fma4(pw[k], stepped(checked(pi[k], N, plan.status)), acc);
        if (G && mix_then_correct) acc = fma4(-(lr_pw ? lr_pw[i] : lr), ldg4(G + (size_t)i * ld + c), acc);
        *reinterpret_cast<float4*>(Xout + (size_t)i * ld + c) = acc;
        if (shadow) *reinterpret_cast<uint2*>(shadow + (size_t)i * ld + c) = pack_bf16x4_rn(acc.x, acc.y, acc.z, acc.w);
    }
}

// The mix of a tensor-core round in which at most half of the workers take part.  The dW GEMMs have then finished the
// weights of the others (x' = x - lr g in their epilogue); what is left is the participants' weights and every worker's
// biases and last layer.  A panel inside a weight block stages and mixes the participants' rows only, and because those
// are few in most rounds of the threshold rule (a tenth to a third of the workers on average), several neighbouring
// panels are staged together, up to half of the buffer with x and the other half with g: copied asynchronously, every
// load of the panels is in flight at once whatever the registers hold.  A panel that reaches outside the weight blocks
// is mixed as by mix_panel_kernel, without the stores that are already done.
// With more participants the round is mix_panel_kernel's (or mix_pipe_kernel's): both are launched, and the one whose round it is not leaves at
// once (about 2 us; as one kernel for both cases the registers of either spilled: 2.01 ms instead of 1.74 for 128 workers
// x 4.2 million columns with all 8 neighbours kept).
struct WeightBlocks {
    int n;                                             // in ascending column order
    long long lo[DBW_MAX_LAYERS], hi[DBW_MAX_LAYERS];  // column ranges whose non-participants are finished
    int p0[DBW_MAX_LAYERS], p1[DBW_MAX_LAYERS];        // panels that lie inside them
    int outside;                                       // panels that do not
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// Bytes behind the staged rows: for every staged row its offset, worker and panel base, and every worker's list position.
inline size_t active_smem(int N, int gs) { return (size_t)N * gs * 16 + (size_t)N * 14; }

template <int GS>
__global__ void __launch_bounds__(kMixThreads, 3)
mix_active_kernel(int N, long long ld, const float* X, const float* __restrict__ G, float lr, const float* __restrict__ lr_pw,
                  float* Xout, uint16_t* __restrict__ shadow, MixPlan plan, int mix_then_correct, int max_merge,
                  ActiveRows active, const __grid_constant__ WeightBlocks blocks) {
    dependent_begin();
    extern __shared__ float4 sm[];  // [N][GS] staged rows, then by staged row v:
    const int n_act = *active.count;
    const int half = active_limit(N);
    if (n_act > half) return;  // mix_panel_kernel's round
    long long* off = reinterpret_cast<long long*>(sm + (size_t)N * GS);  // its float offset from the panels' first column of row 0
    uint16_t* worker = reinterpret_cast<uint16_t*>(off + N);             // its worker
    uint16_t* first = worker + N;                                        // the first staged row of its panel
    int16_t* pos = reinterpret_cast<int16_t*>(first + N);                // worker -> position among the participants, -1
    const int merge = n_act > 0 ? min(half / n_act, max_merge) : 1;
    for (int e = threadIdx.x; e < N; e += kMixThreads) {
        pos[e] = (int16_t)active.pos[e];
        if (e < merge * n_act) {
            const int sub = e / n_act, r = checked(active.list[e - sub * n_act], N, plan.status);
            off[e] = (long long)r * ld + (long long)sub * (4 * GS);
            worker[e] = (uint16_t)r;
            first[e] = (uint16_t)(sub * n_act);
        }
    }
    __syncthreads();
    constexpr int kGroups = kMixThreads / GS;
    const int q = threadIdx.x % GS, gid = threadIdx.x / GS;
    // the panels outside the weight blocks, all rows: the longest work items first
    int item = blockIdx.x;
    for (; item < blocks.outside; item += gridDim.x) {
        int panel = item;
#pragma unroll
        for (int l = 0; l < DBW_MAX_LAYERS - 1; ++l)
            if (l < blocks.n && panel >= blocks.p0[l]) panel += blocks.p1[l] - blocks.p0[l];
        bool done = false;
        const long long c = ((long long)panel * GS + q) * 4;
#pragma unroll
        for (int l = 0; l < DBW_MAX_LAYERS - 1; ++l) done = done || (l < blocks.n && c >= blocks.lo[l] && c < blocks.hi[l]);
        mix_panel_body<GS, kMixThreads>(panel, sm, N, ld, X, G, lr, lr_pw, Xout, shadow, plan, mix_then_correct,
                                        [&](int i) { return !done || pos[i] >= 0; });
        __syncthreads();
    }
    if (n_act == 0) return;
    // the merged panels of every block
#pragma unroll 1
    for (;; item += gridDim.x) {
        int rest = item - blocks.outside, panel = 0, merged = 0;
#pragma unroll
        for (int l = 0; l < DBW_MAX_LAYERS - 1; ++l) {
            if (l < blocks.n && merged == 0) {
                const int groups = (blocks.p1[l] - blocks.p0[l] + merge - 1) / merge;
                if (rest < groups) {
                    panel = blocks.p0[l] + rest * merge;
                    merged = min(merge, blocks.p1[l] - panel);
                }
                rest -= groups;
            }
        }
        if (merged == 0) break;
        const int V = merged * n_act;
        const long long c = ((long long)panel * GS + q) * 4;
        for (int v = gid; v < V; v += kGroups) {
            cp_async16(&sm[v * GS + q], X + off[v] + c);
            cp_async16(&sm[(half + v) * GS + q], G + off[v] + c);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (!mix_then_correct)
            for (int v = gid; v < V; v += kGroups)  // this thread's own copies
                sm[v * GS + q] = fma4(-(lr_pw ? lr_pw[worker[v]] : lr), sm[(half + v) * GS + q], sm[v * GS + q]);
        __syncthreads();
        for (int v = gid; v < V; v += kGroups) {
            const int i = worker[v];
            const float4* rows = sm + (int)first[v] * GS + q;
            const float ws = plan.w_self[i];
            const float4 self = sm[v * GS + q];
            float4 acc = make_float4(ws * self.x, ws * self.y, ws * self.z, ws * self.w);
            const int cnt = plan.cnt[i];
            const int4* pj = reinterpret_cast<const int4*>(active.slot + (size_t)i * plan.stride);
            const float4* pw = reinterpret_cast<const float4*>(plan.w + (size_t)i * plan.stride);
            for (int k = 0; k < cnt; k += 4) {  // list padding is (own row, weight 0)
                int4 j = __ldg(pj + (k >> 2));
                const float4 w = __ldg(pw + (k >> 2));
                j.x = checked(j.x, n_act, plan.status); j.y = checked(j.y, n_act, plan.status);
                j.z = checked(j.z, n_act, plan.status); j.w = checked(j.w, n_act, plan.status);
                acc = fma4(w.x, rows[j.x * GS], acc);
                acc = fma4(w.y, rows[j.y * GS], acc);
                acc = fma4(w.z, rows[j.z * GS], acc);
                acc = fma4(w.w, rows[j.w * GS], acc);
            }
            if (mix_then_correct) acc = fma4(-(lr_pw ? lr_pw[i] : lr), sm[(half + v) * GS + q], acc);
            const long long at = off[v] + c;
            *reinterpret_cast<float4*>(Xout + at) = acc;
            if (shadow) *reinterpret_cast<uint2*>(shadow + at) = pack_bf16x4_rn(acc.x, acc.y, acc.z, acc.w);
        }
        __syncthreads();
    }
}

int auto_group_size(const dbw_handle* h) {
    if (h->mix_panel_cols < 0) return 0;  // direct kernel forced
    if (h->mix_panel_cols >= 1 && h->mix_panel_cols <= 3) return 0;  // staged / tensor-core kernels forced (handled by the caller)
    if (h->mix_panel_cols) return ((size_t)h->N * h->mix_panel_cols * 4 <= (size_t)h->smem_optin) ? h->mix_panel_cols / 4 : 0;
    // few workers and a matrix that streams from HBM (well beyond L2): 256-column panels (1 KB row segments) while
    // three CTAs still share an SM
    if ((size_t)h->N * 64 * 16 <= (size_t)(h->smem_optin) / 3 - 1024 && (size_t)h->N * h->ld * 4 > ((size_t)256 << 20)) return 64;
    // widest panel whose staging buffer still lets two CTAs share an SM
    const size_t budget = (size_t)(h->smem_optin) / 2 - 1024;
    for (int gs = 32; gs >= 4; gs >>= 1)
        if ((size_t)h->N * gs * 16 <= budget) return gs;
    return ((size_t)h->N * 4 * 16 <= (size_t)h->smem_optin) ? 4 : 0;
}

// Algorithm 1's order as a kernel of its own for graphs of many neighbours: without Eq. 3's gradient the registers go to the rows that
// are summed (1965 workers x 74,459 columns, 60 neighbours: 2823 us against 2957; 303 x 197,748: 878 / 911; within 1 % at up to 12
// neighbours).
bool panel_local(const dbw_handle* h) { return !(h->flags & DBW_ORDER_MIX_THEN_CORRECT) && h->nnz > 12 * h->N; }

// Blocks of the panel kernel that share an SM; asked once per handle and width: N and the flags set it.
template <int GS, bool LOCAL>
int panel_blocks(dbw_handle* h, int* per_sm) {
    static PerDeviceOnce once;
    const int rc = once.run(h->device, [h]() -> int {
        DBW_CUDA(cudaFuncSetAttribute(mix_panel_kernel<GS, LOCAL>, cudaFuncAttributeMaxDynamicSharedMemorySize, h->smem_optin));
        return DBW_OK;
    });
    if (rc) return rc;
    int& known = h->panel_per_sm[GS == 64 ? 4 : GS == 32 ? 3 : GS == 16 ? 2 : GS == 8 ? 1 : 0];
    if (known < 1) DBW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&known, mix_panel_kernel<GS, LOCAL>, kMixThreads, (size_t)h->N * GS * 16));
    *per_sm = known;
    return known < 1 ? DBW_ERR_BAD_SHAPE : DBW_OK;
}

template <int GS, bool LOCAL>
int launch_panel_of(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out, uint16_t* shadow, cudaStream_t s,
                          const int* active_count) {
    const size_t smem = (size_t)h->N * GS * 16;
    int per_sm = 0;
    const int rc = panel_blocks<GS, LOCAL>(h, &per_sm);
    if (rc) return rc;
    const int n_panels = (int)((h->ld + 4 * GS - 1) / (4 * GS)), slots = per_sm * h->sm_count;
    const int mtc = (h->flags & DBW_ORDER_MIX_THEN_CORRECT) ? 1 : 0;
    // Placed early where the blocks fill the chip, or are so short that it does not matter where they lie.  Fewer blocks than
    // that end up several to an SM when they are placed among those of the kernel before (502 workers x 4545 columns, 60
    // neighbours: 75 us early, 51 in order; 1032 x 1196: 141 / 62; up to 256 workers early is the better one, by 1 - 2 us), and so
    // do the blocks with a second panel of two, which counts where rows are many neighbours long (1091 x 10,761, 48 neighbours:
    // 242 early, 209 in order).
    // Not behind mix_pipe_kernel either: the SMs would keep its split between shared memory and L1.
    if (active_count != h->d_panel_rows && (n_panels >= (h->nnz > 12 * h->N ? 2 : 1) * slots || h->N <= 256))
        launch(mix_panel_kernel<GS, LOCAL>, std::min(n_panels, slots), kMixThreads, smem, s, h->N, h->ld, X, G, lr, lr_pw, X_out, shadow, h->plan, mtc, n_panels,
               active_count);
    else
        launch<false>(mix_panel_kernel<GS, LOCAL>, std::min(n_panels, slots), kMixThreads, smem, s, h->N, h->ld, X, G, lr, lr_pw, X_out, shadow, h->plan, mtc, n_panels, active_count);
    DBW_LAUNCHED();
    return DBW_OK;
}

template <int GS>
int launch_panel(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out, uint16_t* shadow, cudaStream_t s,
                 const int* active_count = nullptr) {
    return panel_local(h) ? launch_panel_of<GS, true>(h, X, G, lr, lr_pw, X_out, shadow, s, active_count)
                          : launch_panel_of<GS, false>(h, X, G, lr, lr_pw, X_out, shadow, s, active_count);
}

// 64 columns to a panel instead of 128 where the panels are then walked in fewer turns of all blocks: by a twelfth at least, with more
// than twelve neighbours by two fifths.  As many turns of half the width cost more (rows of 256 bytes instead of 512, the mixing
// plan read twice as often), and two rows to a warp take as long as the longer one, which counts where many are kept and not
// equally many.  Measured with 128 / 64 columns: 96 workers x 300,007 columns (6 turns or 11 halves) 111 / 104 us, 78 x 8372 (1 / 1)
// 10.4 / 7.8, 173 x 166,798 (two blocks an SM, 5 / 6) 125 / 108; 109 x 1,298,095 (23 / 46) 950 / 1397, 116 x 1,614,144 (29 / 57) 2074 /
// 2244, 74 x 660,293 (12 / 24) 138 / 156; 205 x 181,206, 24 to 32 of 32 neighbours kept (5 / 7) 300 / 360.
template <bool LOCAL>
int narrower_panel(dbw_handle* h, bool* narrower) {
    int wide = 0, narrow = 0, rc;
    if ((rc = panel_blocks<32, LOCAL>(h, &wide)) || (rc = panel_blocks<16, LOCAL>(h, &narrow))) return rc;
    auto turns = [h](int cols, int per_sm) { return (((h->ld + cols - 1) / cols) + per_sm * h->sm_count - 1) / (per_sm * h->sm_count); };
    *narrower = 100 * turns(64, narrow) < (h->nnz > 12 * h->N ? 120 : 184) * turns(128, wide);
    return DBW_OK;
}

template <int GS>
int launch_active(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out, uint16_t* shadow,
                  cudaStream_t s) {
    const size_t smem = active_smem(h->N, GS);
    int rc = h->mix_panel_cols == 0 && mix_pipe_usable(h, true) ? launch_mix_pipe(h, X, G, lr, lr_pw, X_out, shadow, s, h->active.count)
                                                                 : launch_panel<GS>(h, X, G, lr, lr_pw, X_out, shadow, s, h->active.count);
    if (rc) return rc;
    static PerDeviceOnce once;
    rc = once.run(h->device, [h]() -> int {
        DBW_CUDA(cudaFuncSetAttribute(mix_active_kernel<GS>, cudaFuncAttributeMaxDynamicSharedMemorySize, h->smem_optin));
        return DBW_OK;
    });
    if (rc) return rc;
    int& per_sm = h->active_per_sm[GS == 64 ? 4 : GS == 32 ? 3 : GS == 16 ? 2 : GS == 8 ? 1 : 0];  // asked once per handle: N sets it
    if (per_sm < 1) DBW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mix_active_kernel<GS>, kMixThreads, smem));
    if (per_sm < 1) return DBW_ERR_BAD_SHAPE;
    const int n_panels = (int)((h->ld + 4 * GS - 1) / (4 * GS));
    WeightBlocks blocks{};
    const dbw_model_desc& m = h->model;
    blocks.n = m.n_layers - 1;
    std::pair<long long, long long> range[DBW_MAX_LAYERS];
    for (int l = 0; l < blocks.n; ++l) range[l] = {m.w_off[l], m.w_off[l] + (long long)m.dims[l] * m.dims[l + 1]};
    std::sort(range, range + blocks.n);
    blocks.outside = n_panels;
    for (int l = 0; l < blocks.n; ++l) {
        blocks.lo[l] = range[l].first;
        blocks.hi[l] = range[l].second;
        blocks.p0[l] = (int)((blocks.lo[l] + 4 * GS - 1) / (4 * GS));
        blocks.p1[l] = std::max(blocks.p0[l], (int)(blocks.hi[l] / (4 * GS)));
        blocks.outside -= blocks.p1[l] - blocks.p0[l];
    }
    const int slots = per_sm * h->sm_count;
    // panels staged together: at least two groups for every resident block, so that the blocks stay evenly loaded
    const int max_merge = std::min(32, std::max(1, n_panels / (2 * slots)));
    launch(mix_active_kernel<GS>, n_panels < slots ? n_panels : slots, kMixThreads, smem, s, h->N, h->ld, X, G, lr, lr_pw, X_out, shadow, h->plan, (h->flags & DBW_ORDER_MIX_THEN_CORRECT) ? 1 : 0, max_merge,
        h->active, blocks);
    DBW_LAUNCHED();
    return DBW_OK;
}

}  // namespace

constexpr bool kSparseByDefault = false;

// The tensor-memory staged kernel takes over when it applies and the plain panel kernel could not keep a 32-column
// (128-byte segment) panel with two CTAs per SM.  Beyond 1024 workers its own panels are narrower too (16 columns, from 2049
// workers 8): measured with 8 neighbours, 1300 workers x 131,072 columns 659 us against 847 (16-column panel kernel), 2048
// workers 968 / 1669, 3000 x 65,536 907 / 1303.  The panel kernel stays better
//  - where two of its CTAs share an SM and the matrix is a fraction of L2 (1100 x 4096: 31 us against 35; x 8192: 51 / 50);
//  - with eight-column panels, weights and eight neighbours or more on a matrix that stays in L2 (2652 x 1507, 8 neighbours: 37
//    against 43; 2922 x 4415, 14 neighbours: 115 / 139; uniform weights 2363 x 2376, 12 neighbours: 58 / 45);
//  - where panel and lists leave L1 hardly a line (crowded), unless panels are wide and the matrix streams from HBM (1019 x
//    10,653, 48 neighbours: 36 / 48; 3049 x 11,692, 20 neighbours: 334 / 366; but 926 x 70,855, 48 neighbours: 910 / 507, and a little
//    less crowded 922 x 13,110: 191 / 150).
// Where no panel of all rows leaves the panel kernel any room, the L2 kernel stays for graphs of few neighbours (3790 x 56,509,
// 2 neighbours: 569 us against 840) and for matrices that do not stream from HBM (4033 x 3563, 4 neighbours: 60 / 93); between the
// two where both apply see kept_decides.
static bool use_staged(const dbw_handle* h) {
    if (!mix_staged_usable(h)) return false;
    if (h->mix_panel_cols == 1) return true;
    if (h->mix_panel_cols != 0) return false;
    const int gs = auto_group_size(h);
    const size_t matrix = (size_t)h->N * h->ld * sizeof(float), MB = (size_t)1 << 20;
    const bool crowded = mix_staged_smem(h) > (size_t)(h->N <= 1024 ? 207 : 200) * 1024;
    if (gs >= 8) return false;
    if (gs == 0) return h->nnz >= 6 * h->N && matrix > 256 * MB;
    if (crowded && (h->N > 2048 || matrix <= 64 * MB)) return false;
    if (h->N <= 1024) return true;
    if (h->N > 2048 && !(h->flags & DBW_WEIGHT_UNIFORM) && h->nnz >= 8 * h->N && matrix <= 64 * MB) return false;
    const bool two_ctas = (size_t)h->N * gs * 16 <= (size_t)h->smem_optin / 2 - 1024;
    return !two_ctas || matrix > 32 * MB;
}

// Workers that keep few neighbours, as in most rounds of the threshold rule, leave the L2 kernel little to read again, while the
// staged kernel moves every row through its narrow panels whatever is kept.  How many are kept only the device knows: where the
// two compete (no panel of all rows fits) both are launched, and the one whose round it is not leaves after a look at the
// plan's counts.  At six a worker and more the staged kernel is the faster one (4065 workers x 40,364 columns, 6 neighbours, few
// kept: 370 us against 720; 3971 x 32,355, all 6 kept: 704 / 633; 3848 x 38,685, 5 kept: 691 / 762).
// Always the L2 kernel's are rounds in Eq. 3's order, whose gradient the staged kernel reads in 32-byte pieces (3811 x 65,782, 6
// neighbours: 1004 against 1330), and rounds without gradients (3818 x 36,482, 12 neighbours: 652 / 907).
static bool kept_decides(const dbw_handle* h) { return h->mix_panel_cols == 0 && auto_group_size(h) == 0; }
static bool direct_always(const dbw_handle* h, const float* G) { return kept_decides(h) && (!G || (h->flags & DBW_ORDER_MIX_THEN_CORRECT)); }

// The tensor-core kernel (dense 0/1 selection product) when asked for and applicable.
static bool use_tc(const dbw_handle* h) { return h->mix_panel_cols == 2 && mix_tc_usable(h); }

// The 2:4 structured-sparse tensor-core kernel: when asked for, or automatically where the staged kernel
// would otherwise run with uniform weights (many workers, many kept neighbours) and a 2:4 order exists.
static bool use_sp(const dbw_handle* h) {
    if (!mix_sp_usable(h)) return false;
    if (h->mix_panel_cols == 3) return true;
    return h->mix_panel_cols == 0 && kSparseByDefault && h->N >= 512 && use_staged(h);
}

bool mix_panel_fits(const dbw_handle* h) {
    if (use_sp(h)) return mix_sp_in_place_ok(h);
    return use_tc(h) ? mix_tc_in_place_ok(h) : (use_staged(h) || auto_group_size(h) != 0);
}
// In place only the staged kernel is left where it would share the rounds with the L2 kernel, so a caller is advised against it.
bool mix_in_place_advised(const dbw_handle* h) { return mix_panel_fits(h) && !(use_staged(h) && kept_decides(h)); }
int mix_kernel_kind(const dbw_handle* h) {
    if (use_sp(h)) return 4;
    if (use_tc(h)) return 3;
    if (use_staged(h)) return kept_decides(h) && (h->flags & DBW_ORDER_MIX_THEN_CORRECT) ? 0 : 2;
    return auto_group_size(h) != 0 ? 1 : 0;
}

// With tensor-core layers and a panel of all workers in shared memory the dW GEMMs can take the step of the workers that
// take no part in the round, whose weights then cross HBM once (read x, write x' and its bf16 copy: 10 bytes an element)
// instead of as a gradient written, read back with x and mixed with nothing (18 bytes).
bool mix_active_usable(const dbw_handle* h) {
    return h->active.list && h->has_model && h->model.n_layers >= 2 && mix_kernel_kind(h) == 1 &&
           active_smem(h->N, auto_group_size(h)) <= (size_t)h->smem_optin;
}

int launch_mix_active(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out, cudaStream_t s) {
    uint16_t* shadow = (h->track_params && h->d_shadow) ? h->d_shadow : nullptr;
    h->shadow_valid = shadow != nullptr;
    h->shadow_of = X_out;
    switch (auto_group_size(h)) {
        case 64: return launch_active<64>(h, X, G, lr, lr_pw, X_out, shadow, s);
        case 32: return launch_active<32>(h, X, G, lr, lr_pw, X_out, shadow, s);
        case 16: return launch_active<16>(h, X, G, lr, lr_pw, X_out, shadow, s);
        case 8: return launch_active<8>(h, X, G, lr, lr_pw, X_out, shadow, s);
        case 4: return launch_active<4>(h, X, G, lr, lr_pw, X_out, shadow, s);
        default: return DBW_ERR_BAD_SHAPE;
    }
}

int launch_mix(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out,
               cudaStream_t s) {
    // With parameter tracking the bf16 shadow of X' is written alongside; any other mix call leaves
    // the shadow stale for the buffer it describes.
    uint16_t* shadow = (h->track_params && h->d_shadow) ? h->d_shadow : nullptr;
    h->shadow_valid = shadow != nullptr;
    h->shadow_of = X_out;
    if (use_sp(h)) return launch_mix_sp(h, X, G, lr, lr_pw, X_out, shadow, s);
    if (use_tc(h)) return launch_mix_tc(h, X, G, lr, lr_pw, X_out, shadow, s);
    long long kept_limit = 0;
    if (use_staged(h) && (X_out == X || !direct_always(h, G))) {
        if (X_out != X && kept_decides(h)) kept_limit = 6ll * h->N;
        const int rc = launch_mix_staged(h, X, G, lr, lr_pw, X_out, shadow, kept_limit, s);
        if (rc || kept_limit == 0) return rc;
    }
    int gs = auto_group_size(h);
    const int* left = nullptr;  // mix_pipe_kernel's word on whether it has left the round to the panel kernel
    if (gs >= 8 && h->mix_panel_cols == 0 && mix_pipe_usable(h, G != nullptr)) {
        const long long limit = mix_pipe_kept_limit(h, G != nullptr);
        const int rc = launch_mix_pipe(h, X, G, lr, lr_pw, X_out, shadow, s, nullptr, limit);
        if (rc || limit == 0) return rc;
        left = h->d_panel_rows;
    }
    if (gs == 32 && h->mix_panel_cols == 0 && h->N >= 64) {
        bool narrower = false;
        const int rc = panel_local(h) ? narrower_panel<true>(h, &narrower) : narrower_panel<false>(h, &narrower);
        if (rc) return rc;
        if (narrower) gs = 16;
    }
    switch (gs) {
        case 64: return launch_panel<64>(h, X, G, lr, lr_pw, X_out, shadow, s, left);
        case 32: return launch_panel<32>(h, X, G, lr, lr_pw, X_out, shadow, s, left);
        case 16: return launch_panel<16>(h, X, G, lr, lr_pw, X_out, shadow, s, left);
        case 8: return launch_panel<8>(h, X, G, lr, lr_pw, X_out, shadow, s, left);
        case 4: return launch_panel<4>(h, X, G, lr, lr_pw, X_out, shadow, s, left);
        default: break;
    }
    if (X_out == X) return DBW_ERR_BAD_SHAPE;
    // panel width: the widest of 1024 / 512 / 256 columns whose X and G segments of all rows stay within
    // 12 MB (measured: a small share of L2 keeps the re-reads hitting while the rest of the grid streams
    // through; 128-column panels leave too few threads per block), and no wider than the matrix needs
    int panel_cols = 1024;
    while (panel_cols > 128 && ((panel_cols > 256 && (long long)h->N * panel_cols * 8 > (12ll << 20)) || panel_cols / 2 >= h->ld)) panel_cols >>= 1;
    const long long n_items = ((h->ld + panel_cols - 1) / panel_cols) * h->N;
    long long blocks = (long long)h->sm_count * (2048 / (panel_cols / 4) > 16 ? 16 : 2048 / (panel_cols / 4));
    if (blocks > n_items) blocks = n_items;
    // In order: its blocks keep their places for the whole launch, and placed among those of the kernel before they end up
    // unevenly spread (4229 workers x 29,718 columns, 48 neighbours: 1790 us, placed early 2810).
    launch<false>(mix_direct_kernel, (int)blocks, panel_cols / 4, 0, s, h->N, h->ld, X, G, lr, lr_pw, X_out, shadow, h->plan,
                  (h->flags & DBW_ORDER_MIX_THEN_CORRECT) ? 1 : 0, panel_cols, n_items, kept_limit);
    DBW_LAUNCHED();
    return DBW_OK;
}

}  // namespace dbw
