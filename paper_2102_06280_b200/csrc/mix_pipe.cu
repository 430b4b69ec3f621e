// The shared-memory panel mix as a pipeline: persistent blocks, whose next column panels of X and G are on their way by TMA while the
// current one is mixed.
//
// The plain panel kernel (mix.cu) loads a panel through registers, then sums its rows, then loads the next: between the two the memory
// system has only what the SM's other blocks ask for (96 workers x 300,007 columns, 6 neighbours: 98 us, 0.54 of the copy
// bandwidth; here 76, 0.70).  Here a ring of panels lies in shared memory, a copy of a whole panel is a few instructions of one
// thread, and the loads in flight need neither registers nor L1.  The mixing plan, which L1 then has no room for, is copied to
// shared memory once per block.  A panel is complete before any of it is written and panels are disjoint, so X' may overwrite X.
// Every output is summed as in the plain kernel: the same bits.  What bounds it is HBM, then the blocks' gather.
#include <cuda.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "round_dev.cuh"
#include "tc_ptx.cuh"

namespace dbw {

namespace {

using namespace dev;
using namespace ptx;

constexpr int kThreads = 512;
constexpr int kMaxStages = 4;
constexpr uint32_t kWaitLimit = 1u << 24;
constexpr int kStaticSmem = 256;  // barriers

enum { NO_GRADIENT = 0, LOCAL_STEP = 1, CORRECTED = 2 };  // x, x - lr g mixed (Algorithm 1's order), x mixed and corrected by the own gradient (Eq. 3's)

struct PipeArgs {
    int N, n_panels, stages, boxes, box_rows;  // a panel is `boxes` TMA boxes of box_rows rows
    long long ld;
    float lr;
    const float* lr_pw;
    float* Xout;
    uint16_t* shadow;
    MixPlan plan;
    const int* active_count;  // nullable: with at most active_limit(N) participants the round is mix_active_kernel's
    long long kept_limit;     // with fewer neighbours kept in all it is mix_panel_kernel's, which is told by the number of rows left to it
    int* panel_rows;
};

__device__ __forceinline__ void load_box(void* dst, const CUtensorMap* map, int c, int row, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)), "l"(map), "r"(c), "r"(row),
                 "r"(smem_u32(bar))
                 : "memory");
}

// Shared memory: the ring of panels, float4 [rows][GS] of x (and of g), then the plan: weights [N][stride], own weights [N], rows [N][stride]
// and counts [N] as 16-bit numbers.
constexpr int even4(int n) { return (n + 3) & ~3; }
constexpr size_t plan_bytes(int N, int stride) { return (size_t)N * (stride * 6 + 2) + (size_t)even4(N) * 4; }

template <int GS, int MODE>
__global__ void __launch_bounds__(kThreads, 2) mix_pipe_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_g, const __grid_constant__ PipeArgs a) {
    dependent_begin();
    extern __shared__ __align__(128) uint8_t pipe_smem[];
    __shared__ uint64_t full[kMaxStages];
    __shared__ uint32_t abort_word;
    volatile uint32_t* abort = &abort_word;
    const int N = a.N, tid = threadIdx.x, stride = a.plan.stride;
    if (a.active_count && *a.active_count <= active_limit(N)) return;
    if (a.kept_limit > 0) {
        const bool mine = keeps_at_least(a.plan, N, a.kept_limit);
        if (blockIdx.x == 0 && tid == 0) *a.panel_rows = mine ? 0 : N;
        if (!mine) return;
    }
    const int matrix = a.boxes * a.box_rows * GS * 16, stage = matrix * (MODE == NO_GRADIENT ? 1 : 2);
    uint8_t* panels = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(pipe_smem) + 127) & ~(uintptr_t)127);
    float* w = reinterpret_cast<float*>(panels + (size_t)a.stages * stage);
    float* w_self = w + (size_t)N * stride;
    uint16_t* rows = reinterpret_cast<uint16_t*>(w_self + ((N + 3) & ~3));
    uint16_t* count = rows + (size_t)N * stride;
    auto load = [&](long long panel, int st) {  // by one thread
        if (panel >= a.n_panels) return;
        mbar_expect_tx(&full[st], (uint32_t)stage);
        for (int b = 0; b < a.boxes; ++b) {
            uint8_t* to = panels + (size_t)st * stage + b * a.box_rows * GS * 16;
            load_box(to, &map_x, (int)panel * (4 * GS), b * a.box_rows, &full[st]);
            if (MODE != NO_GRADIENT) load_box(to + matrix, &map_g, (int)panel * (4 * GS), b * a.box_rows, &full[st]);
        }
    };
    if (tid == 0) {
        *abort = 0u;
        for (int s = 0; s < a.stages; ++s) mbar_init(&full[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int s = 0; s < a.stages; ++s) load(blockIdx.x + (long long)s * gridDim.x, s);
    }
    for (int e = tid; e < N * stride; e += kThreads) {
        w[e] = __ldg(a.plan.w + e);
        rows[e] = (uint16_t)checked(__ldg(a.plan.idx + e), N, a.plan.status);
    }
    for (int e = tid; e < N; e += kThreads) {
        w_self[e] = __ldg(a.plan.w_self + e);
        count[e] = (uint16_t)__ldg(a.plan.cnt + e);
    }
    __syncthreads();
    constexpr int kGroups = kThreads / GS;
    const int q = tid % GS, gid = tid / GS;
    int st = 0;
    uint32_t parity = 0u;
    bool live = true;
    long long panel = blockIdx.x;
    for (; panel < a.n_panels; panel += gridDim.x) {
        const bool there = mbar_wait_bounded<false>(&full[st], parity, kWaitLimit, 0, abort, a.plan.status);
        live = __syncthreads_and(there);
        if (!live) break;  // a wait ran out: leave together
        float4* x = reinterpret_cast<float4*>(panels + (size_t)st * stage);
        const float4* g = reinterpret_cast<const float4*>(panels + (size_t)st * stage + matrix);
        if (MODE == LOCAL_STEP) {
#pragma unroll 4
            for (int e = tid; e < N * GS; e += kThreads) x[e] = fma4(-(a.lr_pw ? __ldg(a.lr_pw + e / GS) : a.lr), g[e], x[e]);
            __syncthreads();
        }
        const long long c = (panel * GS + q) * 4;
        if (c < a.ld) {
            for (int i = gid; i < N; i += kGroups) {
                const float ws = w_self[i];
                const float4 self = x[i * GS + q];
                float4 acc = make_float4(ws * self.x, ws * self.y, ws * self.z, ws * self.w);
                const int cnt = count[i];
                const uint16_t* pj = rows + i * stride;
                const float* pw = w + i * stride;
                for (int k = 0; k < cnt; k += 4) {  // list padding is (own row, weight 0)
                    const ushort4 j = *reinterpret_cast<const ushort4*>(pj + k);
                    const float4 wk = *reinterpret_cast<const float4*>(pw + k);
                    const float4 v0 = x[j.x * GS + q], v1 = x[j.y * GS + q], v2 = x[j.z * GS + q], v3 = x[j.w * GS + q];
                    acc = fma4(wk.x, v0, acc);
                    acc = fma4(wk.y, v1, acc);
                    acc = fma4(wk.z, v2, acc);
                    acc = fma4(wk.w, v3, acc);
                }
                if (MODE == CORRECTED) acc = fma4(-(a.lr_pw ? __ldg(a.lr_pw + i) : a.lr), g[i * GS + q], acc);
                *reinterpret_cast<float4*>(a.Xout + (size_t)i * a.ld + c) = acc;
                if (a.shadow) *reinterpret_cast<uint2*>(a.shadow + (size_t)i * a.ld + c) = pack_bf16x4_rn(acc.x, acc.y, acc.z, acc.w);
            }
        }
        __syncthreads();
        if (tid == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the panel has been read: the next copy may overwrite it
            load(panel + (long long)a.stages * gridDim.x, st);
        }
        if (++st == a.stages) {
            st = 0;
            parity ^= 1u;
        }
    }
    if (!live && tid == 0) {  // copies on their way land before the block leaves
        for (int s = 0; s < a.stages && panel < a.n_panels; ++s, panel += gridDim.x) {
            mbar_wait_quiet<false>(&full[st], parity, 1u << 20);
            if (++st == a.stages) {
                st = 0;
                parity ^= 1u;
            }
        }
    }
}

bool make_map(CUtensorMap* map, const float* base, int N, long long ld, int gs, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)ld, (cuuint64_t)N}, strides[1] = {(cuuint64_t)ld * 4};
    cuuint32_t box[2] = {(cuuint32_t)(4 * gs), (cuuint32_t)box_rows}, estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct Shape {
    int gs = 0, per_sm = 0, stages = 0, boxes = 0, box_rows = 0;
    size_t smem = 0;
};

// Panel width (columns / 4), blocks to an SM and depth of the ring; gs = 0: the plain kernel is the faster one.  Two blocks to an SM with
// panels of 64 columns where they fit, then of 32; wider ones only where a panel would have fewer pieces than a block has threads.
// Measured (us, plain / here, other widths in brackets): 96 workers x 300,007 columns, 6 neighbours 98 / 76 (32 columns 80); 128 x
// 1,000,000, 8 407 / 314 (64 columns, one block 342); 192 x 400,000, 6 244 / 181; 192, 24 neighbours 487 / 370 (32 columns 417); 320 x
// 300,000, 8 386 / 248; 400, 6 482 / 286; 750 x 200,000, 4, no gradient 463 / 235; where
// few are kept see mix_pipe_kept_limit.
// The plain kernel stays where the matrices lie in L2 or the blocks have a turn or two each: filling the ring then costs more than
// it hides (15 x 60,000: 8.0 / 10.6, 96 x 20,000: 11.1 / 12.7, 128 x 50,000: 22.5 / 22.8; 256 x 30,000: 31.8 / 29.1, 400 x 20,000:
// 38.6 / 31.1).
Shape shape_of(const dbw_handle* h, bool gradient) {
    Shape s;
    s.boxes = (h->N + 255) / 256;
    s.box_rows = (h->N + s.boxes - 1) / s.boxes;
    const size_t plan = plan_bytes(h->N, h->plan.stride) + 128 /*align slack*/;
    auto fits = [&](int gs, int per_sm) {
        const size_t stage = (size_t)s.boxes * s.box_rows * gs * 16 * (gradient ? 2 : 1);
        const size_t room = (size_t)h->smem_optin / per_sm - 1024 * (per_sm - 1) - kStaticSmem;
        if (plan + 2 * stage > room) return false;
        s.gs = gs;
        s.per_sm = per_sm;
        s.stages = (int)std::min<size_t>(kMaxStages, (room - plan) / stage);
        s.smem = plan + s.stages * stage;
        return true;
    };
    const int first = h->N >= 32 ? 16 : h->N >= 16 ? 32 : 64;
    if (!fits(first, 2) && !(h->N >= 64 && fits(8, 2)) && !fits(16, 1) && !(h->N >= 64 && fits(8, 1))) return s;
    const long long bytes = (long long)h->N * h->ld * (gradient ? 12 : 8), panels = (h->ld + 4 * s.gs - 1) / (4 * s.gs);
    const bool streams = bytes >= (160ll << 20) || (h->N >= 192 && panels >= 4ll * s.per_sm * h->sm_count);
    if (!streams || panels * (4 * s.gs) > 0x7fffffff) s.gs = 0;  // coordinates are 32-bit numbers
    return s;
}

template <int GS, int MODE>
int launch_pipe(dbw_handle* h, const Shape& sh, const CUtensorMap& mx, const CUtensorMap& mg, const PipeArgs& a, cudaStream_t s) {
    static PerDeviceOnce once;
    const int rc = once.run(h->device, [h]() -> int {
        DBW_CUDA(cudaFuncSetAttribute(mix_pipe_kernel<GS, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, h->smem_optin - kStaticSmem));
        return DBW_OK;
    });
    if (rc) return rc;
    launch<false>(mix_pipe_kernel<GS, MODE>, std::min(a.n_panels, sh.per_sm * h->sm_count), kThreads, sh.smem, s, mx, mg, a);
    DBW_LAUNCHED();
    return DBW_OK;
}

}  // namespace

// Not without the driver's tensor maps, which the plain kernel has no need of.
bool mix_pipe_usable(const dbw_handle* h, bool gradient) { return shape_of(h, gradient).gs != 0 && encode_tiled_fn(); }

// Workers that keep hardly a neighbour leave the plain kernel next to nothing to sum, and its panels are up to four times as wide.  How
// many are kept only the device knows: both kernels are launched then, and the one whose round it is not leaves after a look at the
// plan's counts (5 us in all, so not where a mix is short).  Measured with 0 / 0.25 / 0.5 / 1 kept a worker (us; plain, here alone, both): 94
// workers x 2,504,265 columns 531 530 552 619, 585 585 594 602, 535 533 599 602; 64 x 3,000,000 403 407 428 502, 425 434 432 375, 411
// 420 387 399; 200 x 900,000 423 429 454 494, 454 450 447 446, 427 431 450 446; 128 x 1,000,000 280 281 294 337, 296 297 296 306, 289
// 289 307 310.  With more workers the plain kernel's panels are narrow too (256 x 400,000 231 231 242 274, 234 203 209 231; 320 x
// 600,000 507 525 561 627, 403 424 416 435), and without gradients this kernel is always the faster.
long long mix_pipe_kept_limit(const dbw_handle* h, bool gradient) {
    return gradient && h->N <= 224 && (long long)h->N * h->ld * 12 >= (1ll << 30) ? (h->N + 1) / 2 : 0;
}

int launch_mix_pipe(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out, uint16_t* shadow, cudaStream_t s,
                    const int* active_count, long long kept_limit) {
    const Shape sh = shape_of(h, G != nullptr);
    PipeArgs a{};
    a.N = h->N; a.ld = h->ld; a.lr = lr; a.lr_pw = lr_pw; a.Xout = X_out; a.shadow = shadow; a.plan = h->plan; a.active_count = active_count; a.kept_limit = kept_limit; a.panel_rows = h->d_panel_rows;
    a.n_panels = (int)((h->ld + 4 * sh.gs - 1) / (4 * sh.gs));
    a.stages = sh.stages; a.boxes = sh.boxes; a.box_rows = sh.box_rows;
    CUtensorMap mx{}, mg{};
    if (!make_map(&mx, X, h->N, h->ld, sh.gs, sh.box_rows) || (G && !make_map(&mg, G, h->N, h->ld, sh.gs, sh.box_rows))) return DBW_ERR_CUDA;
    const int mode = !G ? NO_GRADIENT : (h->flags & DBW_ORDER_MIX_THEN_CORRECT) ? CORRECTED : LOCAL_STEP;
    auto of = [&](auto gs) {
        constexpr int GS = decltype(gs)::value;
        return mode == NO_GRADIENT ? launch_pipe<GS, NO_GRADIENT>(h, sh, mx, mg, a, s)
               : mode == CORRECTED ? launch_pipe<GS, CORRECTED>(h, sh, mx, mg, a, s) : launch_pipe<GS, LOCAL_STEP>(h, sh, mx, mg, a, s);
    };
    switch (sh.gs) {
        case 64: return of(std::integral_constant<int, 64>{});
        case 32: return of(std::integral_constant<int, 32>{});
        case 16: return of(std::integral_constant<int, 16>{});
        default: return of(std::integral_constant<int, 8>{});
    }
}

}  // namespace dbw
