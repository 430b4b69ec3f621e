// Mix kernel for many workers and many terms per output: one persistent CTA per
// SM, warp-specialised, with the NEXT column panel prefetched into tensor memory.
//
// With N of the order of 1000 a 32-column panel of all rows (N x 128 B; beyond 1024 rows 16 columns, beyond 2048 eight) plus
// the neighbour lists
// fill shared memory, so there is no room for a second panel buffer, and with about 30 terms per
// output the gather out of shared memory takes longer than the HBM stream.  To overlap the two,
// eight producer warps stream the next panel of X and G from HBM (128-bit loads, x - lr*g formed
// in registers) and park it in the SM's tensor memory with tcgen05.st, while twenty-four consumer
// warps gather the current panel out of shared memory (the gather waits on shared-memory round
// trips, so it wants every warp the SM can hold).  When both are done the producers move the parked
// panel from tensor memory into shared memory (tcgen05.ld + 128-bit shared stores) and the roles
// repeat.  The neighbour lists (16-bit entries built once per launch from the mixing plan: a bare row
// index with uniform weights, an index and a weight code with the Metropolis weights) stay
// in shared memory for the whole launch.  HBM traffic is the algorithmic 12 bytes per element; a panel
// is fully staged before any of it is written and panels are disjoint, so X' may overwrite X.
#include "common.cuh"
#include "round_dev.cuh"

namespace dbw {

namespace {

constexpr int kWarps = 32, kThreads = kWarps * 32;
// Producer warps; the others are consumers.  Eight-column panels have little to gather and 32-byte row segments to fetch.
__host__ __device__ constexpr int producer_warps(int W) { return W == 8 ? 16 : 8; }
constexpr int kTmemCols = 256;                            // 128 lanes x 256 columns x 4 B = one 1024 x 32 panel
constexpr int kMaxN = 4096;
// Columns of a panel: the widest whose panel of all rows fits the 128 KB of tensor memory and shared memory it is given.
__host__ __device__ constexpr int staged_width(int N) { return N <= 1024 ? 32 : N <= 2048 ? 16 : 8; }
// Bits of a list entry that hold the row index; with weighted lists the rest of its 16 bits is the weight code.
__host__ __device__ constexpr int index_bits(int W) { return W == 32 ? 10 : W == 16 ? 11 : 12; }
__host__ __device__ constexpr int zero_code(int W) { return (1 << (16 - index_bits(W))) - 1; }  // code of list padding: weight 0
// 16-bit entries of a row's neighbour list: blocks of four.  Rows lie without a gap, so that at some degrees the rows that a warp reads
// together share banks: with 32 neighbours (64 bytes a row) 6 % of the shared-memory wavefronts are conflicts, with weights 8 %.
__host__ __device__ constexpr int list_entries(int maxdeg) { return maxdeg < 4 ? 4 : (maxdeg + 3) / 4 * 4; }

// 1 / (1 + m) for the weight codes m of the weighted lists (Assumption 1: the weight worker i puts on a kept neighbour j is
// 1 / (1 + max(p_i, p_j))), the same fp32 quotient the mixing plan holds.
__constant__ float c_weight[64] = {
    1.0f / 1,  1.0f / 2,  1.0f / 3,  1.0f / 4,  1.0f / 5,  1.0f / 6,  1.0f / 7,  1.0f / 8,  1.0f / 9,  1.0f / 10, 1.0f / 11,
    1.0f / 12, 1.0f / 13, 1.0f / 14, 1.0f / 15, 1.0f / 16, 1.0f / 17, 1.0f / 18, 1.0f / 19, 1.0f / 20, 1.0f / 21, 1.0f / 22,
    1.0f / 23, 1.0f / 24, 1.0f / 25, 1.0f / 26, 1.0f / 27, 1.0f / 28, 1.0f / 29, 1.0f / 30, 1.0f / 31, 1.0f / 32, 1.0f / 33,
    1.0f / 34, 1.0f / 35, 1.0f / 36, 1.0f / 37, 1.0f / 38, 1.0f / 39, 1.0f / 40, 1.0f / 41, 1.0f / 42, 1.0f / 43, 1.0f / 44,
    1.0f / 45, 1.0f / 46, 1.0f / 47, 1.0f / 48, 1.0f / 49, 1.0f / 50, 1.0f / 51, 1.0f / 52, 1.0f / 53, 1.0f / 54, 1.0f / 55,
    1.0f / 56, 1.0f / 57, 1.0f / 58, 1.0f / 59, 1.0f / 60, 1.0f / 61, 1.0f / 62, 1.0f / 63, 0.0f};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float4 (&v)[4]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "f"(v[0].x), "f"(v[0].y), "f"(v[0].z), "f"(v[0].w), "f"(v[1].x), "f"(v[1].y), "f"(v[1].z), "f"(v[1].w),
        "f"(v[2].x), "f"(v[2].y), "f"(v[2].z), "f"(v[2].w), "f"(v[3].x), "f"(v[3].y), "f"(v[3].z), "f"(v[3].w)
        : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float4 (&v)[4]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[0].z), "=f"(v[0].w), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[1].z), "=f"(v[1].w),
          "=f"(v[2].x), "=f"(v[2].y), "=f"(v[2].z), "=f"(v[2].w), "=f"(v[3].x), "=f"(v[3].y), "=f"(v[3].z), "=f"(v[3].w)
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ float4 ldg4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
// The same with the whole 128-byte line asked of L2: the blocks of the neighbouring panels read the rest of it.
__device__ __forceinline__ float4 ldg4_line(const float* p) {
    float4 v;
    asm("ld.global.nc.L2::128B.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ void add4(float4& a, const float4 v) {
    a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
}
__device__ __forceinline__ void fma4(float4& a, const float w, const float4 v) {
    a.x = fmaf(w, v.x, a.x); a.y = fmaf(w, v.y, a.y); a.z = fmaf(w, v.z, a.z); a.w = fmaf(w, v.w, a.w);
}
__device__ __forceinline__ float4 mul4(const float4 v, const float w) { return make_float4(w * v.x, w * v.y, w * v.z, w * v.w); }

struct StagedArgs {
    int N, n_panels, mix_then_correct, list_row;  // list_row: 16-bit entries per neighbour-list row (multiple of 4)
    long long ld;
    const float* X;
    const float* G;
    float lr;
    const float* lr_pw;
    float* Xout;
    uint16_t* shadow;
    MixPlan plan;
    long long kept_limit;  // 0, or the kept entries of the round from which on it is this kernel's
};

// Shared memory: panel float4 [N + 1][W / 4] (row N is all zero: the target of list padding), then the neighbour lists
// uint16 [N][list_row], 64 weights, and LOCAL: every row's own weight or scale, float [N], and list length in blocks of 4,
// uint8 [N].  What a block leaves of the SM's 256 KB is L1, whose lines the loads on their way need, so those two stay in global
// memory where they would make it the smallest (kRoomyBytes): 4096 workers, 65,536 columns, 8 neighbours 1348 us with 197 KB of
// shared memory, 1709 with 217.  Where there is room they are better local: 3000 workers 878 us against 931.
constexpr size_t kRoomyBytes = 195 * 1024;
// WEIGHTED = false: uniform weights, a list entry is a bare 16-bit row index and the sum is scaled once per row.
// WEIGHTED = true: a list entry is a row index and a weight code; padding is (own row, weight 0).
// LPR lanes share an output row.  With weights and 128-byte rows there are four, each lane with two 16-byte pieces: two rows to
// a quarter-warp phase of a 128-bit shared load, the odd groups of lanes reading the second half first so that the two never
// share a bank.  A list or weight read then serves eight rows instead of four (1418 us against 1632 for 1024 workers x 262,144
// columns, 32 neighbours).  Without weight reads eight lanes of one piece are better (1254 us against 1288).
template <bool WEIGHTED, int W, bool LOCAL>
__global__ void __launch_bounds__(kThreads, 1) mix_staged_kernel(StagedArgs a) {
    dependent_begin();
    constexpr int SLOTS = W / 4, PIECES = W == 32 && WEIGHTED ? 2 : 1, LPR = SLOTS / PIECES, RPW = 32 / LPR;  // RPW: output rows per warp
    constexpr uint32_t kIdx = WEIGHTED ? (1u << index_bits(W)) - 1 : 0xffffu;
    constexpr int kProdWarps = producer_warps(W), kConsWarps = kWarps - kProdWarps;
    constexpr int kCodeShift = index_bits(W), ZERO = zero_code(W);
    extern __shared__ float4 smem4[];
    float4* panel = smem4;
    const int N = a.N;
    if (a.kept_limit > 0 && !dev::keeps_at_least(a.plan, N, a.kept_limit)) return;  // mix_direct_kernel's round
    const int lrow = a.list_row;
    uint16_t* lists = reinterpret_cast<uint16_t*>(panel + (size_t)(N + 1) * SLOTS);
    float* wtab = reinterpret_cast<float*>(lists + (size_t)N * lrow);  // weights by code (weighted lists)
    float* scale = wtab + 64;
    uint8_t* nblk = reinterpret_cast<uint8_t*>(scale + N);
    __shared__ uint32_t tmem_slot;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // neighbour lists, scales and the zero row: once per launch
    for (int e = tid; e < N * (lrow / 4); e += kThreads) {
        const int i = e / (lrow / 4), k0 = (e % (lrow / 4)) * 4;
        const int cnt = a.plan.cnt[i];
        auto entry = [&](int k) -> uint32_t {
            if (!WEIGHTED) return k < cnt ? (uint32_t)checked(a.plan.idx[(size_t)i * a.plan.stride + k], N, a.plan.status) : (uint32_t)N;
            if (k >= cnt) return (uint32_t)i | ((uint32_t)ZERO << kCodeShift);
            // the plan's weight is 1 / (1 + m): recover m (exact for m <= 62) and keep it as the code
            const int m = __float2int_rn(1.0f / a.plan.w[(size_t)i * a.plan.stride + k]) - 1;
            return (uint32_t)checked(a.plan.idx[(size_t)i * a.plan.stride + k], N, a.plan.status) | ((uint32_t)min(max(m, 0), ZERO - 1) << kCodeShift);
        };
        *reinterpret_cast<uint2*>(lists + (size_t)i * lrow + k0) =
            make_uint2(entry(k0) | (entry(k0 + 1) << 16), entry(k0 + 2) | (entry(k0 + 3) << 16));
    }
    for (int i = tid; LOCAL && i < N; i += kThreads) {
        scale[i] = a.plan.w_self[i];
        nblk[i] = (uint8_t)max((a.plan.cnt[i] + 3) / 4, 1);
    }
    if (WEIGHTED && tid <= ZERO) wtab[tid] = tid == ZERO ? 0.f : c_weight[tid];
    if (tid < SLOTS) panel[(size_t)N * SLOTS + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_slot;

    constexpr int RPS = 32 / SLOTS;                      // rows a producer warp stages per instruction
    constexpr int IT_ROWS = kProdWarps * RPS;            // rows the producer warps stage per iteration: N needs at most 32
    const int n_its = (N + IT_ROWS - 1) / IT_ROWS;
    const bool producer = warp < kProdWarps;
    // producer coordinates: row (within an iteration) and 16-byte slot of the row segment
    const int p_row = warp * RPS + lane / SLOTS, slot = lane % SLOTS;
    const uint32_t p_taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * (kTmemCols / (kProdWarps / 4)));
    // consumer coordinates: groups of LPR lanes, each owns rows grp, grp + kRowsPar, ...
    constexpr int kRowsPar = kConsWarps * RPW;
    const int grp = (warp - kProdWarps) * RPW + lane / LPR;

    auto stage = [&](int pn) {  // HBM -> registers -> tensor memory
        const long long c = (long long)pn * W + 4 * slot;
        const bool c_ok = c < a.ld;
        for (int bt = 0; bt < n_its; bt += 4) {
            float4 x[4], g[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = (bt + u) * IT_ROWS + p_row;
                const bool ok = c_ok && r < N;
                x[u] = ok ? (W < 32 ? ldg4_line(a.X + (size_t)r * a.ld + c) : ldg4(a.X + (size_t)r * a.ld + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            if (a.G && !a.mix_then_correct) {  // G == nullptr: consensus-only round, G = 0
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int r = (bt + u) * IT_ROWS + p_row;
                    const bool ok = c_ok && r < N;
                    g[u] = ok ? (W < 32 ? ldg4_line(a.G + (size_t)r * a.ld + c) : ldg4(a.G + (size_t)r * a.ld + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int r = (bt + u) * IT_ROWS + p_row;
                    const float nlr = -((a.lr_pw && r < N) ? a.lr_pw[r] : a.lr);
                    x[u].x = fmaf(nlr, g[u].x, x[u].x);
                    x[u].y = fmaf(nlr, g[u].y, x[u].y);
                    x[u].z = fmaf(nlr, g[u].z, x[u].z);
                    x[u].w = fmaf(nlr, g[u].w, x[u].w);
                }
            }
            tmem_st16(p_taddr + (uint32_t)(4 * bt), x);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    };
    auto unpark = [&]() {  // tensor memory -> shared-memory panel
        for (int bt = 0; bt < n_its; bt += 4) {
            float4 x[4];
            tmem_ld16(p_taddr + (uint32_t)(4 * bt), x);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = (bt + u) * IT_ROWS + p_row;
                if (r < N) panel[(size_t)r * SLOTS + slot] = x[u];
            }
        }
    };
    auto gather = [&](int pn) {  // every output row of the panel out of shared memory
        // this lane's pieces of a row: 16-byte slots piece[0], piece[1]
        int piece[PIECES];
        piece[0] = lane % LPR;
        if (PIECES == 2) {
            const int odd = (lane / LPR) & 1;
            piece[PIECES - 1] = piece[0] + LPR * (1 - odd);
            piece[0] += LPR * odd;
        }
        // Flattened loop over (row, list block) with the NEXT block's entries fetched before the current block's rows are
        // gathered, so that no shared-memory round trip sits between two gathers.
        int i = grp;
        if (i >= N) return;
        const uint2* lp = reinterpret_cast<const uint2*>(lists + (size_t)i * lrow);
        auto blocks_of = [&](int row) -> int { return LOCAL ? nblk[row] : max((__ldg(a.plan.cnt + row) + 3) / 4, 1); };
        auto self_weight = [&](int row) { return LOCAL ? scale[row] : __ldg(a.plan.w_self + row); };
        int nb = blocks_of(i), kb = 0;  // a row without kept neighbours gathers one block
        float ws = self_weight(i);
        uint2 u = lp[0];
        float4 acc[PIECES];
        auto first = [&](int row, float4 (&q)[PIECES]) {  // uniform: the own row, scaled with the sum at the end; weighted: own weight x own row
#pragma unroll
            for (int h = 0; h < PIECES; ++h) {
                q[h] = panel[(size_t)row * SLOTS + piece[h]];
                if (WEIGHTED) q[h] = mul4(q[h], ws);
            }
        };
        first(i, acc);
        while (true) {
            const bool last = kb + 1 >= nb;
            const int i2 = i + kRowsPar;
            const bool more = !last || i2 < N;
            const uint2* lp2 = last ? reinterpret_cast<const uint2*>(lists + (size_t)i2 * lrow) : lp;
            uint2 un = u;
            if (more) un = lp2[last ? 0 : kb + 1];
            const uint32_t e[4] = {u.x & 0xffffu, u.x >> 16, u.y & 0xffffu, u.y >> 16};
            float4 v[4][PIECES];
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int h = 0; h < PIECES; ++h) v[k][h] = panel[(size_t)(e[k] & kIdx) * SLOTS + piece[h]];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (!WEIGHTED) {
#pragma unroll
                    for (int h = 0; h < PIECES; ++h) add4(acc[h], v[k][h]);
                } else {  // weights out of a table in shared memory, list order
                    const float w = wtab[e[k] >> kCodeShift];
#pragma unroll
                    for (int h = 0; h < PIECES; ++h) fma4(acc[h], w, v[k][h]);
                }
            }
            u = un;
            if (!last) {
                ++kb;
                continue;
            }
#pragma unroll
            for (int h = 0; h < PIECES; ++h) {
                const long long c = (long long)pn * W + 4 * piece[h];
                float4 o = WEIGHTED ? acc[h] : mul4(acc[h], ws);
                if (c < a.ld) {
                    if (a.G && a.mix_then_correct) {
                        const float4 gi = ldg4(a.G + (size_t)i * a.ld + c);
                        const float nlr = -(a.lr_pw ? a.lr_pw[i] : a.lr);
                        o.x = fmaf(nlr, gi.x, o.x); o.y = fmaf(nlr, gi.y, o.y);
                        o.z = fmaf(nlr, gi.z, o.z); o.w = fmaf(nlr, gi.w, o.w);
                    }
                    *reinterpret_cast<float4*>(a.Xout + (size_t)i * a.ld + c) = o;
                    if (a.shadow) *reinterpret_cast<uint2*>(a.shadow + (size_t)i * a.ld + c) = pack_bf16x4_rn(o.x, o.y, o.z, o.w);
                }
            }
            if (i2 >= N) break;
            i = i2;
            lp = lp2;
            nb = blocks_of(i);
            ws = self_weight(i);
            kb = 0;
            first(i, acc);
        }
    };

    for (int pn = blockIdx.x, prev = -1; prev >= 0 || pn < a.n_panels; prev = pn < a.n_panels ? pn : -1, pn += gridDim.x) {
        if (producer) {
            if (pn < a.n_panels) stage(pn);
        } else if (prev >= 0) {
            gather(prev);
        }
        __syncthreads();  // the previous panel consumed, the next one parked
        if (pn >= a.n_panels) break;
        if (producer) unpark();
        __syncthreads();  // the next panel in shared memory
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

size_t staged_smem(const dbw_handle* h, bool local) {
    const size_t N = (size_t)h->N;
    return (N + 1) * (size_t)(staged_width(h->N) * 4) + N * (size_t)list_entries(h->maxdeg) * 2 + 256 + (local ? (N * 5 + 15) / 16 * 16 : 0);
}
bool staged_local(const dbw_handle* h) { return staged_smem(h, true) <= kRoomyBytes && list_entries(h->maxdeg) <= 4 * 255; }

template <bool WEIGHTED, int W, bool LOCAL>
int launch_staged(const dbw_handle* h, StagedArgs& a, cudaStream_t s) {
    static PerDeviceOnce once;
    const int rc = once.run(h->device, [h]() -> int {
        DBW_CUDA(cudaFuncSetAttribute(mix_staged_kernel<WEIGHTED, W, LOCAL>, cudaFuncAttributeMaxDynamicSharedMemorySize, h->smem_optin - 256));
        return DBW_OK;
    });
    if (rc) return rc;
    a.n_panels = (int)((h->ld + W - 1) / W);
    const int grid = a.n_panels < h->sm_count ? a.n_panels : h->sm_count;
    launch<false>(mix_staged_kernel<WEIGHTED, W, LOCAL>, grid, kThreads, staged_smem(h, LOCAL), s, a);
    DBW_LAUNCHED();
    return DBW_OK;
}

template <int W>
int launch_staged_width(const dbw_handle* h, StagedArgs& a, cudaStream_t s) {
    const bool uniform = (h->flags & DBW_WEIGHT_UNIFORM) != 0;
    if (staged_local(h)) return uniform ? launch_staged<false, W, true>(h, a, s) : launch_staged<true, W, true>(h, a, s);
    return uniform ? launch_staged<false, W, false>(h, a, s) : launch_staged<true, W, false>(h, a, s);
}

}  // namespace

// Usable when a panel of all rows and the lists fit; with uniform weights a list entry is a bare 16-bit index (one scale per
// row), with the Metropolis weights it carries a weight code next to the index (degrees up to 62, 30 or 14).
bool mix_staged_usable(const dbw_handle* h) {
    if (h->N > kMaxN || h->N < 64) return false;
    if (!(h->flags & DBW_WEIGHT_UNIFORM) && h->maxdeg > zero_code(staged_width(h->N)) - 1) return false;
    return staged_smem(h, false) + 256 <= (size_t)h->smem_optin;
}

size_t mix_staged_smem(const dbw_handle* h) { return staged_smem(h, false); }

int launch_mix_staged(dbw_handle* h, const float* X, const float* G, float lr, const float* lr_pw, float* X_out,
                      uint16_t* shadow, long long kept_limit, cudaStream_t s) {
    StagedArgs a{};
    a.N = h->N;
    a.ld = h->ld;
    a.mix_then_correct = (h->flags & DBW_ORDER_MIX_THEN_CORRECT) ? 1 : 0;
    const int W = staged_width(h->N);
    a.list_row = list_entries(h->maxdeg);
    a.X = X; a.G = G; a.lr = lr; a.lr_pw = lr_pw; a.Xout = X_out; a.shadow = shadow; a.plan = h->plan;
    a.kept_limit = kept_limit;
    switch (W) {
        case 32: return launch_staged_width<32>(h, a, s);
        case 16: return launch_staged_width<16>(h, a, s);
        default: return launch_staged_width<8>(h, a, s);
    }
}

}  // namespace dbw
