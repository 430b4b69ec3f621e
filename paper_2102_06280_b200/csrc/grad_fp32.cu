// Mini-batch stochastic gradient (Eq. 2) of the ReLU MLP with softmax cross-entropy in fp32, for all
// workers at once: every kernel is batched over workers (blockIdx.z), whose weights are slices of their
// rows of X.  On the CUDA cores, but for backward GEMMs of many multiply-adds, which run on the tensor
// cores at fp32 precision (gemm_split.cuh).
#include "common.cuh"
#include "gemm_split.cuh"
#include "round_dev.cuh"

namespace dbw {

namespace {

using namespace dev;

// ------------------------------------------------------------------ kernels (bodies in round_dev.cuh)
// EARLY: placed while the kernel before runs, which costs every block two instructions of its own (28,000 blocks of 32 features: a
// call 12 us longer than with a plain launch).  So only where all blocks are placed at once (launch_grad_fp32).
template <bool EARLY>
__global__ void gather_batch_kernel(int B, int S, int in_dim, int C, const float* __restrict__ feat,
                                    const int32_t* __restrict__ labels, const int32_t* __restrict__ batch_idx,
                                    float* __restrict__ A0, int32_t* __restrict__ ylab, uint32_t* status) {
    if (EARLY) dependent_begin();
    gather_row(blockIdx.x, blockIdx.y, B, S, in_dim, C, feat, labels, batch_idx, A0, ylab, status);
}

template <int R, int TK>
__global__ void __launch_bounds__(256) gemm_simt_kernel(GemmArgs g) {
    constexpr int T = 16 * R;
    __shared__ __align__(16) float As[TK][T + 4];
    __shared__ __align__(16) float Bs[TK][T + 4];
    gemm_tile<R, TK>(g, blockIdx.z, blockIdx.y * T, blockIdx.x * T, As, Bs);
}

__global__ void __launch_bounds__(256)
softmax_ce_kernel(int B, int C, const float* __restrict__ logits, const int32_t* __restrict__ ylab,
                  float* dz, float* __restrict__ loss, float* __restrict__ G, long long ld, long long b_off) {
    __shared__ float sl[8];
    softmax_ce_worker(blockIdx.x, B, C, logits, ylab, dz, loss, G, ld, b_off, sl);
}

__global__ void bias_grad_kernel(int B, int out_dim, const float* __restrict__ dz, float* __restrict__ G,
                                 long long ld, long long b_off) {
    bias_grad_col<false>(blockIdx.y, blockIdx.x * blockDim.x + threadIdx.x, B, out_dim, dz, G, ld, b_off, B);
}

// The GEMM for operands whose unit-stride dimension allows 128-bit accesses (every layer whose width and
// batch are multiples of four).  A CTA of WM warps owns a tile of 2 RM WM x 64 outputs; a warp owns 2 RM rows x 64
// columns of it as RM x 4 per thread (RM = 8 or 4; lane / 16 picks the row half, lane mod 16 the columns), so that per
// k a warp reads RM + 4 floats through 128-bit shared-memory loads of which the row loads are broadcasts:
// with RM = 8, 32 multiply-adds per thread for about four shared-memory wavefronts per warp, where the
// 4 x 4 layout of gemm_simt_kernel needs the same four wavefronts for 16.  Global loads and stores are
// 128-bit along the operand's unit-stride dimension.  Every output element is summed over k in ascending
// order, exactly as in gemm_simt_kernel: the two give the same bits.
// SUMS: the blocks of the first columns also add every row of A over k (g.rowsum): the bias gradient of a dW GEMM.
template <int WM, int RM, bool SUMS>
__global__ void __launch_bounds__(32 * WM) gemm_vec_kernel(GemmArgs g) {
    dependent_begin();
    constexpr int BM = 2 * RM * WM, BN = 64, TK = 16, THREADS = 32 * WM;
    constexpr int PA = BM * TK / 4 / THREADS, PB = BN * TK / 4 / THREADS;  // float4 per thread and k-step
    __shared__ __align__(16) float As[TK][BM + 4];
    __shared__ __align__(16) float Bs[TK][BN + 4];
    const int z = blockIdx.z, m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const float* __restrict__ A = g.A + (size_t)z * g.sAz;
    const float* __restrict__ B = g.B + (size_t)z * g.sBz;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int mw = warp * 2 * RM + (lane >> 4) * RM, nw = (lane & 15) * 4;
    const bool a_k_fast = g.sAk == 1, b_k_fast = g.sBk == 1;
    float acc[RM][4] = {};
    const bool sums = SUMS && n0 == 0 && tid < BM;
    float rowsum = 0.f;
    float4 pa[PA], pb[PB];
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](int k0) {
#pragma unroll
        for (int r = 0; r < PA; ++r) {
            const int e = tid + r * THREADS;
            if (a_k_fast) {  // four consecutive k of row e / 4
                const int m = m0 + (e >> 2), k = k0 + 4 * (e & 3);
                pa[r] = (m < g.M && k < g.K) ? __ldg(reinterpret_cast<const float4*>(A + (size_t)m * g.sAm + k)) : zero4;
            } else {         // four consecutive rows at k = e / (BM / 4)
                const int m = m0 + 4 * (e % (BM / 4)), k = k0 + e / (BM / 4);
                pa[r] = (m < g.M && k < g.K) ? __ldg(reinterpret_cast<const float4*>(A + (size_t)k * g.sAk + m)) : zero4;
            }
        }
#pragma unroll
        for (int r = 0; r < PB; ++r) {
            const int e = tid + r * THREADS;
            if (b_k_fast) {
                const int n = n0 + (e >> 2), k = k0 + 4 * (e & 3);
                pb[r] = (n < g.N && k < g.K) ? __ldg(reinterpret_cast<const float4*>(B + (size_t)n * g.sBn + k)) : zero4;
            } else {
                const int n = n0 + 4 * (e % (BN / 4)), k = k0 + e / (BN / 4);
                pb[r] = (n < g.N && k < g.K) ? __ldg(reinterpret_cast<const float4*>(B + (size_t)k * g.sBk + n)) : zero4;
            }
        }
    };
    fetch(0);
    for (int k0 = 0; k0 < g.K; k0 += TK) {
#pragma unroll
        for (int r = 0; r < PA; ++r) {
            const int e = tid + r * THREADS;
            if (a_k_fast) {
                const int m = e >> 2, k = 4 * (e & 3);
                As[k][m] = pa[r].x; As[k + 1][m] = pa[r].y; As[k + 2][m] = pa[r].z; As[k + 3][m] = pa[r].w;
            } else {
                *reinterpret_cast<float4*>(&As[e / (BM / 4)][4 * (e % (BM / 4))]) = pa[r];
            }
        }
#pragma unroll
        for (int r = 0; r < PB; ++r) {
            const int e = tid + r * THREADS;
            if (b_k_fast) {
                const int n = e >> 2, k = 4 * (e & 3);
                Bs[k][n] = pb[r].x; Bs[k + 1][n] = pb[r].y; Bs[k + 2][n] = pb[r].z; Bs[k + 3][n] = pb[r].w;
            } else {
                *reinterpret_cast<float4*>(&Bs[e / (BN / 4)][4 * (e % (BN / 4))]) = pb[r];
            }
        }
        __syncthreads();
        fetch(k0 + TK);  // all zero past the end
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            float av[RM];
#pragma unroll
            for (int i = 0; i < RM; i += 4) {
                const float4 a4 = *reinterpret_cast<const float4*>(&As[kk][mw + i]);
                av[i] = a4.x; av[i + 1] = a4.y; av[i + 2] = a4.z; av[i + 3] = a4.w;
            }
            const float4 b4 = *reinterpret_cast<const float4*>(&Bs[kk][nw]);
            const float bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        if (SUMS && sums) {
#pragma unroll
            for (int kk = 0; kk < TK; ++kk) rowsum += As[kk][tid];  // zero past the end
        }
        __syncthreads();
    }
    if (SUMS && sums && m0 + tid < g.M) g.rowsum[(size_t)z * g.sRz + m0 + tid] = rowsum;
    float* C = g.C + (size_t)z * g.sCz;
    const float* bias = g.bias ? g.bias + (size_t)z * g.sBiasz : nullptr;
    const float* mask = g.mask ? g.mask + (size_t)z * g.sMz : nullptr;
    const int n = n0 + nw;
    if (n >= g.N) return;  // N is a multiple of four: the thread's four columns are inside or outside together
    float bb[4] = {0.f, 0.f, 0.f, 0.f};
    if (bias) {
#pragma unroll
        for (int j = 0; j < 4; ++j) bb[j] = __ldg(bias + n + j);
    }
#pragma unroll
    for (int i = 0; i < RM; ++i) {
        const int m = m0 + mw + i;
        if (m >= g.M) break;
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[j] = acc[i][j];
            if (bias) v[j] += bb[j];
            if (g.relu) v[j] = fmaxf(v[j], 0.f);
        }
        if (mask) {
            const float4 mk = __ldg(reinterpret_cast<const float4*>(mask + (size_t)m * g.sMm + n));
            if (!(mk.x > 0.f)) v[0] = 0.f;
            if (!(mk.y > 0.f)) v[1] = 0.f;
            if (!(mk.z > 0.f)) v[2] = 0.f;
            if (!(mk.w > 0.f)) v[3] = 0.f;
        }
        *reinterpret_cast<float4*>(C + (size_t)m * g.sCm + n) = make_float4(v[0], v[1], v[2], v[3]);
    }
}

// The same for backward GEMMs of few tiles (fewer than the chip has schedulers).  Too few warps to hide latency behind, so a warp owns a tile of
// 64 x 32 outputs, 8 x 8 per thread (below that shared-memory reads bound it: a 128-bit read takes four cycles of a pipe that
// the SM's four schedulers share), with a ring of its own (three steps of eight k, asynchronous copies, no block barriers), and
// the kSlices warps of a block share one tile: each sums its slice of k in ascending order and the slices are added in order.
// Operands are staged as they lie in memory: one with its unit stride along k (AK) as rows of eight k, of which a thread
// reads four at once (neighbouring lanes on neighbouring rows: distinct banks), one with its unit stride along the output as
// eight rows.  (10 workers, 256 x 256 x 1024: 46 us against 60; with more tiles the block-tile kernel is better: 10 workers,
// 1024 x 256 x 256: 41.5 against 45.5.)
constexpr int kTileM = 64, kTileN = 32, kSlices = 4, kStepK = 8, kSteps = 3;

// One operand of a warp's tile: R outputs, T of them per thread, LANES threads along it; KF: unit stride along k.
template <int R, int T, int LANES, bool KF>
struct GemmOperand {
    static constexpr int kPitch = KF ? kStepK : R + 4;
    static constexpr int kFloats = KF ? R * kPitch : kStepK * kPitch;
    static __device__ __forceinline__ int index(int t, int i) { return KF ? t + i * LANES : 4 * t + (i / 4) * (4 * LANES) + i % 4; }
    // outputs past the edge are copies of the last ones (never stored); k past the slice is zero
    static __device__ __forceinline__ void stage(float* sm, const float* src, long long stride, int row0, int rows, int k0, int k_end, int lane) {
#pragma unroll
        for (int u = 0; u < R * kStepK / 128; ++u) {
            const int e = lane + 32 * u;
            const int r = KF ? e / 2 : 4 * (e % (R / 4)), k = KF ? 4 * (e % 2) : e / (R / 4);
            const float* from = KF ? src + (long long)min(row0 + r, rows - 1) * stride + (k0 + k) : src + (long long)(k0 + k) * stride + min(row0 + r, rows - 4);
            const int valid = KF ? max(0, min(4, k_end - k0 - k)) * 4 : (k0 + k < k_end ? 16 : 0);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(sm + (KF ? r * kPitch + k : k * kPitch + r))),
                         "l"(valid ? from : src), "r"(valid)
                         : "memory");
        }
    }
    float v[4][T];  // the thread's outputs' values at k = kq .. kq + 3
    __device__ __forceinline__ void load(const float* sm, int t, int kq) {
        if (KF) {
#pragma unroll
            for (int i = 0; i < T; ++i) {
                const float4 x = *reinterpret_cast<const float4*>(sm + index(t, i) * kPitch + kq);
                v[0][i] = x.x; v[1][i] = x.y; v[2][i] = x.z; v[3][i] = x.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int i = 0; i < T; i += 4) {
                    const float4 x = *reinterpret_cast<const float4*>(sm + (kq + k) * kPitch + index(t, i));
                    v[k][i] = x.x; v[k][i + 1] = x.y; v[k][i + 2] = x.z; v[k][i + 3] = x.w;
                }
        }
    }
};

template <bool SUMS, bool AK>
__global__ void __launch_bounds__(kSlices * 32, 3) gemm_slice_kernel(const __grid_constant__ GemmArgs g) {
    dependent_begin();
    constexpr int TM = 8, TN = 8, TX = kTileN / TN, TY = kTileM / TM;
    typedef GemmOperand<kTileM, TM, TY, AK> OpA;
    typedef GemmOperand<kTileN, TN, TX, false> OpB;
    constexpr int kRing = kSteps * (OpA::kFloats + OpB::kFloats), kExchange = TM * TN * 32 + 64;
    constexpr int kPerWarp = (kRing > kExchange ? kRing : kExchange + 3) / 4 * 4;
    __shared__ __align__(16) float sm[kSlices][kPerWarp];
    const int z = blockIdx.z, lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int m0 = blockIdx.y * kTileM, n0 = blockIdx.x * kTileN;
    const int ty = lane / TX, tx = lane % TX;
    const float* A = g.A + (size_t)z * g.sAz;
    const float* B = g.B + (size_t)z * g.sBz;
    const int k_lo = part * g.slice, k_hi = min(g.K, k_lo + g.slice);
    const int steps = (k_hi - k_lo + kStepK - 1) / kStepK;
    float* ring = sm[part];
    auto fetch = [&](int step, int slot) {
        if (step < steps) {
            float* st = ring + slot * (OpA::kFloats + OpB::kFloats);
            OpA::stage(st, A, AK ? g.sAm : g.sAk, m0, g.M, k_lo + step * kStepK, k_hi, lane);
            OpB::stage(st + OpA::kFloats, B, g.sBk, n0, g.N, k_lo + step * kStepK, k_hi, lane);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int s = 0; s < kSteps - 1; ++s) fetch(s, s);
    float acc[TM][TN] = {};
    float rows[2] = {0.f, 0.f};
    const bool sums = SUMS && n0 == 0;
    int slot = 0;
#pragma unroll 1
    for (int step = 0; step < steps; ++step) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kSteps - 2) : "memory");
        __syncwarp();  // this step's copies have landed for every lane, and every lane is done with the step before
        fetch(step + kSteps - 1, slot == 0 ? kSteps - 1 : slot - 1);
        const float* a_sm = ring + slot * (OpA::kFloats + OpB::kFloats);
        const float* b_sm = a_sm + OpA::kFloats;
        slot = slot == kSteps - 1 ? 0 : slot + 1;
#pragma unroll
        for (int kq = 0; kq < kStepK; kq += 4) {
            OpA a;
            OpB b;
            a.load(a_sm, ty, kq);
            b.load(b_sm, tx, kq);
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a.v[k][i], b.v[k][j], acc[i][j]);
        }
        if (SUMS && !AK && sums) {
#pragma unroll
            for (int k = 0; k < kStepK; ++k) {  // zero past the end
                rows[0] += a_sm[k * OpA::kPitch + lane];
                rows[1] += a_sm[k * OpA::kPitch + lane + 32];
            }
        }
    }
    constexpr int IPW = TM / kSlices;  // rows of a thread's outputs that its warp finishes
    {  // the slices through shared memory: warp p adds up the outputs i = p IPW .. of every lane
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        float4* ex = reinterpret_cast<float4*>(ring);
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; j += 4) ex[(i * (TN / 4) + j / 4) * 32 + lane] = make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
        if (sums) {
            ring[TM * TN * 32 + lane] = rows[0];
            ring[TM * TN * 32 + 32 + lane] = rows[1];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < IPW; ++i)
#pragma unroll
            for (int j = 0; j < TN; j += 4) {
                const int at = ((part * IPW + i) * (TN / 4) + j / 4) * 32 + lane;
                float4 t = reinterpret_cast<const float4*>(sm[0])[at];
#pragma unroll
                for (int p = 1; p < kSlices; ++p) {
                    const float4 x = reinterpret_cast<const float4*>(sm[p])[at];
                    t.x += x.x; t.y += x.y; t.z += x.z; t.w += x.w;
                }
                acc[i][j] = t.x; acc[i][j + 1] = t.y; acc[i][j + 2] = t.z; acc[i][j + 3] = t.w;
            }
        if (sums && part == 0) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int p = 1; p < kSlices; ++p) rows[h] += sm[p][TM * TN * 32 + 32 * h + lane];
        }
    }
    if (sums && part == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (m0 + lane + 32 * h < g.M) g.rowsum[(size_t)z * g.sRz + m0 + lane + 32 * h] = rows[h];
    }
    float* C = g.C + (size_t)z * g.sCz;
    const float* mask = g.mask ? g.mask + (size_t)z * g.sMz : nullptr;
#pragma unroll
    for (int i = 0; i < IPW; ++i) {
        const int m = m0 + OpA::index(ty, part * IPW + i);
        if (m >= g.M) continue;
        float* c = C + (size_t)m * g.sCm;
        const float* mk = mask ? mask + (size_t)m * g.sMm : nullptr;
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
            const int n = n0 + OpB::index(tx, j);
            if (n >= g.N) continue;  // N is a multiple of four: the four columns are inside or outside together
            float4 v = make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
            if (mk) {
                const float4 x = __ldg(reinterpret_cast<const float4*>(mk + n));
                v.x = x.x > 0.f ? v.x : 0.f; v.y = x.y > 0.f ? v.y : 0.f; v.z = x.z > 0.f ? v.z : 0.f; v.w = x.w > 0.f ? v.w : 0.f;
            }
            *reinterpret_cast<float4*>(c + n) = v;
        }
    }
}

// A forward GEMM (bias, ReLU), whose sums stay in ascending k.  A block is one warp with a tile of 32 x 32 outputs, 4 x 8 per
// thread, and a ring of its own: no block barriers, hardly a partial tile, and an even spread over the schedulers.  What bounds it
// is a step's latency, so operands are read from shared memory half a step ahead and a copy's addresses are formed once.
constexpr int kWarpTile = 32, kWarpSteps = 6;
__global__ void __launch_bounds__(32, 8) gemm_warp_kernel(const __grid_constant__ GemmArgs g) {
    dependent_begin();
    constexpr int TM = 4, TN = 8;
    typedef GemmOperand<kWarpTile, TM, kWarpTile / TM, true> OpA;
    typedef GemmOperand<kWarpTile, TN, kWarpTile / TN, true> OpB;
    constexpr int kStep = OpA::kFloats + OpB::kFloats;
    __shared__ __align__(16) float ring[kWarpSteps * kStep];
    const int z = blockIdx.z, lane = threadIdx.x;
    const int m0 = blockIdx.y * kWarpTile, n0 = blockIdx.x * kWarpTile;
    const int ty = lane / (kWarpTile / TN), tx = lane % (kWarpTile / TN);
    const float* A = g.A + (size_t)z * g.sAz;
    const float* B = g.B + (size_t)z * g.sBz;
    const int steps = (g.K + kStepK - 1) / kStepK;
    // copies u = 0, 1 of each operand: 16 bytes at row (lane + 32 u) / 2, k = 4 (lane % 2) of a step
    const int kc = 4 * (lane & 1);
    const float *pa[2], *pb[2];
    uint32_t to[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int r = (lane + 32 * u) / 2;
        pa[u] = A + (long long)min(m0 + r, g.M - 1) * g.sAm + kc;
        pb[u] = B + (long long)min(n0 + r, g.N - 1) * g.sBn + kc;
        to[u] = (uint32_t)__cvta_generic_to_shared(ring + r * kStepK + kc);
    }
    auto fetch = [&](int step, int slot) {
        const int k0 = step * kStepK;
        if (step < steps) {
            const int valid = k0 + kc < g.K ? 16 : 0, at = valid ? k0 : 0;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to[u] + slot * kStep * 4), "l"(pa[u] + at - (valid ? 0 : kc)), "r"(valid) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to[u] + (slot * kStep + OpA::kFloats) * 4), "l"(pb[u] + at - (valid ? 0 : kc)), "r"(valid) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int s = 0; s < kWarpSteps - 1; ++s) fetch(s, s);
    float acc[TM][TN] = {};
    auto multiply = [&](const OpA& a, const OpB& b) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a.v[k][i], b.v[k][j], acc[i][j]);
    };
    OpA a[2];
    OpB b[2];
    asm volatile("cp.async.wait_group %0;" ::"n"(kWarpSteps - 2) : "memory");
    __syncwarp();
    a[0].load(ring, ty, 0);
    b[0].load(ring + OpA::kFloats, tx, 0);
    int slot = 0;
#pragma unroll 1
    for (int step = 0; step < steps; ++step) {
        a[1].load(ring + slot * kStep, ty, 4);
        b[1].load(ring + slot * kStep + OpA::kFloats, tx, 4);
        multiply(a[0], b[0]);
        asm volatile("cp.async.wait_group %0;" ::"n"(kWarpSteps - 3) : "memory");
        __syncwarp();  // the next step's copies have landed for every lane, and every lane is done with the step before
        fetch(step + kWarpSteps - 1, slot == 0 ? kWarpSteps - 1 : slot - 1);
        slot = slot == kWarpSteps - 1 ? 0 : slot + 1;
        a[0].load(ring + slot * kStep, ty, 0);  // past the end: a slot's old values, not used
        b[0].load(ring + slot * kStep + OpA::kFloats, tx, 0);
        multiply(a[1], b[1]);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    float* C = g.C + (size_t)z * g.sCz;
    const float* bias = g.bias + (size_t)z * g.sBiasz;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
        const int n = n0 + OpB::index(tx, j);
        if (n >= g.N) continue;
        const float bn = __ldg(bias + n);
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            const int m = m0 + OpA::index(ty, i);
            if (m < g.M) C[(size_t)m * g.sCm + n] = g.relu ? fmaxf(acc[i][j] + bn, 0.f) : acc[i][j] + bn;
        }
    }
}

// A call of its own: inlined, dA's kernel with two blocks to an SM spills 132 bytes for 68 (10 workers, 1024 x 256 x 256: 2 us a round).
__device__ __noinline__ void sum_again(const split::Block& blk, const GemmArgs& g, const split::Tiles& tiles) { split::sum_on_cuda_cores<true>(blk, g, tiles, blockIdx.x); }

// On the tensor cores (gemm_split.cuh), a block to a tile.  DEEP: a block to an SM with loads two steps ahead and a ring of four, for
// launches of no more tiles than SMs, which wait for their chain of k steps; else two blocks to an SM with half of that each.
template <int KIND, bool VEC, bool DEEP>
__global__ void __launch_bounds__(split::kFillThreads + 32, DEEP ? 1 : 2) gemm_split_kernel(const __grid_constant__ GemmArgs g, const split::Tiles tiles) {
    dependent_begin();
    constexpr int RING = DEEP ? 4 : 2, AHEAD = DEEP ? 2 : 1;
    extern __shared__ uint8_t split_smem[];
    __shared__ split::BlockSmem fixed;
    split::Block blk;
    bool finite = true;
    if (threadIdx.x < split::kFillThreads) {
        finite = split::gemm_tile<KIND, VEC, true, RING, AHEAD, true>(blk, g, tiles, blockIdx.x, [&] { split::block_begin(blk, split_smem, fixed); });
    } else {
        split::block_begin(blk, split_smem, fixed);
        split::issue_tile<KIND, RING>(blk, g);
    }
    const bool again = split::block_end(blk, !finite);
    if (again && threadIdx.x < split::kFillThreads) {
        if constexpr (KIND == split::DA) sum_again(blk, g, tiles);
        else split::sum_on_cuda_cores<true>(blk, g, tiles, blockIdx.x);
    }
}

template <int KIND, bool VEC, bool DEEP>
int launch_split_of(dbw_handle* h, const GemmArgs& g, const split::Tiles& tiles, cudaStream_t s) {
    static PerDeviceOnce once;
    constexpr size_t smem = split::smem_bytes(DEEP ? 4 : 2);
    const int rc = once.run(h->device, []() -> int {
        DBW_CUDA(cudaFuncSetAttribute(gemm_split_kernel<KIND, VEC, DEEP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        return DBW_OK;
    });
    if (rc) return rc;
    launch<false>(gemm_split_kernel<KIND, VEC, DEEP>, tiles.total, split::kFillThreads + 32, smem, s, g, tiles);
    DBW_LAUNCHED();
    return DBW_OK;
}

template <int KIND>
int launch_split(dbw_handle* h, const GemmArgs& g, int batch, cudaStream_t s) {
    const split::Tiles tiles(g.M, g.N, batch);
    if (tiles.total <= h->sm_count)
        return split::aligned<KIND>(g) ? launch_split_of<KIND, true, true>(h, g, tiles, s) : launch_split_of<KIND, false, true>(h, g, tiles, s);
    return split::aligned<KIND>(g) ? launch_split_of<KIND, true, false>(h, g, tiles, s) : launch_split_of<KIND, false, false>(h, g, tiles, s);
}

// 128-bit accesses are possible: unit stride along k or along the output dimension, everything else a multiple of four floats
bool gemm_vec_ok(const GemmArgs& g) {
    auto al = [](const void* p) { return ((uintptr_t)p & 15) == 0; };
    const bool a_ok = (g.sAk == 1 && g.K % 4 == 0 && g.sAm % 4 == 0) || (g.sAm == 1 && g.M % 4 == 0 && g.sAk % 4 == 0);
    const bool b_ok = (g.sBk == 1 && g.K % 4 == 0 && g.sBn % 4 == 0) || (g.sBn == 1 && g.N % 4 == 0 && g.sBk % 4 == 0);
    if (g.sAk != 1 && g.sBk == 1) return false;  // no GEMM of the path has this pair of layouts
    const bool c_ok = g.N % 4 == 0 && g.sCm % 4 == 0 && g.sCz % 4 == 0 && al(g.C);
    const bool m_ok = !g.mask || (g.sMm % 4 == 0 && g.sMz % 4 == 0 && al(g.mask));
    return a_ok && b_ok && c_ok && m_ok && g.sAz % 4 == 0 && g.sBz % 4 == 0 && al(g.A) && al(g.B);
}

// Last layer with at most 32 classes: forward + loss by a warp per U samples, backward by a block per worker
// and 128 or 64 features (bodies in round_dev.cuh).
template <int CP, int U, bool VEC>
__global__ void __launch_bounds__(256)
last_layer_forward_kernel(int N, int B, int in, int C, HeadRows rows, const float* __restrict__ X, long long ld, long long w_off,
                          long long b_off, float* __restrict__ dz, float* __restrict__ loss_s, uint32_t* status) {
    dependent_begin();
    const int item = blockIdx.x * 8 + (threadIdx.x >> 5), groups = (B + U - 1) / U;
    if (item >= N * groups) return;
    const int i = item / groups;
    head_forward_samples<CP, U, VEC, true>(i, item % groups * U, B, in, C, rows, X + (size_t)i * ld + w_off, X + (size_t)i * ld + b_off, dz, loss_s, status);
}

template <int CP, int SLICES, bool VEC>
__global__ void __launch_bounds__(256)
last_layer_backward_kernel(int B, int in, int C, HeadRows rows, const float* __restrict__ dz, const float* __restrict__ loss_s,
                           const float* __restrict__ X, float* __restrict__ G, long long ld, long long w_off, long long b_off,
                           float* __restrict__ loss, float* __restrict__ dz_prev, long long b_off_prev, float* __restrict__ partial, uint32_t* status) {
    dependent_begin();
    extern __shared__ __align__(16) float head_smem[];
    const int i = blockIdx.y, k_lo = blockIdx.x * head_chunk4(SLICES);
    const int k_hi = min((in + 3) >> 2, k_lo + head_chunk4(SLICES));
    const int s_lo = blockIdx.z * kHeadPart, s_hi = min(B, s_lo + kHeadPart);
    float *Gw = G + (size_t)i * ld + w_off, *Gb = G + (size_t)i * ld + b_off, *Gp = G + (size_t)i * ld + b_off_prev, *li = loss ? loss + i : nullptr;
    float scale = 1.0f / (float)B;
    if (gridDim.z > 1) {
        Gw = partial + ((size_t)blockIdx.z * gridDim.y + i) * fp32_head_partial(in, C);
        Gb = Gw + (size_t)C * in;
        Gp = Gb + C;
        li = Gp + in;
        scale = 1.f;
    }
    head_backward_part<CP, SLICES, VEC, true>(i, s_lo, s_hi, scale, k_lo, k_hi, B, in, C, rows, dz, loss_s, X + (size_t)i * ld + w_off, Gw, Gb, li, dz_prev, Gp,
                                      head_smem, status);
}

__global__ void __launch_bounds__(256)
last_layer_add_parts_kernel(int parts, int N, int B, int in, int C, const float* __restrict__ partial, float* __restrict__ G, long long ld, long long w_off,
                            long long b_off, long long b_off_prev, float* __restrict__ loss) {
    dependent_begin();
    const int i = blockIdx.y, e = blockIdx.x * 256 + threadIdx.x;
    float* Gi = G + (size_t)i * ld;
    if (e <= C * in + C + in) head_add_parts(i, e, parts, N, B, in, C, partial, Gi + w_off, Gi + b_off, b_off_prev >= 0 ? Gi + b_off_prev : nullptr, loss ? loss + i : nullptr);
}

template <int WM, int RM>
void launch_gemm_vec(const GemmArgs& g, int batch, cudaStream_t s) {
    const dim3 grid((g.N + 63) / 64, (g.M + 2 * RM * WM - 1) / (2 * RM * WM), batch);
    if (g.rowsum)
        launch<false>(gemm_vec_kernel<WM, RM, true>, grid, 32 * WM, 0, s, g);
    else
        launch<false>(gemm_vec_kernel<WM, RM, false>, grid, 32 * WM, 0, s, g);
}

void launch_gemm_slice(const GemmArgs& g, int batch, cudaStream_t s) {
    const dim3 grid((g.N + kTileN - 1) / kTileN, (g.M + kTileM - 1) / kTileM, batch);
    if (g.sAk != 1 && g.rowsum)
        launch<false>(gemm_slice_kernel<true, false>, grid, kSlices * 32, 0, s, g);
    else if (g.sAk != 1)
        launch<false>(gemm_slice_kernel<false, false>, grid, kSlices * 32, 0, s, g);
    else
        launch<false>(gemm_slice_kernel<false, true>, grid, kSlices * 32, 0, s, g);
}

enum GemmStep { GEMM_FORWARD, GEMM_DW, GEMM_DA };
int run_gemm(dbw_handle* h, GemmArgs& g, GemmStep step, int batch, cudaStream_t s) {
    const int sm_count = h->sm_count;
    g.status = h->d_status;
    if (step != GEMM_FORWARD && fp32_gemm_split(g.M, g.N, g.K, batch, step == GEMM_DW))
        return step == GEMM_DW ? launch_split<split::DW>(h, g, batch, s) : launch_split<split::DA>(h, g, batch, s);
    g.slice = step == GEMM_FORWARD ? g.K : fp32_gemm_slice(g.M, g.N, g.K, batch, step == GEMM_DW, sm_count);
    if (gemm_vec_ok(g) && g.slice < g.K) {
        launch_gemm_slice(g, batch, s);
        DBW_LAUNCHED();
        return DBW_OK;
    }
    // One-warp blocks where every SM gets at least two of them and none more than the eight that fit it at once.  Measured (workers,
    // M x N x K, tiles: one-warp / block-tile kernel, us): 32, 64 x 200 x 784, 448: 30.3 / 38.2; 64 of them, 896: 48.8 / 64.7; 60,
    // 128 x 128 x 256, 960: 19.4 / 23.2.  Fewer tiles leave the schedulers idle: 64, 64 x 64 x 784, 256: 29.8 / 28.6; 3, 64 x 200 x
    // 784, 42: 27.6 / 24.9.  More run in waves: 10, 1024 x 256 x 784, 2560: 118 / 120, and a round with two such of K = 256
    // 335 / 328.  A short sum does not pay for filling the ring: 60, 64 x 128 x 64, 480: 6.0 / 5.2.
    const long long warp_tiles = (long long)((g.N + kWarpTile - 1) / kWarpTile) * ((g.M + kWarpTile - 1) / kWarpTile) * batch;
    if (gemm_vec_ok(g) && step == GEMM_FORWARD && g.K >= 128 && warp_tiles >= 2LL * sm_count && warp_tiles <= 8LL * sm_count) {
        launch<false>(gemm_warp_kernel, dim3((g.N + kWarpTile - 1) / kWarpTile, (g.M + kWarpTile - 1) / kWarpTile, batch), 32, 0, s, g);
        DBW_LAUNCHED();
        return DBW_OK;
    }
    if (gemm_vec_ok(g)) {
        // 8 x 4 outputs per thread where that still gives every SM several warps, else 4 x 4 (twice the warps
        // for the same tile), on tiles of 64, 32 or 16 rows
        const long long t64 = (long long)((g.N + 63) / 64) * ((g.M + 63) / 64) * batch;
        const long long t32 = (long long)((g.N + 63) / 64) * ((g.M + 31) / 32) * batch;
        if (t64 >= 2LL * sm_count)
            launch_gemm_vec<4, 8>(g, batch, s);
        else if (t32 >= sm_count)
            launch_gemm_vec<4, 4>(g, batch, s);
        else
            launch_gemm_vec<2, 4>(g, batch, s);
        DBW_LAUNCHED();
        return DBW_OK;
    }
    const long long big = (long long)((g.N + 63) / 64) * ((g.M + 63) / 64) * batch;
    if (big >= 4LL * sm_count) {
        dim3 grid((g.N + 63) / 64, (g.M + 63) / 64, batch);
        launch<false>(gemm_simt_kernel<4, 16>, grid, 256, 0, s, g);
    } else {
        dim3 grid((g.N + 31) / 32, (g.M + 31) / 32, batch);
        const long long ctas = (long long)grid.x * grid.y * grid.z;
        if (g.K >= 128 && ctas < 2LL * sm_count)  // few CTAs, long reduction
            launch<false>(gemm_simt_kernel<2, 64>, grid, 256, 0, s, g);
        else
            launch<false>(gemm_simt_kernel<2, 16>, grid, 256, 0, s, g);
    }
    DBW_LAUNCHED();
    return DBW_OK;
}

}  // namespace

// Which backward GEMMs run on the tensor cores: those of many multiply-adds; fewer where operand rows are not whole 16-byte groups and
// the CUDA-core kernel is the scalar one.  Measured on 900 GEMMs of 4 - 64 workers (us, CUDA cores / tensor cores): 10 workers, M x
// N x K = 1024 x 256 x 256 42 / 24.8, 32, 200 x 784 x 64 26.6 / 20.1; at the lines 49, 92 x 168 x 92 (70 million) 10.4 / 10.4 and 12, 32 x
// 256 x 307 (30 million) 10.4 / 13.9; unaligned 7, 58 x 276 x 457 (51 million) 12.4 / 16.5.  What it costs is a launch's chain:
// operands to bf16 pieces, MMAs and a barrier between them for every 32 k, about 0.5 us whatever the size; a k of one such step
// does not pay for it (38, 252 x 784 x 28: 24.7 / 26.5), nor does a long one of few multiply-adds.
bool fp32_gemm_split(int M, int N, int K, int batch, bool is_dw) {
    const bool rows_aligned = N % 4 == 0 && (is_dw ? M : K) % 4 == 0;
    return (long long)M * N * K * batch >= (rows_aligned || K > 512 ? 60000000 : 30000000) && (K > split::kStep || !rows_aligned);
}

// is_dw: dZ^T A, both operands with their unit stride along the output; else with the first one's along k.
int fp32_gemm_slice(int M, int N, int K, int batch, bool is_dw, int sm_count) {
    if (N % 4 || (is_dw ? M : K) % 4) return K;  // not for gemm_slice_kernel
    const long long tiles = (long long)((M + kTileM - 1) / kTileM) * ((N + kTileN - 1) / kTileN) * batch;
    if (tiles >= 4LL * sm_count || K < 32 * kSlices) return K;  // enough tiles, or slices of less than four steps
    return ((K + kSlices - 1) / kSlices + kStepK - 1) / kStepK * kStepK;
}

int grad_fp32_alloc(dbw_handle* h) {
    const dbw_model_desc& m = h->model;
    const size_t NB = (size_t)h->N * m.batch;
    for (int l = 0; l <= m.n_layers; ++l) {
        DBW_CUDA(cudaMalloc(&h->d_act[l], NB * m.dims[l] * sizeof(float)));
        if (l >= 1) DBW_CUDA(cudaMalloc(&h->d_dz[l], NB * m.dims[l] * sizeof(float)));
    }
    DBW_CUDA(cudaMalloc(&h->d_ylab, NB * sizeof(int32_t)));
    const int parts = fp32_head_parts(m.batch);
    if (parts > 1 && m.dims[m.n_layers] <= 32)
        DBW_CUDA(cudaMalloc(&h->d_head_part, (size_t)parts * h->N * fp32_head_partial(m.dims[m.n_layers - 1], m.dims[m.n_layers]) * sizeof(float)));
    return DBW_OK;
}

void grad_fp32_free(dbw_handle* h) {
    for (int l = 0; l <= DBW_MAX_LAYERS; ++l) {
        if (h->d_act[l]) cudaFree(h->d_act[l]);
        if (h->d_dz[l]) cudaFree(h->d_dz[l]);
        h->d_act[l] = h->d_dz[l] = nullptr;
    }
    if (h->d_ylab) cudaFree(h->d_ylab);
    h->d_ylab = nullptr;
    if (h->d_head_part) cudaFree(h->d_head_part);
    h->d_head_part = nullptr;
}

int launch_grad_fp32(dbw_handle* h, const float* X, const int32_t* batch_idx, float* G, float* loss,
                     cudaStream_t s, const std::function<int()>* beside) {
    const dbw_model_desc& m = h->model;
    const int B = m.batch, L = m.n_layers, N = h->N;
    // A last layer of at most 32 classes runs as two kernels of its own instead of a GEMM, the loss kernel and
    // two more GEMMs; a one-layer model then needs no gathered copy of the mini-batch either.
    const bool head = fp32_head_usable(h), head_aligned = fp32_head_aligned(h) && (((uintptr_t)X | (uintptr_t)G) & 15) == 0;
    const int Lg = head ? L - 1 : L;  // layers that run as GEMMs
    if (Lg > 0 || !head) {
        if ((long long)B * N <= 16LL * h->sm_count)
            launch(gather_batch_kernel<true>, dim3(B, N), 128, 0, s, B, h->S, m.dims[0], m.dims[L], h->feat, h->labels, batch_idx, h->d_act[0],
                   h->d_ylab, h->d_status);
        else
            launch<false>(gather_batch_kernel<false>, dim3(B, N), 128, 0, s, B, h->S, m.dims[0], m.dims[L], h->feat, h->labels, batch_idx,
                          h->d_act[0], h->d_ylab, h->d_status);
        DBW_LAUNCHED();
    }
    int rc;
    // forward: Z_l = A_{l-1} W_l^T + b_l, A_l = ReLU(Z_l), logits for the last layer
    for (int l = 0; l < Lg; ++l) {
        const int in = m.dims[l], out = m.dims[l + 1];
        GemmArgs g{};
        g.A = h->d_act[l]; g.sAz = (long long)B * in; g.sAm = in; g.sAk = 1;
        g.B = X + m.w_off[l]; g.sBz = h->ld; g.sBn = in; g.sBk = 1;
        g.C = h->d_act[l + 1]; g.sCz = (long long)B * out; g.sCm = out;
        g.bias = X + m.b_off[l]; g.sBiasz = h->ld;
        g.M = B; g.N = out; g.K = in; g.relu = l < L - 1;
        if ((rc = run_gemm(h, g, GEMM_FORWARD, N, s)) != DBW_OK) return rc;
    }
    if (beside && (rc = (*beside)())) return rc;
    if (head) {
        const int in = m.dims[L - 1], C = m.dims[L];
        HeadRows rows{};
        if (L > 1) {
            rows.act = h->d_act[L - 1]; rows.ylab = h->d_ylab;
        } else {
            rows.feat = h->feat; rows.labels = h->labels; rows.batch_idx = batch_idx; rows.S = h->S;
        }
        float* loss_s = h->d_act[L];  // [N][B] of the logits' buffer: the logits themselves are never stored
        float* dz_prev = L > 1 ? h->d_dz[L - 1] : nullptr;
        const int parts = fp32_head_parts(B);
        const int slices = fp32_head_slices(h);
        const dim3 bgrid(((in + 3) / 4 + head_chunk4(slices) - 1) / head_chunk4(slices), N, parts);
        const long long b_prev = L > 1 ? m.b_off[L - 2] : -1;
        const size_t smem = fp32_head_smem_bytes(B, C);
        // Four samples to a warp once that still gives every SM a dozen warps.
        const bool four = (long long)N * ((B + 3) / 4) >= 12LL * h->sm_count && C <= 16;
        const long long b_prev_off = L > 1 ? b_prev : 0;
        auto both = [&](auto cp, auto samples, auto vec) -> int {
            constexpr int CP = decltype(cp)::value, U = decltype(samples)::value;
            constexpr bool VEC = decltype(vec)::value;
            launch<false>(last_layer_forward_kernel<CP, U, VEC>, (N * ((B + U - 1) / U) + 7) / 8, 256, 0, s, N, B, in, C, rows, X, h->ld, m.w_off[L - 1], m.b_off[L - 1], h->d_dz[L],
                          loss_s, h->d_status);
            DBW_LAUNCHED();
            launch<false>(slices == 16 ? last_layer_backward_kernel<CP, 16, VEC> : last_layer_backward_kernel<CP, 8, VEC>, bgrid, 256, smem, s, B, in, C, rows, h->d_dz[L], loss_s,
                          X, G, h->ld, m.w_off[L - 1], m.b_off[L - 1], loss, dz_prev, b_prev_off, h->d_head_part, h->d_status);
            DBW_LAUNCHED();
            return DBW_OK;
        };
        using std::integral_constant;
        using one = integral_constant<int, 1>;
        using several = integral_constant<int, 4>;
        if (C > 16)
            rc = head_aligned ? both(integral_constant<int, 32>{}, one{}, std::true_type{}) : both(integral_constant<int, 32>{}, one{}, std::false_type{});
        else if (four)
            rc = head_aligned ? both(integral_constant<int, 16>{}, several{}, std::true_type{}) : both(integral_constant<int, 16>{}, several{}, std::false_type{});
        else
            rc = head_aligned ? both(integral_constant<int, 16>{}, one{}, std::true_type{}) : both(integral_constant<int, 16>{}, one{}, std::false_type{});
        if (rc) return rc;
        if (parts > 1) {
            launch(last_layer_add_parts_kernel, dim3((C * in + C + in + 256) / 256, N), 256, 0, s, parts, N, B, in, C, h->d_head_part, G, h->ld, m.w_off[L - 1],
                                                                                            m.b_off[L - 1], b_prev, loss);
            DBW_LAUNCHED();
        }
    } else {
        launch<false>(softmax_ce_kernel, N, 256, 0, s, B, m.dims[L], h->d_act[L], h->d_ylab, h->d_dz[L], loss, G, h->ld, m.b_off[L - 1]);
        DBW_LAUNCHED();
    }
    // backward
    for (int l = Lg - 1; l >= 0; --l) {
        const int in = m.dims[l], out = m.dims[l + 1];
        GemmArgs g{};  // dW_l[o][k] = sum_m dZ[m][o] A_{l}[m][k]
        g.A = h->d_dz[l + 1]; g.sAz = (long long)B * out; g.sAm = 1; g.sAk = out;
        g.B = h->d_act[l]; g.sBz = (long long)B * in; g.sBn = 1; g.sBk = in;
        g.C = G + m.w_off[l]; g.sCz = h->ld; g.sCm = in;
        g.M = out; g.N = in; g.K = B;
        const bool needs_db = l < L - 1 && !(head && l == L - 2), db_here = needs_db && (fp32_gemm_split(g.M, g.N, g.K, N, true) || gemm_vec_ok(g));
        if (db_here) {  // the sums of dZ's columns come with the GEMM that reads them
            g.rowsum = G + m.b_off[l];
            g.sRz = h->ld;
        }
        if ((rc = run_gemm(h, g, GEMM_DW, N, s)) != DBW_OK) return rc;
        if (needs_db && !db_here) {  // the last layer's bias gradient came out of the loss kernel, the one before's out of the last layer's backward kernel
            launch<false>(bias_grad_kernel, dim3((out + 127) / 128, N), 128, 0, s, B, out, h->d_dz[l + 1], G, h->ld, m.b_off[l]);
            DBW_LAUNCHED();
        }
        if (l > 0) {  // dZ_{l}[m][k] = (sum_o dZ_{l+1}[m][o] W_l[o][k]) * [A_l[m][k] > 0]
            GemmArgs a{};
            a.A = h->d_dz[l + 1]; a.sAz = (long long)B * out; a.sAm = out; a.sAk = 1;
            a.B = X + m.w_off[l]; a.sBz = h->ld; a.sBn = 1; a.sBk = in;
            a.C = h->d_dz[l]; a.sCz = (long long)B * in; a.sCm = in;
            a.mask = h->d_act[l]; a.sMz = (long long)B * in; a.sMm = in;
            a.M = B; a.N = in; a.K = out;
            if ((rc = run_gemm(h, a, GEMM_DA, N, s)) != DBW_OK) return rc;
        }
    }
    return DBW_OK;
}

}  // namespace dbw
