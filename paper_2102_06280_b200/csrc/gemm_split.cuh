// The backward fp32 GEMM tiles of the gradient path on the tensor cores, at fp32 precision.  (Forward sums stay in ascending k: whether a
// pre-activation of zero up to rounding passes its ReLU follows from the order of its sum.)  Every fp32 operand value is the exact sum of three
// bf16 pieces (each the rounded rest of the ones before), x = h + m + l, and a product is the sum of the piece products
//   h h + (h m + m h) + (h l + m m + l h) + (m l + l m),
// what is left out, l l, being below 2^-32 of the product.  Pieces are formed while an operand tile is staged in shared memory and the
// MMAs accumulate in tensor memory.  Those accumulators are truncated, not rounded, at every MMA, and always towards zero: over a
// long sum of h h that alone would be worse than fp32 multiply-adds (K = 784: -5e-7 of the result), so every 32 k the sums of h h
// move to registers and are added there with rounding.  The smaller products, 2^-8 of the sum and less, stay.
//
// Against 64 bits, relative to fp32 multiply-adds in ascending k: a sum with a single non-zero product is rounded as theirs is, sums of
// several products of similar magnitude are closer (root mean square of 2, 4, 8, 32, 128 normal ones: 0.82, 0.65, 0.53, 0.40, 0.30);
// where the magnitudes are spread over 24 binades truncation shows in sums of a few (2, 4, 8, 32, 128: 1.03, 1.11, 1.10, 0.77,
// 0.44).  Dense sums (relative 2-norm, this / theirs): K = 64 5.2e-8 / 1.5e-7, 256 7.1e-8 / 2.9e-7, 3000 1.8e-7 /
// 9.5e-7.
//
// Shared by the stand-alone kernel (grad_fp32.cu) and the single-launch round (round_fused.cu), which give the same bits.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "round_dev.cuh"
#include "tc_ptx.cuh"

namespace dbw {
namespace split {

using namespace dev;
using namespace ptx;

// Tile: 128 outputs along the index that is contiguous in C (the MMA's M, a lane of tensor memory each, so that stores are
// coalesced whatever the alignment) x 64 along the other.  The k loop goes in steps of 32 through a ring of RING halves of 64-deep
// buffers: eight warps fill one half while the MMAs read others.  The MMAs are issued by a ninth warp, or by the first of the eight
// (the single launch has no more).
constexpr int kM = 128, kN = 64, kStep = 32, kFillWarps = 8, kFillThreads = 32 * kFillWarps;
constexpr int kPieceA = kM * 128, kPieceB = kN * 128;  // bytes of one piece: 64 k of every row
constexpr int kTmemCols = 4 * kN;                      // two sums of h h, used by turns, and two of the smaller products between them
constexpr int kBufferBytes = 3 * (kPieceA + kPieceB);  // three pieces of the 128-row operand, then of the 64-row operand
__host__ __device__ constexpr size_t smem_bytes(int ring) { return (size_t)(ring / 2) * kBufferBytes + 1024 /*align slack*/; }
constexpr uint32_t kWaitLimit = 1u << 24;
// Pieces are formed of 2^24 times the value.  A bf16 number has the exponents of a float, so the last piece of a value below 2^-110 would
// be less than the smallest of them; scaled, the pieces of every float, subnormal ones included, are normal numbers.  Values and sums
// beyond the other end (2^104 and 2^80) come out infinite or NaN and are summed again (sum_on_cuda_cores).
constexpr float kScale = 16777216.f, kUnscale = 1.f / kScale / kScale;

// Barriers and tensor memory of a block, set up once and used for any number of tiles.
struct Block {
    uint8_t* buffers;         // 1024-byte aligned
    uint64_t *filled, *read;  // [RING] each: a slot is filled (an arrival per warp) / has been read by the MMAs
    volatile uint32_t* abort;
    uint32_t tmem;
    uint32_t parity;          // of each slot's next wait, a bit each: `filled` for who issues, `read` for who fills ...
    uint32_t used;            // ... and whether it has been filled at all
};
constexpr int kMaxRing = 4;
struct BlockSmem {
    uint64_t bars[2 * kMaxRing];
    uint32_t tmem, abort;
};

__device__ __forceinline__ void block_begin(Block& b, uint8_t* smem, BlockSmem& fixed) {
    b.buffers = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem) + 1023) & ~(uintptr_t)1023);
    b.filled = fixed.bars;
    b.read = fixed.bars + kMaxRing;
    b.abort = &fixed.abort;
    b.parity = b.used = 0u;
    if (threadIdx.x == 0) {
        *b.abort = 0u;
        for (int r = 0; r < kMaxRing; ++r) {
            mbar_init(&b.filled[r], kFillWarps);
            mbar_init(&b.read[r], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&fixed.tmem)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    b.tmem = __shfl_sync(0xffffffffu, fixed.tmem, 0);
}
// Returns whether `p` holds in any thread of the block.
__device__ __forceinline__ bool block_end(const Block& b, bool p = false) {
    tc_fence_before();
    p = __syncthreads_or(p);
    if (threadIdx.x < 32) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(b.tmem), "r"(kTmemCols) : "memory");
    }
    return p;
}

// By a converged warp, one lane of which issues.
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, leader;\n\t"
        "elect.sync _|leader, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@leader tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void commit(uint64_t* bar) {
    asm volatile(
        "{\n\t.reg .pred leader;\n\t"
        "elect.sync _|leader, 0xffffffff;\n\t"
        "@leader tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
        ::"r"(smem_u32(bar))
        : "memory");
}
// D = f32, A = B = bf16, M = 128, N = n; bits 15 / 16: A / B along MN
__host__ __device__ constexpr uint32_t idesc(int n, bool a_mn, bool b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
}
__device__ __forceinline__ void ld16(uint32_t taddr, float (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]),
          "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
        : "r"(taddr)
        : "memory");
    tc_ld_wait();
}

// Two neighbouring elements: the bf16 pieces of kScale times them, packed.
__device__ __forceinline__ void split2(float x, float y, uint32_t& h, uint32_t& m, uint32_t& l) {
    x *= kScale;
    y *= kScale;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(y), "f"(x));
    x -= __uint_as_float(h << 16);
    y -= __uint_as_float(h & 0xffff0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(m) : "f"(y), "f"(x));
    x -= __uint_as_float(m << 16);
    y -= __uint_as_float(m & 0xffff0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l) : "f"(y), "f"(x));
}

// One operand of a tile: R outputs.  KF: unit stride along k, row r of the operand is an output and the elements of a row are k;
// else rows are k and the elements of a row outputs.  A thread takes runs of eight neighbouring elements of a row.  Rows need not be
// aligned: a run is read as the two or (VEC = false) three 16-byte groups it lies in.  Outputs past the edge are copies of others
// or zero (never stored); k past the end is zero.
template <int R, bool KF, bool VEC, bool NC>
struct Operand {
    static constexpr int kRuns = R / 64, kGroups = VEC ? 2 : 3;
    static constexpr uint32_t kBytes = R * 128;
    static constexpr int kRowLanes = KF ? 4 : R / 8;   // lanes along a row
    static constexpr int kNext = KF ? 64 : 2;          // rows between a thread's runs
    typedef float4 Runs[kRuns][kGroups];
    const float* p[kRuns];       // the group of the run's first element in the step that is fetched next
    int shift[VEC ? 1 : kRuns];  // elements between the two, the same in every step
    uint32_t off;                // the first run's place in a piece
    int K, row, left;            // KF: elements of the row from the run of step 0 on; else row of k inside a step, elements of a row from the run on
    long long advance;

    __device__ __forceinline__ void begin(const float* base, long long pitch, int out0, int outs, int k_end) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, a = 8 * (lane % kRowLanes);
        K = k_end;
        if (KF) {  // a quarter warp takes rows that differ in bit 2: with the 128-byte swizzle their halves of a row lie in different banks
            row = warp * 8 + 4 * ((lane >> 2) & 1) + (lane >> 3);
            off = row * 128 + ((2 * a) ^ ((row & 7) << 4));
            left = K - a;
            advance = kStep;
        } else {
            row = warp * 4 + lane / kRowLanes;
            off = (a >> 6) * 8192 + row * 128 + ((2 * (a & 63)) ^ ((row & 7) << 4));
            left = outs - out0 - a;
            advance = (long long)kStep * pitch;
        }
#pragma unroll
        for (int i = 0; i < kRuns; ++i) {
            p[i] = KF ? base + (long long)min(out0 + row + kNext * i, outs - 1) * pitch + a : base + (long long)(row + kNext * i) * pitch + out0 + a;
            if (!VEC) {
                shift[VEC ? 0 : i] = (int)((reinterpret_cast<uintptr_t>(p[i]) >> 2) & 3);
                p[i] -= shift[VEC ? 0 : i];
            }
        }
    }
    // the runs of the step that begins at k0 (the pointers move on)
    __device__ __forceinline__ void fetch(int k0, Runs& run) {
#pragma unroll
        for (int i = 0; i < kRuns; ++i) {
            int there = min(KF ? left - k0 : (k0 + row + kNext * i < K ? left : 0), 8);
            if (!VEC && there > 0) there += shift[VEC ? 0 : i];
#pragma unroll
            for (int u = 0; u < kGroups; ++u) {
                run[i][u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (4 * u < there) run[i][u] = load_g<NC>(reinterpret_cast<const float4*>(p[i]) + u);
            }
            p[i] += advance;
        }
    }
    // the elements of a run (VEC: K is a multiple of four, a group is inside or outside)
    __device__ __forceinline__ void elements(int k0, int i, const Runs& run, float (&x)[8]) const {
        const float4 a = run[i][0], b = run[i][1], c = run[i][kGroups - 1];
        if (VEC) {
            x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
            x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
        } else {
            const float e[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
            const bool two = shift[VEC ? 0 : i] & 2, one = shift[VEC ? 0 : i] & 1;
            float t[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) t[k] = two ? e[k + 2] : e[k];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = one ? t[k + 1] : t[k];
            if (KF && K - k0 < kStep) {
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (k >= left - k0) x[k] = 0.f;
            }
        }
    }
    // its pieces into half `half` of the buffer, in the order h, m, l or reversed
    __device__ __forceinline__ void store(uint8_t* tile, int half, int i, bool reversed, const float (&x)[8]) const {
        uint32_t h[4], m[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) split2(x[2 * e], x[2 * e + 1], h[e], m[e], l[e]);
        uint8_t* to = tile + (KF ? off ^ (half << 6) : (off + half * 4096) ^ ((i * kNext) << 4)) + i * kNext * 128;
        const uint32_t h_at = reversed ? 2 * kBytes : 0, l_at = 2 * kBytes - h_at;
        *reinterpret_cast<uint4*>(to + h_at) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(to + kBytes) = make_uint4(m[0], m[1], m[2], m[3]);
        *reinterpret_cast<uint4*>(to + l_at) = make_uint4(l[0], l[1], l[2], l[3]);
    }
};

enum { DW = 0, DA = 1 };
// Operand rows are 16-byte aligned and whole groups of four: VEC.
template <int KIND>
__host__ __device__ inline bool aligned(const GemmArgs& g) {
    auto ok = [](const float* p, long long z, long long pitch, int cols) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && ((z | pitch | cols) & 3) == 0; };
    return ok(g.A, g.sAz, KIND == DW ? g.sAk : g.sAm, KIND == DW ? g.M : g.K) && ok(g.B, g.sBz, g.sBk, g.N);
}

// The MMAs of k step s of a tile by a converged warp; `tiles`, `half`: where its operands lie.  The pieces of the 64-row operand lie
// behind each other like 64 more outputs each, so one MMA multiplies a piece of the other operand by several of them.  Steps
// alternate between
//   pieces h, m, l:   columns [0, 192)  += h x [h m l],   [64, 192) += m x [h m],   [128, 192) += l x h + l x m + m x l   and
//   pieces l, m, h:   columns [64, 256) += h x [l m h],   [64, 192) += m x [m h],   [64, 128)  += l x h + l x m + m x l,
// which leaves the sums of h h in the first or the last 64 columns and those of the smaller products in the two between.
template <int KIND>
__device__ __forceinline__ void issue_step(uint32_t tmem, uint32_t tiles, int s, int half, uint64_t* done) {
    constexpr bool AK = KIND != DW;
    const bool odd = s & 1;
    const uint32_t sn = tiles, sm = tiles + 3 * kPieceA;
    const uint64_t dn0 = mnmajor_sw128_desc(sn, 8192), dm0 = AK ? kmajor_sw128_desc(sm) : mnmajor_sw128_desc(sm, kPieceB);
    constexpr uint32_t i1 = idesc(kN, true, !AK), i2 = idesc(2 * kN, true, !AK), i3 = idesc(3 * kN, true, !AK);
    const uint32_t d_h = tmem + (odd ? kN : 0), d_m = tmem + kN, d_l = tmem + (odd ? kN : 2 * kN);
    const uint32_t m_at = kPieceB >> 4, h_at = (odd ? 2 * kPieceB : 0) >> 4, l_at = (odd ? 0 : 2 * kPieceB) >> 4;
#pragma unroll
    for (int j = 0; j < kStep / 16; ++j) {
        const uint64_t dn = dn0 + (((half * 32 + j * 16) * 128) >> 4), dm = dm0 + ((AK ? half * 64 + j * 32 : (half * 32 + j * 16) * 128) >> 4);
        if (j == 0) {  // the step's sum of h h begins anew; those of the smaller products run on
            mma(odd ? tmem + 3 * kN : tmem, dn, dm + h_at, i1, 0u);
            mma(tmem + kN, dn, dm + (odd ? 0 : kPieceB >> 4), i2, s > 0);
        } else {
            mma(d_h, dn, dm, i3, 1u);
        }
        mma(d_m, dn + (kPieceA >> 4), dm + (odd ? m_at : 0), i2, 1u);
        mma(d_l, dn + (2 * kPieceA >> 4), dm + h_at, i1, 1u);
        mma(d_l, dn + (2 * kPieceA >> 4), dm + m_at, i1, 1u);
        mma(d_l, dn + (kPieceA >> 4), dm + l_at, i1, 1u);
    }
    commit(done);
}

// Adds COLS columns of tensor memory to a thread's sums.
template <int COLS>
__device__ __forceinline__ void add_columns(uint32_t taddr, float (&v)[COLS]) {
#pragma unroll
    for (int c = 0; c < COLS; c += 16) {
        float t[16];
        ld16(taddr + c, t);
#pragma unroll
        for (int j = 0; j < 16; ++j) v[c + j] += t[j];
    }
}
// ... and the two columns' worth of smaller products of a tile whose tensor memory begins at taddr.
template <int COLS>
__device__ __forceinline__ void add_smaller(uint32_t taddr, float (&v)[COLS]) {
#pragma unroll
    for (int c = 0; c < COLS; c += 16) {
        float t[16], u[16];
        ld16(taddr + kN + c, t);
        ld16(taddr + 2 * kN + c, u);
#pragma unroll
        for (int j = 0; j < 16; ++j) v[c + j] += t[j] + u[j];
    }
}

// Stores outputs (m1 .. m1 + COLS - 1, n) of a thread: the mask (DA).  Returns whether they are finite.
template <int KIND, bool NC, int COLS>
__device__ __forceinline__ bool finish(const GemmArgs& g, int z, int m1, int n, const float (&v)[COLS]) {
    if (n >= g.N) return true;
    const int count = min(COLS, g.M - m1);
    float* C = g.C + (size_t)z * g.sCz + (size_t)m1 * g.sCm + n;
    const float* mask = KIND == DA ? g.mask + (size_t)z * g.sMz + (size_t)m1 * g.sMm + n : nullptr;
    float none = 0.f;  // NaN as soon as one of the outputs is not finite
#pragma unroll
    for (int j = 0; j < COLS; ++j) {
        if (j < count) {
            none = fmaf(v[j], 0.f, none);
            float x = v[j] * kUnscale;
            if (KIND == DA && !(load_g<NC>(mask) > 0.f)) x = 0.f;
            *C = x;
            C += g.sCm;
            if (KIND == DA) mask += g.sMm;
        }
    }
    return none == 0.f;
}
struct Tiles {
    int n, m, total;  // along n (walked first), along m, in all
    __host__ __device__ Tiles(int M, int N, int batch) : n((N + kM - 1) / kM), m((M + kN - 1) / kN), total(n * m * batch) {}
    __device__ __forceinline__ void at(int tile, int& z, int& m0, int& n0) const {
        n0 = (tile % n) * kM;
        m0 = ((tile / n) % m) * kN;
        z = tile / (n * m);
    }
};

// Step s of a tile by a converged warp once its slot is filled.  What orders the fill warps' stores before the MMAs' reads is the proxy fence
// here: in the fill warps it would wait for their loads of the steps ahead.
template <int KIND, int SLOT>
__device__ __forceinline__ void issue_when_filled(Block& blk, const GemmArgs& g, int s) {
    const bool there = mbar_wait_bounded<false>(&blk.filled[SLOT], (blk.parity >> SLOT) & 1, kWaitLimit, 0, blk.abort, g.status);
    if (!__all_sync(0xffffffffu, there)) return;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_after();
    issue_step<KIND>(blk.tmem, smem_u32(blk.buffers) + (SLOT >> 1) * kBufferBytes, s, SLOT & 1, &blk.read[SLOT]);
}

// Calls step(s, slot) for the steps of a tile; the slot is a compile-time constant.
template <int RING, class F>
__device__ __forceinline__ void for_steps(int steps, F step) {
    for (int s = 0; s < steps; s += RING) {
        step(s, std::integral_constant<int, 0>{});
        if (s + 1 < steps) step(s + 1, std::integral_constant<int, 1>{});
        if constexpr (RING == 4) {
            if (s + 2 < steps) step(s + 2, std::integral_constant<int, 2>{});
            if (s + 3 < steps) step(s + 3, std::integral_constant<int, 3>{});
        }
    }
}

// A tile with an output that is not finite: an operand or the result is infinite or NaN, or so large that the scaled one is.  Its
// outputs are summed again as the CUDA-core kernels do, by the eight filling warps with the buffer (which no MMA reads any more) as
// staging.
template <bool NC>
__device__ __forceinline__ void sum_on_cuda_cores(const Block& blk, const GemmArgs& g, const Tiles& tiles, int tile) {
    float(*As)[68] = reinterpret_cast<float(*)[68]>(blk.buffers);
    int z, m0, n0;
    tiles.at(tile, z, m0, n0);
#pragma unroll 1
    for (int n1 = n0; n1 < min(n0 + kM, g.N); n1 += 64) dev::gemm_tile<4, 16, NC, false, kFillThreads>(g, z, m0, n1, As, As + 16);
}

// Tile `tile` of the products C[z][m][n] = epilogue(sum_k A(m, k) B(k, n)) by the eight warps of a block.  DW: both operands along the
// outputs, with the sums of A over k if wanted; DA: A along k, B along n, masked.  AHEAD: steps whose loads
// are on their way.  `ready` (block_begin) is called with the first loads on their way.  MMA_WARP: a ninth warp issues the MMAs
// (issue_tile).  Returns whether the thread's outputs are finite; where one's are not the tile is for sum_on_cuda_cores, once every
// thread is here.
template <int KIND, bool VEC, bool NC, int RING, int AHEAD, bool MMA_WARP, class Ready>
__device__ __forceinline__ bool gemm_tile(Block& blk, const GemmArgs& g, const Tiles& tiles, int tile, Ready ready) {
    constexpr bool AK = KIND != DW;
    typedef Operand<kM, false, VEC, NC> OpN;  // the operand with C's contiguous index
    typedef Operand<kN, AK, VEC, NC> OpM;
    const int steps = (g.K + kStep - 1) / kStep, tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31, q = warp & 3, mh = warp >> 2;  // a warp finishes 32 outputs along n (its lanes of tensor memory) x 32 along m
    int z, m0, n0;
    tiles.at(tile, z, m0, n0);
    OpN on;
    OpM om;
    on.begin(g.B + (size_t)z * g.sBz, g.sBk, n0, g.N, g.K);
    om.begin(g.A + (size_t)z * g.sAz, AK ? g.sAm : g.sAk, m0, g.M, g.K);
    typename OpN::Runs fn[AHEAD];
    typename OpM::Runs fm[AHEAD];
#pragma unroll
    for (int s = 0; s < AHEAD; ++s) {
        on.fetch(s * kStep, fn[s]);
        om.fetch(s * kStep, fm[s]);
    }
    ready();
    const uint32_t t0 = blk.tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(mh * 32);
    const bool sums = KIND == DW && g.rowsum && n0 == 0;
    float v[32] = {};
    float rows[KIND == DW ? 8 : 1] = {};  // sums of this thread's eight outputs of A over its row of k in every step
    auto wait = [&](int slot) {           // the MMAs of the slot's last step, and all before them, are complete
        if ((blk.used >> slot) & 1) mbar_wait_bounded<false>(&blk.read[slot], ((blk.parity >> slot) & 1) ^ 1, kWaitLimit, 0, blk.abort, g.status);
    };
    for_steps<RING>(steps, [&](int s, auto slot_of) {
        constexpr int slot = decltype(slot_of)::value, half = slot & 1, ahead = slot % AHEAD;
        wait(slot);
        if (s >= 2) {  // add up the sums of h h of two steps ago
            if (RING > 2) wait((slot + RING - 2) % RING);
            __syncwarp();
            tc_fence_after();
            add_columns<32>(t0 + (s & 1) * 3 * kN, v);
            tc_fence_before();
        }
        uint8_t *tn = blk.buffers + (slot >> 1) * kBufferBytes, *tm = tn + 3 * kPieceA;
#pragma unroll
        for (int i = 0; i < OpN::kRuns; ++i) {
            float x[8];
            on.elements(s * kStep, i, fn[ahead], x);
            on.store(tn, half, i, false, x);
        }
        {
            float x[8];
            om.elements(s * kStep, 0, fm[ahead], x);
            om.store(tm, half, 0, s & 1, x);
            if constexpr (KIND == DW) {
                if (sums) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) rows[e] += x[e];
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&blk.filled[slot]);
        on.fetch((s + AHEAD) * kStep, fn[ahead]);  // nothing past the end
        om.fetch((s + AHEAD) * kStep, fm[ahead]);
        if (!MMA_WARP && warp == 0) issue_when_filled<KIND, slot>(blk, g, s);
        blk.parity ^= 1u << slot;
        blk.used |= 1u << slot;
    });
#pragma unroll
    for (int r = 0; r < RING; ++r) wait(r);
    __syncwarp();
    tc_fence_after();
    if (steps > 1) add_columns<32>(t0 + (steps & 1) * 3 * kN, v);  // the last two steps' have not been added yet
    add_columns<32>(t0 + ((steps - 1) & 1) * 3 * kN, v);
    add_smaller<32>(t0, v);
    tc_fence_before();
    if constexpr (KIND == DW) {
        if (sums) {  // the buffer is free: the 32 rows of k, added in order
            float* part = reinterpret_cast<float*>(blk.buffers) + om.row * kN + 8 * (lane % OpM::kRowLanes);
#pragma unroll
            for (int e = 0; e < 8; ++e) part[e] = rows[e];
            __syncwarp();
            asm volatile("bar.sync 1, %0;" ::"n"(kFillThreads) : "memory");
            if (tid < kN && m0 + tid < g.M) {
                float t = 0.f;
#pragma unroll
                for (int r = 0; r < 32; ++r) t += reinterpret_cast<const float*>(blk.buffers)[r * kN + tid];
                g.rowsum[(size_t)z * g.sRz + m0 + tid] = t;
            }
            __syncwarp();
            asm volatile("bar.sync 1, %0;" ::"n"(kFillThreads) : "memory");  // before the next tile is filled
        }
    }
    return finish<KIND, NC, 32>(g, z, m0 + 32 * mh, n0 + 32 * q + lane, v);
}

// The ninth warp's part of a tile.
template <int KIND, int RING>
__device__ __forceinline__ void issue_tile(Block& blk, const GemmArgs& g) {
    for_steps<RING>((g.K + kStep - 1) / kStep, [&](int s, auto slot_of) {
        constexpr int slot = decltype(slot_of)::value;
        issue_when_filled<KIND, slot>(blk, g, s);
        blk.parity ^= 1u << slot;
    });
}

}  // namespace split
}  // namespace dbw
