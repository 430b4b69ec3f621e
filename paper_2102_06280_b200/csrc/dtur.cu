// Distributed threshold-based update rule (Section 4.1) and one iteration of Algorithm 2.
// One CTA: the state is N-1 flags and two counters, the work is O(N + nnz).
#include "common.cuh"

namespace dbw {

namespace {

constexpr int kThreads = 1024;

__device__ __forceinline__ double time_or_inf(double t, uint32_t* status) {
    if (t != t) {
        atomicOr(status, DBW_STATUS_NAN_TIME);
        return __longlong_as_double(0x7ff0000000000000LL);
    }
    return t;
}

// Bound by the latency of its dependent loads, so each phase issues all of its loads at once: the times (ordered, NaN last)
// go to shared memory while the links are on their way, every thread takes kPer links, and later kPer workers, side by side.
// 4096 workers, 8 neighbours: 7.9 us (8.4 with one link and one neighbour at a time, times from L2).
// STAGED = false: more workers than shared memory has room for; the times are read through L2.
constexpr int kPer = 4;
constexpr int kMaxStaged = 6016;  // times in shared memory: 47 KB

// LANES lanes share a worker in the last phase: eight where all workers then fit one pass (up to 512: 64 workers with 13
// neighbours take 5.4 us, with one lane 9.1), else one (4096 workers: 7.9 us, with eight 13).
template <bool STAGED, int LANES>
__global__ void __launch_bounds__(kThreads)
update_backups_kernel(int N, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                      const int32_t* __restrict__ links, int32_t* covered, int32_t* epoch,
                      const double* __restrict__ t, int32_t* __restrict__ b_out, double* theta_out,
                      uint32_t* status) {
    dependent_begin();
    extern __shared__ double times[];
    const int D = N - 1;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double inf = __longlong_as_double(0x7ff0000000000000LL);
    auto time_of = [&](int j) { return STAGED ? times[j] : time_or_inf(t[j], status); };
    if (STAGED) {
        for (int j0 = tid; j0 < N; j0 += kPer * kThreads) {
            double v[kPer];
#pragma unroll
            for (int u = 0; u < kPer; ++u) v[u] = j0 + u * kThreads < N ? t[j0 + u * kThreads] : 0.0;
#pragma unroll
            for (int u = 0; u < kPer; ++u)
                if (j0 + u * kThreads < N) times[j0 + u * kThreads] = time_or_inf(v[u], status);
        }
    }
    // theta: earliest establishment time max(t_u, t_v) among the uncovered links, first on ties
    double best = inf;
    int best_pos = 0x7fffffff;
    bool staged = !STAGED;
    for (int pos0 = tid; pos0 < D || !staged; pos0 += kPer * kThreads) {
        int cov[kPer];
        int2 uv[kPer];
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int pos = pos0 + u * kThreads;
            cov[u] = pos < D ? covered[pos] : 1;
            uv[u] = pos < D ? __ldg(reinterpret_cast<const int2*>(links) + pos) : make_int2(0, 0);
        }
        if (!staged) {
            __syncthreads();  // the times are in shared memory
            staged = true;
        }
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            if (cov[u]) continue;
            const int pos = pos0 + u * kThreads;
            const double est = fmax(time_of(checked(uv[u].x, N, status)), time_of(checked(uv[u].y, N, status)));
            if (est < best || (est == best && pos < best_pos)) {
                best = est;
                best_pos = pos;
            }
        }
    }
    // The rows of the first workers (eight lanes: their first eight neighbours too) do not depend on theta: on their way during
    // the reduction.
    constexpr int kGroups = kThreads / LANES;
    const int sub = tid % LANES, group = tid / LANES;
    int lo[kPer], hi[kPer], c[kPer];
    auto rows_of = [&](int j0) {
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int j = j0 + u * kGroups;
            lo[u] = j < N ? rowptr[j] : 0;
            hi[u] = j < N ? rowptr[j + 1] : 0;
        }
    };
    rows_of(group);
    if (LANES > 1) {
#pragma unroll
        for (int u = 0; u < kPer; ++u) c[u] = lo[u] + sub < hi[u] ? col[lo[u] + sub] : -1;
    }
    __shared__ double s_best[32];
    __shared__ int s_pos[32];
    __shared__ double s_theta;
    __shared__ int s_clear;
    auto reduce = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int op = __shfl_xor_sync(0xffffffffu, best_pos, o);
            if (ob < best || (ob == best && op < best_pos)) {
                best = ob;
                best_pos = op;
            }
        }
    };
    reduce();
    if (lane == 0) {
        s_best[warp] = best;
        s_pos[warp] = best_pos;
    }
    __syncthreads();
    if (warp == 0) {
        best = s_best[lane];
        best_pos = s_pos[lane];
        reduce();
        if (lane == 0) {
            int clear = 0;
            if (best_pos != 0x7fffffff) {
                covered[best_pos] = 1;
                const int step = epoch[0] + 1;
                epoch[1] = best_pos;
                clear = step == D;
                epoch[0] = clear ? 0 : step;
            }
            s_theta = best;
            s_clear = clear;
            if (theta_out) *theta_out = best;
        }
    }
    __syncthreads();
    const double theta = s_theta;
    if (s_clear)
        for (int pos = tid; pos < D; pos += kThreads) covered[pos] = 0;
    // threshold rule: on-time workers wait for their on-time neighbours, late workers for nobody
    if (LANES > 1) {
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int j = group + u * kGroups;
            if (j >= N) break;  // the same for the lanes of a worker
            int p = 0;
            if (time_of(j) <= theta) {
                if (c[u] >= 0) p = time_of(checked(c[u], N, status)) <= theta;
                for (int e = lo[u] + LANES + sub; e < hi[u]; e += LANES) p += time_of(checked(col[e], N, status)) <= theta;
            }
#pragma unroll
            for (int o = LANES / 2; o > 0; o >>= 1) p += __shfl_xor_sync(0xffu << (tid & 24), p, o);
            if (sub == 0) b_out[j] = hi[u] - lo[u] - p;
        }
        return;
    }
    for (int j0 = tid; j0 < N; j0 += kPer * kThreads) {
        if (j0 != tid) rows_of(j0);
        int p[kPer], longest = 0;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int j = j0 + u * kThreads;
            p[u] = lo[u] - hi[u];  // minus the degree, then plus one for every neighbour waited for
            if (j < N && time_of(j) <= theta) longest = max(longest, hi[u] - lo[u]);
            else hi[u] = lo[u];  // late
        }
        for (int k = 0; k < longest; k += 2) {
            int e[kPer][2];
#pragma unroll
            for (int u = 0; u < kPer; ++u)
#pragma unroll
                for (int f = 0; f < 2; ++f) e[u][f] = lo[u] + k + f < hi[u] ? col[lo[u] + k + f] : -1;
#pragma unroll
            for (int u = 0; u < kPer; ++u)
#pragma unroll
                for (int f = 0; f < 2; ++f)
                    if (e[u][f] >= 0) p[u] += time_of(checked(e[u][f], N, status)) <= theta;
        }
#pragma unroll
        for (int u = 0; u < kPer; ++u)
            if (j0 + u * kThreads < N) b_out[j0 + u * kThreads] = -p[u];
    }
}

}  // namespace

int launch_update_backups(dbw_handle* h, const double* t, int32_t* b_out, double* theta_out, cudaStream_t s) {
    if (h->N <= kPer * kThreads / 8)
        launch(update_backups_kernel<true, 8>, 1, kThreads, (size_t)h->N * sizeof(double), s, h->N, h->d_rowptr, h->d_col, h->d_links, h->d_covered,
                                                                                         h->d_epoch, t, b_out, theta_out, h->d_status);
    else if (h->N <= kMaxStaged)
        launch(update_backups_kernel<true, 1>, 1, kThreads, (size_t)h->N * sizeof(double), s, h->N, h->d_rowptr, h->d_col, h->d_links, h->d_covered,
                                                                                      h->d_epoch, t, b_out, theta_out, h->d_status);
    else
        launch(update_backups_kernel<false, 1>, 1, kThreads, 0, s, h->N, h->d_rowptr, h->d_col, h->d_links, h->d_covered, h->d_epoch, t, b_out,
                                                            theta_out, h->d_status);
    DBW_LAUNCHED();
    return DBW_OK;
}

}  // namespace dbw
