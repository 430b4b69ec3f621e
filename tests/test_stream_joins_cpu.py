"""A round forks work onto the handle's side stream.  Whatever call of the CUDA runtime fails, that work is ordered before the caller's
stream again: a later synchronisation of that stream covers it and a stream capture stays joined.

The host side of a round (api.cu, plain C++) is compiled against a stand-in runtime that keeps, for both streams, what is ordered
before their ends, and fails one call at a time."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = next((p for p in ("/usr/local/cuda/include", "/opt/cuda/include") if os.path.exists(os.path.join(p, "cuda_runtime.h"))), None)

SOURCE = r"""
#include "api.cu"
#include <cstdio>
#include <cstdlib>

// ---- two streams; before[a][b]: how much of stream b's work is ordered before the end of stream a
static int work[2], before[2][2], calls, fail_at;
static bool unjoinable;
static int at(cudaStream_t s) { return (size_t)s == 2; }  // 1 = the caller's stream, 2 = the side stream
struct Event { int seen[2]; };
static bool failing() { return ++calls == fail_at; }
static cudaError_t queue(cudaStream_t s) {
    if (failing()) return cudaErrorUnknown;
    before[at(s)][at(s)] = ++work[at(s)];
    return cudaSuccess;
}
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (failing()) return cudaErrorUnknown;
    for (int k = 0; k < 2; ++k) ((Event*)e)->seen[k] = before[at(s)][k];
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (failing()) { unjoinable = at(s) == 0; return cudaErrorUnknown; }  // the join itself
    for (int k = 0; k < 2; ++k) before[at(s)][k] = std::max(before[at(s)][k], ((Event*)e)->seen[k]);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t s) { return queue(s); }
}

namespace dbw {
int launch_select(dbw_handle*, const double*, const int32_t*, uint8_t*, double*, double*, double*, bool, cudaStream_t s, bool) { DBW_CUDA(queue(s)); return DBW_OK; }
int launch_update_backups(dbw_handle*, const double*, int32_t*, double*, cudaStream_t s) { DBW_CUDA(queue(s)); return DBW_OK; }
int launch_mix(dbw_handle*, const float*, const float*, float, const float*, float*, cudaStream_t s) { DBW_CUDA(queue(s)); return DBW_OK; }
int launch_mix_active(dbw_handle*, const float*, const float*, float, const float*, float*, cudaStream_t s) { DBW_CUDA(queue(s)); return DBW_OK; }
bool mix_active_usable(const dbw_handle*) { return true; }
bool mix_panel_fits(const dbw_handle*) { return true; }
bool round_fused_usable(const dbw_handle*) { return false; }
int launch_grad_fp32(dbw_handle*, const float*, const int32_t*, float*, float*, cudaStream_t s, const std::function<int()>* beside) {
    DBW_CUDA(queue(s));
    if (beside) { const int rc = (*beside)(); if (rc) return rc; }
    DBW_CUDA(queue(s));
    return DBW_OK;
}
// with its last reductions on the side stream, as the tensor-core gradients have them
int launch_grad_bf16(dbw_handle* h, const float*, const int32_t*, float*, float*, cudaStream_t s, const StepArgs* step, const std::function<int()>* beside) {
    DBW_CUDA(queue(s));
    if (beside) { const int rc = (*beside)(); if (rc) return rc; }
    if (step) DBW_CUDA(cudaStreamWaitEvent(s, step->selected, 0));
    DBW_CUDA(cudaEventRecord(h->ev_dz, s));
    DBW_CUDA(queue(s));
    DBW_CUDA(cudaStreamWaitEvent(h->side, h->ev_dz, 0));
    DBW_CUDA(queue(h->side));
    DBW_CUDA(cudaEventRecord(h->ev_tail, h->side));
    DBW_CUDA(cudaStreamWaitEvent(s, h->ev_tail, 0));
    return DBW_OK;
}
}  // namespace dbw

int main() {
    static float X[64], Y[64], G[64], feat[4];
    static double t[2]; static int32_t b[2], idx[2]; static uint8_t kept[4];
    int bad = 0, joined = 0;
    for (int bf16 = 0; bf16 < 2; ++bf16)
        for (int host = 0; host < 2; ++host)
            for (int call = 0; call < 3; ++call)  // a round with gradients, one without, the gradients alone
                for (fail_at = 0;; ++fail_at) {
                    dbw_handle* h = new dbw_handle();
                    static Event ev[6];
                    std::memset(ev, 0, sizeof ev);
                    h->N = 2; h->ld = 8; h->nnz = 2; h->has_model = true; h->model.batch = 1; h->feat = feat; h->d_G = G;
                    h->flags = bf16 ? DBW_GEMM_BF16 : 0u;
                    h->side = (cudaStream_t)2;
                    h->ev_fork = (cudaEvent_t)&ev[0]; h->ev_join = (cudaEvent_t)&ev[1]; h->ev_loss = (cudaEvent_t)&ev[2];
                    h->ev_read = (cudaEvent_t)&ev[3]; h->ev_dz = (cudaEvent_t)&ev[4]; h->ev_tail = (cudaEvent_t)&ev[5];
                    h->s_t = t;
                    std::memset(work, 0, sizeof work);
                    std::memset(before, 0, sizeof before);
                    calls = 0; unjoinable = false;
                    int rc;
                    if (call == 2)
                        rc = dbw_grad(h, X, idx, G, nullptr, (void*)1);
                    else if (host)
                        rc = dbw_round_host(h, X, t, nullptr, call == 0 ? idx : nullptr, nullptr, 0.1f, Y, kept, t, t, X, b, (void*)1);
                    else
                        rc = dbw_round(h, X, t, b, call == 0 ? idx : nullptr, G, 0.1f, nullptr, Y, kept, t, nullptr, t, nullptr, (void*)1);
                    const bool done = fail_at > 0 && calls < fail_at;
                    if ((fail_at == 0 || done) != (rc == DBW_OK)) { std::printf("bf16 %d host %d call %d: failure %d returned %d\n", bf16, host, call, fail_at, rc); ++bad; }
                    if (before[0][1] != work[1] && !unjoinable) { std::printf("bf16 %d host %d call %d: not joined after failure %d\n", bf16, host, call, fail_at); ++bad; }
                    joined += work[1] > 0;
                    if (done) break;
                }
    std::printf("%d calls with work on the side stream\n", joined);
    std::fflush(stdout);
    std::_Exit(bad ? 1 : joined > 40 ? 0 : 2);
}
"""


@pytest.mark.skipif(CUDA is None or shutil.which("g++") is None, reason="needs g++ and the CUDA headers")
def test_side_stream_is_joined_whatever_call_fails(tmp_path):
    src, exe = tmp_path / "joins.cpp", tmp_path / "joins"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O0", "-I" + CUDA, "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_2102_06280_b200", "csrc"), str(src), "-o", str(exe), "-Wl,--unresolved-symbols=ignore-all"],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
