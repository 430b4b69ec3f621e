"""Which rounds the pipelined panel mix takes, and with what panels: the host side of mix_pipe.cu, compiled against a stand-in for the driver's tensor maps."""
import os
import shutil
import subprocess

import pytest

from tests.test_gpu_kernels import PIPE_SHAPES

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

SOURCE = r"""
#define encode_tiled_fn driver_encode_tiled_fn
#include "tc_ptx.cuh"
#undef encode_tiled_fn
namespace dbw {
static bool there = true;
static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                       CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
static EncodeTiledFn encode_tiled_fn() { return there ? encode : nullptr; }
}
#include "mix_pipe.cu"
#include <cstdio>
#include <cstdlib>
namespace dbw { std::atomic<long long> g_launches; std::atomic<int> g_last_cuda_error; }
int main(int argc, char** argv) {
    using namespace dbw;
    for (int k = 1; k + 2 < argc; k += 3) {
        dbw_handle h;
        h.N = std::atoi(argv[k]); h.ld = (std::atoll(argv[k + 2]) + 3) / 4 * 4; h.sm_count = 148; h.smem_optin = 232448;
        h.plan.stride = std::max(4, (std::atoi(argv[k + 1]) + 3) / 4 * 4);
        for (bool gradient : {true, false}) {
            there = true;
            const Shape s = mix_pipe_usable(&h, gradient) ? shape_of(&h, gradient) : Shape{};
            there = false;
            if (mix_pipe_usable(&h, gradient)) return 1;  // the plain kernel's then
            std::printf("%d %d ", 4 * s.gs, s.gs ? s.per_sm : 0);
        }
        std::printf("\n");
    }
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("needs nvcc")
    at = tmp_path_factory.mktemp("pipe")
    (at / "shapes.cu").write_text(SOURCE)
    subprocess.run([NVCC, "-std=c++17", "-O0", "-gencode", "arch=compute_100a,code=sm_100a", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2102_06280_b200", "csrc"), "-o", str(at / "shapes"), str(at / "shapes.cu")],
                   check=True, capture_output=True, text=True)

    def of(cases):
        r = subprocess.run([str(at / "shapes")] + [str(v) for c in cases for v in c], capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, "taken without tensor maps"
        return [tuple(int(v) for v in line.split()) for line in r.stdout.splitlines()]
    return of


def test_shapes_of_the_gpu_test_reach_every_panel_width(shapes):
    """Columns of a panel and blocks to an SM, with and without gradients, of the rounds that are compared with the plain kernel on the GPU."""
    assert shapes([c[:3] for c in PIPE_SHAPES]) == [c[3] for c in PIPE_SHAPES]
    with_gradient, without = {c[3][:2] for c in PIPE_SHAPES}, {c[3][2:] for c in PIPE_SHAPES}
    for reached in (with_gradient, without):
        assert reached >= {(256, 2), (128, 2), (64, 2), (32, 2), (32, 1)}


def test_small_matrices_are_left_to_the_plain_kernel(shapes):
    assert shapes([(15, 4, 60_000), (96, 6, 20_000), (128, 8, 50_000), (1024, 8, 1_000_000)]) == [(0, 0, 0, 0)] * 4
