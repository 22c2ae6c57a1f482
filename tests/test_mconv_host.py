"""Host side of csrc/mconv.cu, csrc/fconv.cu and csrc/bnorm.cu without a GPU: their objects linked against a runtime that records launches and refuses the
ones it is told to."""
import os
import subprocess

import pytest

from paper_2509_05679_b200 import build

FAKE = r"""
#include "kernels.h"
#include "launch.h"
#include <algorithm>
#include <cstdio>
#include <cstdlib>
using namespace fdg;

static cudaError_t last = cudaSuccess;      // CUDA's last error
static int refuse = 0;                      // this many launches are refused
static std::vector<const void*> ran;        // kernels of the others
static std::vector<std::pair<dim3, size_t>> grids;      // and their grids and shared memory
extern "C" {
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { abort(); }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
unsigned __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return 0; }
}
namespace fdg {
cudaError_t allow_smem(OncePerDevice&, const void*, int) { return cudaSuccess; }
cudaError_t launch_raw(const void* f, dim3 grid, dim3, size_t smem, cudaStream_t, void**, const size_t*, int, int) {
    if (refuse > 0) { --refuse; return last = cudaErrorInvalidConfiguration; }
    ran.push_back(f);
    grids.push_back({grid, smem});
    return cudaSuccess;
}
Scope::Scope(int, double, double, cudaStream_t) {}
Scope::~Scope() {}
}
static ConvGeom conv(int n, int h, int w, int c, int co, int r, int stride) {
    ConvGeom g{}; g.N = n; g.H = h; g.W = w; g.C = c; g.Co = co; g.R = r; g.stride = stride; g.pad = r == 3;
    g.Ho = (h + 2 * g.pad - r) / stride + 1; g.Wo = (w + 2 * g.pad - r) / stride + 1;
    return g;
}
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
"""

REFUSED = r"""
int main() {
    alignas(16) static char b[16];
    const ConvGeom g = conv(8, 16, 16, 32, 32, 3, 1);
    const Packed pk{b, 0};
    PackArgs a{}; a.n = 1; a.layer[0] = PackLayer{0, 0, 32, 32, 9, 0};
    for (int dt = 0; dt < 2; ++dt) {
        // taken: one launch, the tensor-core kernel's
        CHECK(fconv_forward(dt, b, b, nullptr, b, g, 0, 1, 0, 0, nullptr, pk, 0) && ran.size() == 1);
        const void* const tensor = ran[0]; ran.clear();
        // refused: the packed-FMA kernel computes the same layer, and nobody finds an error afterwards
        refuse = 1;
        CHECK(fconv_forward(dt, b, b, nullptr, b, g, 0, 1, 0, 0, nullptr, pk, 0));
        CHECK(ran.size() == 1 && ran[0] != tensor && last == cudaSuccess); ran.clear();
        refuse = 1;
        CHECK(fconv_dgrad(dt, b, b, b, g, 0, 1, 0, pk, 0) && ran.size() == 1 && ran[0] != tensor && last == cudaSuccess); ran.clear();
        refuse = 1;
        CHECK(fconv_wgrad(dt, b, b, (float*)b, (float*)b, g, 1, 0, false, true, 0) && ran.size() == 2 && last == cudaSuccess); ran.clear();    // and its reduction
        // the layout of the weights says whether it is there
        CHECK(mconv_pack(dt, b, 0, b, 0, a, 4, 1, 0) && ran.size() == 1); ran.clear();
        refuse = 1;
        CHECK(!mconv_pack(dt, b, 0, b, 0, a, 4, 1, 0) && ran.empty() && last == cudaSuccess);
    }
    return 0;
}
"""


def run(tmp_path, program):
    inc = "/usr/local/cuda/include"
    if not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    build.build_lib()
    objs = [os.path.join(build.CSRC, f) for f in ("mconv.o", "fconv.o", "bnorm.o")]
    if not all(os.path.exists(o) for o in objs):
        pytest.skip("the library was built elsewhere: no objects")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(FAKE + program)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", inc, "-I", build.CSRC, str(src), *objs, "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_a_refused_launch_is_made_up_for(tmp_path):
    run(tmp_path, REFUSED)


ONE_WAVE = r"""
int main() {
    alignas(16) static char b[16];
    for (int dt = 0; dt < 2; ++dt)
        for (const ConvGeom& g : {conv(64, 28, 28, 32, 64, 3, 2), conv(192, 32, 32, 16, 32, 3, 2), conv(768, 4, 4, 64, 64, 3, 1), conv(192, 16, 16, 32, 32, 3, 1), conv(500, 2, 2, 16, 16, 3, 1),
                                  conv(96, 32, 32, 16, 16, 1, 1), conv(64, 12, 20, 48, 32, 3, 2)}) {
            grids.clear();
            CHECK(fconv_wgrad(dt, b, b, (float*)b, (float*)b, g, 1, 0, false, true, 0));
            const dim3 n = grids[0].first;
            CHECK((long)n.x * n.y * n.z <= std::min(dt ? 3 : 4, (int)(228 * 1024 / (grids[0].second + 1024))) * 148L);
        }
    return 0;
}
"""


def test_a_weight_gradient_is_one_wave(tmp_path):
    """As many CTAs as 148 SMs hold at a time: registers for four (bf16 storage three), 228 KB of shared memory with 1 KB more for each than it asks for."""
    run(tmp_path, ONE_WAVE)


TAKEN = r"""
// the kernel that a launch ran is the one that mconv_takes says
static bool agrees(int dt, const ConvGeom& g, int groups, bool back, bool& taken) {
    alignas(16) static char b[16];
    const void* ran_[2];
    for (int p = 0; p < 2; ++p) {
        const Packed pk{p ? b : nullptr, 0};
        ran.clear();
        if (!(back ? fconv_dgrad(dt, b, b, b, g, 0, groups, 0, pk, 0) : fconv_forward(dt, b, b, nullptr, b, g, 0, groups, 0, 0, nullptr, pk, 0)) || ran.size() != 1) { taken = false; return !mconv_takes(dt, g, groups, back); }
        ran_[p] = ran[0];
    }
    taken = ran_[0] != ran_[1];
    return taken == mconv_takes(dt, g, groups, back);
}
int main() {
    int n[2] = {};
    for (int dt = 0; dt < 2; ++dt) for (int r : {1, 3}) for (int st : {1, 2}) for (int h : {1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 13, 14, 16, 17, 20, 28, 32}) for (int w : {1, 2, 5, h})
        for (int c : {16, 48, 64}) for (int images : {1, 4, 12, 192}) for (int groups : {1, 4}) for (int back = 0; back < 2; ++back) {
            if (images % groups) continue;
            bool taken;
            CHECK(agrees(dt, conv(images, h, w, c, 32, r, st), groups, back, taken));
            ++n[taken];
        }
    CHECK(n[0] > 1000 && n[1] > 1000);
    // ordinary sizes, and the ends of each line of the rule
    struct { int dt, images, side, c, co, r, st; bool back, taken; } list[] = {
        {0, 192, 32, 16, 16, 3, 1, false, true}, {0, 192, 8, 64, 64, 3, 1, true, true}, {0, 192, 32, 16, 32, 3, 2, false, true}, {0, 192, 32, 16, 32, 3, 2, true, true}, {0, 192, 32, 16, 32, 1, 2, false, true},
        {0, 192, 14, 64, 64, 3, 1, false, true}, {0, 16, 14, 16, 16, 3, 1, false, true}, {0, 192, 5, 32, 32, 3, 1, false, false}, {0, 768, 9, 64, 64, 3, 1, false, true}, {0, 768, 5, 64, 64, 3, 1, false, false}, {0, 768, 1, 16, 16, 3, 1, false, false},
        {0, 192, 28, 16, 16, 3, 2, false, false}, {0, 768, 4, 32, 64, 3, 2, true, true}, {0, 16, 4, 32, 64, 3, 2, true, false},
        {0, 4, 32, 16, 16, 1, 1, false, true}, {0, 16, 16, 16, 16, 1, 1, false, false}, {0, 64, 16, 48, 48, 1, 1, false, true}, {0, 768, 3, 64, 64, 1, 1, false, false}, {0, 768, 5, 64, 64, 1, 1, false, true},
        {1, 192, 1, 16, 16, 3, 1, false, false}, {1, 4096, 1, 256, 256, 3, 1, false, true}, {1, 192, 2, 16, 16, 3, 1, false, true}, {1, 16, 2, 64, 64, 1, 1, false, false}, {1, 192, 2, 64, 64, 1, 1, false, true}};
    for (const auto& l : list) {
        bool taken;
        if (!agrees(l.dt, conv(l.images, l.side, l.side, l.c, l.co, l.r, l.st), 1, l.back, taken) || taken != l.taken)
            { printf("dt%d %d images of %d, %d -> %d k%d s%d %s: %d\n", l.dt, l.images, l.side, l.c, l.co, l.r, l.st, l.back ? "back" : "forward", taken); return 1; }
    }
    return 0;
}
"""


def test_one_rule_says_who_takes_a_launch(tmp_path):
    """What decides whether weights are laid out is what decides who reads them."""
    run(tmp_path, TAKEN)


SLICES = r"""
static int slice(int channels, int workers, long rows, int modules) {
    alignas(16) static char b[16];
    const float* const f = (const float*)b;
    grids.clear();
    bnc_forward(b, f, f, nullptr, b, (float*)b, workers, workers, modules, rows, channels, true, 0);
    return channels * 8 / (int)grids[0].first.x;         // eight CTAs a cluster
}
int main() {
    // 12288 rows: 24 a thread of 32 channels
    CHECK(slice(64, 2, 12288, 1) == 16 && slice(64, 2, 12288, 2) == 32 && slice(64, 2, 12288, 4) == 32);
    CHECK(slice(32, 4, 12288, 1) == 16 && slice(32, 4, 12288, 2) == 16 && slice(32, 4, 12288, 3) == 32);
    // 18 rows, 20 rows a thread and one row more
    CHECK(slice(64, 2, 9216, 1) == 32 && slice(32, 4, 10240, 1) == 32 && slice(32, 4, 10241, 1) == 16);
    return 0;
}
"""


def test_batch_norm_slices_leave_the_other_modules_room(tmp_path):
    run(tmp_path, SLICES)
