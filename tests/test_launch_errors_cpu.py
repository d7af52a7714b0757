"""A kernel launch that fails is reported by the launcher and leaves no error
behind in the runtime, where the next launch of another context would report it
as its own.  The launchers run against a fake runtime whose launches fail."""
import subprocess
from pathlib import Path

from paper_1510_04068_gb300 import build

FAKE = r"""
#include <cstdio>
#include "sp2_internal.h"

static cudaError_t last = cudaSuccess;
static int launches = 0;
extern "C" {
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) {
    ++launches;
    return last = cudaErrorInvalidConfiguration;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t __cudaGetKernel(void **, const void *) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void *, dim3, dim3, void **, size_t, cudaStream_t) { return cudaSuccess; }
}

using namespace sp2;
static int bad = 0;
static void expect(const char *what, cudaError_t e) {
    if (e != cudaErrorInvalidConfiguration || last != cudaSuccess) {
        std::printf("%s: returned %d, left %d\n", what, int(e), int(last));
        ++bad;
    }
    last = cudaSuccess;
}

int main() {
    JStore js{}, cached{};
    cached.dsc = reinterpret_cast<float4 *>(64);
    expect("scatter", launch_scatter_j(js, nullptr, 1, 1, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0));
    expect("dscache", launch_dscache(4, cached, 0, 1, 0));
    for (int order = 2; order <= 6; order += 2)
        for (int mixed = 0; mixed < 2; ++mixed) {
            expect("predict", launch_predict(order, mixed, js, 1, 0.0, nullptr, 0));
            expect("predict from the cache", launch_predict(order, mixed, cached, 1, 0.0, nullptr, 0));
            expect("block predict", launch_block_predict(order, mixed, cached, 1, nullptr, BlockStep{}, 0));
        }
    for (int mixed = 0; mixed < 2; ++mixed) {
        expect("pack", launch_pack_state(mixed, 1, nullptr, nullptr, nullptr, nullptr, 0));
        expect("predict pack", launch_h4_predict_pack(mixed, 1, 0.0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0));
        expect("vjp pre", launch_h4_vjp_pre(mixed, 1, 0.0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0));
        expect("pack vjp", launch_pack_vjp(mixed, 1, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0));
    }
    expect("correct", launch_h4_correct(1, 0.0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0));
    expect("vjp post", launch_h4_vjp_post(1, 0.0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0));
    expect("block correct", launch_block_correct_dev(js, BlockStep{}, 1, nullptr, nullptr, 0.0, 0.0, 0));
    expect("lists", launch_nb_finish(nullptr, 1, 1, nullptr, nullptr, 0));
    for (int nn = 0; nn < 2; ++nn) {
        ForceParams p{};
        p.n_i = p.split = 2;
        expect("reduce", launch_reduce_h2m(KernelKey{K_FORCE, 2, 1, nn, 1}, p, 0));
    }
    std::printf("%d launches\n", launches);
    return bad;
}
"""


def test_failed_launches_are_reported_once(tmp_path):
    build.build()
    src, exe = tmp_path / "fake.cpp", tmp_path / "fake"
    src.write_text(FAKE)
    cuda = Path(build._nvcc()).resolve().parents[1]
    objs = [build.BUILD / "obj" / f"{name}.o" for name in ("sp2_predict", "sp2_kernels_h2m")]
    # the other runtime calls of the force kernels' file are not reached
    subprocess.run(["g++", "-std=c++17", f"-I{build.CSRC}", f"-I{build.INCLUDE}", f"-I{cuda}/include", str(src),
                    *map(str, objs), "-Wl,--unresolved-symbols=ignore-all", "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout.split()[0]) >= 30
