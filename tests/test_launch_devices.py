"""Kernel launches on every device of a process, without a GPU: the library's
launchers are linked against a CUDA runtime of this file's own, which has three
devices and, like the real one, refuses a launch with more than 48 KB of dynamic
shared memory unless the kernel was given as much on the device that is current.
A launcher must set that up on each device that it launches on, not only on the
first one."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1208_2407_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <map>
#include <utility>
#include <vector>
#include "internal.h"

static int device = 0;
static int refused = 0, launched = 0, most = 0;
static std::map<std::pair<int, const void *>, int> limit;
static cudaError_t last = cudaSuccess;

extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *,
                            void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
int __cudaPopCallConfiguration(void *, void *, size_t *, void *) { return 0; }
cudaError_t __cudaGetKernel(void **, const void *) { return cudaErrorUnknown; }
cudaError_t __cudaLaunchKernel() { return cudaErrorUnknown; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *)
{ return cudaErrorUnknown; }
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v)
{
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limit[{device, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int,
                                                                   size_t, unsigned)
{ *n = 2; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **)
{
    const int smem = (int)c->dynamicSmemBytes;
    ++launched;
    if (smem > most) most = smem;
    auto it = limit.find({device, f});
    if (smem <= 48 << 10 || (it != limit.end() && it->second >= smem)) return cudaSuccess;
    ++refused;
    return last = cudaErrorInvalidValue;
}
}

namespace ts {
void count_launches(int64_t) {}
}

static void check(cudaError_t e, const char *what, int K, int i)
{
    if (e != cudaSuccess) printf("device %d: %s depth %d (%d) refused\n", device, what, K, i);
}

int main()
{
    static ts::ScaledCoef sc;
    static CUtensorMap tm;
    for (device = 0; device < 3; ++device) {
        if (ts::num_sms() != 152) printf("SM count\n");
        for (int K = 1; K <= ts::TILE_MAX_K; ++K) {
            ts::TileLaunch t = {};
            t.nx = t.ny = 300;
            t.pitch = 320;
            t.sc = &sc;
            for (int s = 0; s < ts::TILE_SHAPES; ++s)
                check(ts::launch_tile(K, s, t, nullptr), "tiles", K, s);
            for (int s = 0; s < 3; ++s)
                check(ts::launch_tile_multi(K, s, nullptr, 2, 7, 0, nullptr), "multi-grid tiles", K, s);
            ts::TileAdjoint a = {};
            a.nx = a.ny = 300;
            a.pitch = 320;
            check(ts::launch_tile_adjoint(K, a, sc, nullptr), "backward tiles", K, 0);
        }
        for (int scaled = 0; scaled < 2; ++scaled) {
            ts::FusedLaunch f = {};
            f.tm_state = f.tm_phase = f.tm_b = &tm;
            f.nx = f.ny = 5000;
            f.pitch = 5024;
            f.sc = scaled ? &sc : nullptr;
            const int most_k = scaled ? ts::FUSED_MAX_K : ts::FUSED_LIFT_MAX_K;
            for (int K = 1; K <= most_k; ++K) {
                check(ts::launch_fused(K, f, nullptr), "steps", K, scaled);
                if (K <= ts::FUSED_DRIVE_MAX_K)
                    check(ts::launch_fused_drive(K, f, nullptr), "driven steps", K, scaled);
                if (K <= ts::FUSED_ADJ_MAX_K)
                    check(ts::launch_fused_adjoint(K, f, nullptr), "backward steps", K, scaled);
                check(ts::fused_multi_prepare(K), "preparation", K, scaled);
                const int nx[2] = {5000, 300}, ny[2] = {5000, 200};
                ts::EpochEntry tab[2];
                ts::MultiPlan plan = ts::fused_multi_plan(K, scaled, 2, nx, ny, tab);
                check(ts::launch_fused_multi(K, scaled, tab, 2, plan, 0, nullptr, nullptr),
                      "multi-grid steps", K, scaled);
            }
            check(ts::launch_fused_u4(f, nullptr), "fourth-order step", 5, scaled);
            check(ts::launch_fused3d(f, 30, nullptr), "3-D step", 1, scaled);
        }
    }
    printf("%d launches, %d refused, at most %d bytes\n", launched, refused, most);
    return refused || most <= 48 << 10;   // (some kernel must need the larger size)
}
"""


def test_every_launcher_works_on_every_device(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    from paper_1208_2407_gb300 import build
    try:
        nvcc = build.nvcc()
    except Exception:
        pytest.skip("nvcc not available")
    build.build()
    include = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    src, exe = tmp_path / "devices.cpp", tmp_path / "devices"
    src.write_text(PROGRAM)
    names = ["tile", "tile_adjoint"] + ["fused_%d" % i for i in range(build.FUSED_PARTS)]
    objs = [os.path.join(build.BUILD, n + ".o") for n in names]
    cmd = ["g++", "-std=c++17", "-O1", "-I" + CSRC, "-I" + include, str(src), "-o", str(exe)] + objs
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout[-3000:]
