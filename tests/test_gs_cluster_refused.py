"""A Gauss-Seidel sweep whose cluster launch the runtime refuses (a partition of the
SMs too small for a cluster) goes on colour by colour: the host side of the sweep
against a runtime that only records the launches."""
import ctypes
import os
import subprocess

import pytest

from paper_2102_01734_gb300 import build

RUNTIME = r"""
#include <cstddef>
#include <cstring>
#include <map>
#include <string>
struct dim3 { unsigned x, y, z; };
static std::map<const void *, std::string> names;
static std::string log_;
static int refuse_from = 1 << 30, clusters = 0, last = 0;
extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *f, char *, const char *name, int, void *, void *, void *, void *, int *) {
    names[f] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
static dim3 g_, b_;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t, void *) { g_ = g; b_ = b; return 0; }
int __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *m, void *s) {
    *g = g_;
    *b = b_;
    *m = 0;
    *(void **)s = nullptr;
    return 0;
}
int __cudaGetKernel(const void **k, const void *f) { *k = f; return 0; }
int __cudaLaunchKernel(const void *f, dim3, dim3, void **args, size_t, void *) {
    log_ += names[f].find("gs_colour_kernel") != std::string::npos ? "c" + std::to_string(*(int *)args[4]) + " " : "? ";
    return 0;
}
int cudaLaunchKernel(const void *f, dim3 g, dim3 b, void **args, size_t m, void *s) { return __cudaLaunchKernel(f, g, b, args, m, s); }
int cudaLaunchKernelExC(const void *, const void *f, void **args) {
    const bool plane = names[f].find("gs_plane_kernel") != std::string::npos;
    if (clusters++ >= refuse_from) return last = 912;
    log_ += plane ? "p" + std::to_string(*(int *)args[4]) + " " : "? ";
    return 0;
}
int cudaLaunchCooperativeKernel(const void *, dim3, dim3, void **, size_t, void *) { return 0; }
int cudaFuncSetAttribute(const void *, int, int) { return 0; }
int cudaGetLastError() { const int e = last; last = 0; return e; }
int cudaMemsetAsync(void *, int, size_t, void *) { return 0; }
const char *launches() { return log_.c_str(); }
void refuse(int n) { refuse_from = n; clusters = 0; last = 0; log_.clear(); }
}
namespace rt3d { int device_sm_count() { return 152; } }
"""

CALL = r"""
#include "rt3d_internal.cuh"
extern "C" int sweep(int nx, int ny, int nz, int pz, int *n) {
    static double d[1];
    return (int)rt3d::launch_gs_sweep(nx, ny, nz, rt3d::colour_geo(nx, ny, nz), d, true, d, d, d, d, nullptr, nullptr,
                                      1, 1e-3, nullptr, nullptr, rt3d::Periodic{true, true, pz != 0}, n);
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    build.build()
    d = str(tmp_path_factory.mktemp("host"))
    paths = {n: os.path.join(d, n) for n in ("runtime.cpp", "call.cu", "call.o", "host.so")}
    for name, text in (("runtime.cpp", RUNTIME), ("call.cu", CALL)):
        with open(paths[name], "w") as f:
            f.write(text)
    subprocess.run([build.nvcc(), *build._flags(["-I", build.SRC_DIR]), "-c", paths["call.cu"], "-o", paths["call.o"]],
                   check=True)
    # -Bsymbolic: this runtime also where the process has loaded the real one
    subprocess.run(["g++", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-o", paths["host.so"], paths["runtime.cpp"],
                    paths["call.o"], os.path.join(build.OUT_DIR, "ali.o")], check=True)
    lib = ctypes.CDLL(paths["host.so"])
    lib.launches.restype = ctypes.c_char_p
    return lib


@pytest.mark.parametrize("n,periodic_z,refused_after,expected", [
    ((65, 64, 33), False, 99, "p0 p1"),
    ((65, 64, 1), False, 99, "p0"),
    ((65, 64, 33), True, 99, "c0 c1 c2 c3 c4 c5 c6 c7"),
    ((65, 64, 33), False, 0, "c0 c1 c2 c3 c4 c5 c6 c7"),
    ((65, 64, 33), False, 1, "p0 c4 c5 c6 c7"),
    ((65, 64, 1), False, 0, "c0 c1 c2 c3 c4 c5 c6 c7"),
])
def test_sweep(host, n, periodic_z, refused_after, expected):
    host.refuse(refused_after)
    count = ctypes.c_int()
    assert host.sweep(*n, int(periodic_z), ctypes.byref(count)) == 0
    assert host.launches().decode().strip() == expected
    assert count.value == len(expected.split())
    assert host.cudaGetLastError() == 0  # the refusal is not left for the next caller
