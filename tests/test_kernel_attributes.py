"""Kernel attributes (large shared memory, clusters above the portable size) belong to one device: the library sets
them, and picks its cluster sizes, on every device a process uses.  Checked on the host: the library's objects linked
against a runtime of two devices that records what is set on which."""
import os
import subprocess

from paper_2012_13618_gb300 import _build

_SRC = r"""
#include <cstdio>
#include <map>
#include <set>
#include <utility>

static int g_dev = 0;
static std::set<std::pair<int, const void *>> g_set[2];

extern "C" {
int cudaGetDevice(int *d) { *d = g_dev; return 0; }
int cudaGetLastError() { return 0; }
const char *cudaGetErrorString(int) { return ""; }
int cudaFuncSetAttribute(const void *f, int attr, int) { g_set[g_dev].insert({attr, f}); return 0; }
int cudaOccupancyMaxActiveClusters(int *n, const void *, const void *config) {
    // the second device runs clusters of at most 8 blocks
    *n = g_dev == 1 && *static_cast<const unsigned *>(config) > 8 ? 0 : 1;
    return 0;
}
void **__cudaRegisterFatBinary(void *) { static void *h = nullptr; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
int __cudaGetKernel(void **, const void *) { return 0; }
int cudaGetFuncBySymbol(void **, const void *) { return 0; }
}

namespace bp {
void refine_init();
void coarsen_init();
int tail_cluster();
}

int main() {
    int c[2];
    for (int round = 0; round < 2; ++round)
        for (g_dev = 0; g_dev < 2; ++g_dev) {
            bp::refine_init();
            bp::coarsen_init();
            c[g_dev] = bp::tail_cluster();
        }
    std::printf("attributes %zu %zu, clusters %d %d\n", g_set[0].size(), g_set[1].size(), c[0], c[1]);
    return !(g_set[0].size() == 6 && g_set[1] == g_set[0] && c[0] == 16 && c[1] == 8);
}
"""


def test_attributes_are_set_on_every_device(tmp_path):
    _build.build()
    objs = []
    for name in ("refine_loop", "coarsen", "tail"):
        obj = os.path.join(_build.BUILD, name + ".cu.o")
        if not os.path.exists(obj):
            obj = str(tmp_path / (name + ".o"))
            subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-c", os.path.join(_build.CSRC, name + ".cu"),
                            "-o", obj], check=True, capture_output=True)
        objs.append(obj)
    src = tmp_path / "attributes.cpp"
    src.write_text(_SRC)
    exe = tmp_path / "attributes"
    r = subprocess.run(["g++", "-O1", "-std=c++17", "-o", str(exe), str(src), *objs, "-lpthread",
                        "-Wl,--unresolved-symbols=ignore-all"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
