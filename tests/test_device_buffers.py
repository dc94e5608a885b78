"""Device buffers hold what the kernels' 16-byte accesses need, checked on the host: the library's buffer type
compiled against an allocator that hands out exact pieces at any offset and records them.  Whatever sizes a reused
buffer sees, it starts on a 16-byte boundary, 16 bytes of its allocation follow the size last asked for, and the
allocator gets back the pointer and size it gave."""
import subprocess

from paper_2012_13618_gb300 import _build

_SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "internal.h"

static size_t g_offset = 0;
static std::map<char *, size_t> g_live;
static int g_errors = 0;

namespace bp {
void *dev_alloc(size_t bytes, cudaStream_t, AllocTag *) {
    static char *next = reinterpret_cast<char *>(size_t(1) << 40);  // never touched
    char *p = next + g_offset;
    next += (bytes / 4096 + 2) * 4096;
    g_live[p] = bytes;
    return p;
}
void dev_free(void *p, size_t bytes, cudaStream_t, const AllocTag &) {
    auto it = g_live.find(static_cast<char *>(p));
    if (it == g_live.end() || it->second != bytes) ++g_errors;
    else g_live.erase(it);
}
void zero_fill(void *, size_t, cudaStream_t) {}
void note_realloc() {}
}  // namespace bp

static void check(const bp::Buf &b, size_t bytes, const char *what) {
    const char *p = b.as<char>();
    for (auto &a : g_live)
        if (p >= a.first && p < a.first + a.second) {
            const bool aligned = (reinterpret_cast<size_t>(p) & 15) == 0;
            const bool slack = p + bytes + 16 <= a.first + a.second;
            if (!aligned || !slack) {
                if (g_errors++ < 5) std::printf("%s: offset %zu, %zu bytes, aligned %d, slack %d\n", what, g_offset, bytes, aligned, slack);
            }
            return;
        }
    ++g_errors;
    std::printf("%s: not in an allocation\n", what);
}

int main() {
    for (g_offset = 0; g_offset < 16; ++g_offset) {
        {
            // node weights of two requests on one workspace: 4 * 45,065 bytes are what the first call left room for
            bp::Buf nw;
            nw.ensure(4 * 40001, nullptr);
            check(nw, 4 * 40001, "weights");
            nw.ensure(4 * 45065, nullptr);
            check(nw, 4 * 45065, "weights again");
        }
        for (size_t first : {1, 7, 16, 100, 4097, 100000}) {
            bp::Buf b;
            for (size_t n = first; n < first + first / 4 + 600; ++n) {
                b.ensure(n, nullptr);
                check(b, n, "growing");
            }
        }
        {
            bp::Buf z;
            z.ensure_zero(100, nullptr);
            check(z, 100, "zeroed");
        }
    }
    if (!g_live.empty()) ++g_errors;
    std::printf("errors %d\n", g_errors);
    return g_errors != 0;
}
"""


def test_buffers_are_aligned_with_slack(tmp_path):
    src = tmp_path / "buffers.cu"
    src.write_text(_SRC)
    exe = tmp_path / "buffers"
    r = subprocess.run([_build.nvcc(), *_build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", _build.INCLUDE,
                        "-I", _build.CSRC, "-o", str(exe), str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
