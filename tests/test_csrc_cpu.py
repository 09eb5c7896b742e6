"""Checks of the native sources that need no GPU: rules that every file of csrc/ keeps, and host-side helpers compiled
with the system compiler and run here."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_09772_gb300", "csrc")


def _code():
    """file name -> source without comments"""
    out = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*"))):
        if f.endswith((".cu", ".cuh", ".h")):
            s = re.sub(r"/\*.*?\*/", "", open(f).read(), flags=re.S)
            out[os.path.basename(f)] = re.sub(r"//[^\n]*", "", s)
    return out


def test_every_copy_names_its_stream():
    """A copy or a fill without a stream runs on the legacy stream, which a caller's non-blocking stream does not wait
    for, and one from pageable memory may return before its transfer has ended: a kernel could read a table that is not
    there yet."""
    bad = [f"{name}: {m.group(0)}" for name, s in _code().items()
           for m in re.finditer(r"\bcudaMem(cpy|cpy2D|cpy3D|cpyToSymbol|cpyFromSymbol|set|set2D)\s*\(", s)]
    assert not bad, bad


GROW = r"""
#include <assert.h>
#include <stdlib.h>
#include <vector>
#include "rism_grow.h"
static long budget;  // bytes the allocator still gives
static int allocs, live;
struct Host {
    static int alloc(void** p, size_t n) {
        ++allocs;
        if ((long)n > budget) return 2;
        budget -= (long)n, ++live;
        *p = malloc(n);
        return 0;
    }
    static void release(void* p) { if (p) --live; free(p); }
};
using namespace rism;
int main() {
    double* a = nullptr;
    int* b = nullptr;
    int64_t cap = 0;
    budget = 10000;
    assert(grow_with<Host>(cap, 100, buf(a, 100), buf(b, 200)) == 0 && cap == 100 && a && b && live == 2);
    a[99] = 1.0, b[199] = 1;
    // a smaller or equal need keeps the buffers
    allocs = 0;
    double* a0 = a;
    assert(grow_with<Host>(cap, 7, buf(a, 7), buf(b, 14)) == 0 && grow_with<Host>(cap, 100, buf(a, 100), buf(b, 200)) == 0);
    assert(allocs == 0 && a == a0 && cap == 100);
    // the first, then the second allocation of the group fails: the capacity is gone with the pointers
    for (int second = 0; second < 2; ++second) {
        budget = second ? 8 * 1000 : 100;
        assert(grow_with<Host>(cap, 1000, buf(a, 1000), buf(b, 2000)) == 2 && cap == 0 && !b);
        assert(!a == !second);
        // ... so a smaller need than the one the group held before allocates again
        budget = 10000;
        allocs = 0;
        assert(grow_with<Host>(cap, 50, buf(a, 50), buf(b, 100)) == 0 && cap == 50 && allocs == 2 && a && b && live == 2);
        a[49] = 1.0, b[99] = 1;
    }
    // an int capacity, and a need of nothing still gives a buffer
    char* c = nullptr;
    int icap = 0;
    assert(grow_with<Host>(icap, 0, buf(c, 0)) == 0 && icap == 1 && c);
    c[0] = 1;
    Host::release(a), Host::release(b), Host::release(c);
    assert(live == 0);
    return 0;
}
"""


def test_a_failed_allocation_leaves_no_capacity(tmp_path):
    src, exe = tmp_path / "grow.cpp", tmp_path / "grow"
    src.write_text(GROW)
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-I", CSRC, str(src), "-o", str(exe)])
    subprocess.check_call([str(exe)])


def test_every_buffer_goes_through_the_grow_helper():
    """A capacity kept across a failed allocation lets the next, smaller call launch kernels on null pointers: only the
    helper allocates (rism_internal.cuh holds its two allocators)."""
    for name, s in _code().items():
        n = len(re.findall(r"\bcudaMalloc(Host|Async|Managed)?\s*\(", s))
        assert n == (2 if name == "rism_internal.cuh" else 0), (name, n)


def test_every_capacity_is_kept_beside_its_buffer():
    """A buffer that serves one call after another only grows: its capacity is a member of the object that owns it, so a
    smaller (or a repeated) need neither frees nor allocates."""
    for name, s in _code().items():
        for m in re.finditer(r"\bgrow(?:_with<\w+>)?\(\s*([^,;]+),[^;]*?\bbuf\(", s):
            if name not in ("rism_grow.h", "rism_internal.cuh"):
                assert re.match(r"(c|s)->\w+|A\.\w+", m.group(1)), f"{name}: {m.group(0)}"


ORDER = r"""
#include <stdio.h>
#include <stdlib.h>
#include "rism_order.h"
int main() {
    // extents along x, y, z and the number of atoms: a globule, a plane, lines short and long, one atom, two far apart
    const double ext[][4] = {{40, 40, 40, 5000}, {300, 300, 0, 3000}, {1e4, 0, 0, 700}, {1e9, 0, 0, 64}, {1e13, 1e-3, 0, 700},
                             {0, 1e200, 0, 33}, {1e308, 1e308, 0, 40}, {0, 0, 0, 1}, {0, 0, 0, 90}, {0, 0, 1e12, 2}};
    for (const auto& e : ext) {
        const int n = (int)e[3];
        std::vector<double> raw(6 * (size_t)n, 0.0);
        srand(7);
        for (int i = 0; i < n; ++i)
            for (int d = 0; d < 3; ++d)
                raw[6 * (size_t)i + d] = e[d] * (i == 0 ? -0.5 : i == n - 1 ? 0.5 : rand() / (RAND_MAX + 1.0) - 0.5);
        std::vector<int> perm((size_t)n, -1), seen((size_t)n, 0);
        rism::lra_order(raw.data(), n, perm.data());
        for (int p : perm) {
            if (p < 0 || p >= n || seen[(size_t)p]++) return printf("extents %g %g %g\n", e[0], e[1], e[2]), 1;
        }
    }
    return 0;
}
"""


def test_spatial_order_of_any_solute(tmp_path):
    """The order of the all-space pair sum is a permutation for solutes of any shape, also where a cell index computed in
    floating point exceeds the integers (a line of atoms 1e13 A long)."""
    src, exe = tmp_path / "order.cpp", tmp_path / "order"
    src.write_text(ORDER)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-D_GLIBCXX_ASSERTIONS", "-I", CSRC, str(src), "-o", str(exe)])
    subprocess.check_call([str(exe)])


def test_no_sm_count_in_the_code():
    """Grids and dispatch rules take the number of SMs from the device."""
    for name, s in _code().items():
        assert not re.search(r"\b(152|1824)\b", s), name
