"""Growth of a workspace's reduced-system buffers (host logic, CPU only).

The header is compiled with the host compiler and driven with an allocator that can
be told to fail: after a failure the workspace holds no buffer at all, its capacity
is zero and its generation has moved on, so that neither a capacity check nor a
captured launch sequence can reach the freed memory, and the next growth starts
afresh.
"""
import ctypes as C
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2312_02999_gb300", "csrc")

_SRC = r'''
#include <cstdlib>
#include <set>
#include "workspace.h"
using namespace fsim;
struct Work {
  double* Bc = nullptr; int* bocc = nullptr; double* red = nullptr; float* redf = nullptr;
  long red_cap = 0; int nc_cap = 0, red_gen = 0;
};
static Work w;
static std::set<void*> live;
static size_t last_bytes = 0;
static int gen_at_release = -1;
extern "C" int fits(int nc) { return reduced_fits(w, nc); }
extern "C" int grow(int nc, int n2, long elems, int fail) {
  const int cap = grown_reduced_cap(nc, w.nc_cap, n2);
  const int gen = w.red_gen;
  return grow_reduced(w, cap, elems,
      [&](size_t b) -> void* {
        last_bytes = b;
        if (fail) return nullptr;
        void* p = std::malloc(b); live.insert(p); return p;
      },
      [&](void* p) { gen_at_release = w.red_gen - gen; live.erase(p); std::free(p); });
}
extern "C" void state(long* out) {
  out[0] = w.Bc != nullptr; out[1] = w.bocc != nullptr; out[2] = w.red != nullptr;
  out[3] = w.redf != nullptr; out[4] = w.nc_cap; out[5] = w.red_cap; out[6] = w.red_gen;
  out[7] = (long)live.size(); out[8] = gen_at_release;
}
// the buffers end inside the block and do not overlap
extern "C" int laid_out() {
  const size_t c = w.nc_cap, e = w.red_cap;
  const char* b = (const char*)w.Bc;
  return (const char*)(w.Bc + 9 * c * c) <= (const char*)w.bocc &&
         (const char*)(w.bocc + 2 * c * c + c + 32) <= (const char*)w.red &&
         (const char*)(w.red + e) <= (const char*)w.redf &&
         (const char*)(w.redf + e) <= b + last_bytes && live.count((void*)b);
}
'''


@pytest.fixture()
def lib(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, so = tmp_path / "w.cpp", tmp_path / "w.so"
    src.write_text(_SRC)
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)],
                   check=True)
    L = C.CDLL(str(so))
    L.grow.argtypes = [C.c_int, C.c_int, C.c_long, C.c_int]

    def state():
        out = (C.c_long * 9)()
        L.state(out)
        return list(out)
    L.now = state
    return L


def test_failed_growth_leaves_nothing_behind(lib):
    assert lib.grow(20, 1000, 5001, 0) and lib.laid_out()
    *have, cap, elems, gen, live, _ = lib.now()
    assert have == [1, 1, 1, 1] and (cap, elems, live) == (20, 5001, 1)
    assert lib.fits(20) and not lib.fits(21)
    # the larger block is refused
    assert not lib.grow(70, 1000, 60000, 1)
    *have, cap, elems, gen2, live, before = lib.now()
    assert have == [0, 0, 0, 0] and (cap, elems, live) == (0, 0, 0)
    assert gen2 > gen and before == 1        # moved on before the old block went
    assert not any(lib.fits(nc) for nc in (1, 16, 20, 70))
    # and the next frame starts from nothing
    assert lib.grow(3, 1000, 900, 0) and lib.laid_out()
    *have, cap, _, gen3, live, _ = lib.now()
    assert have == [1, 1, 1, 1] and (cap, live) == (16, 1) and gen3 > gen2


@pytest.mark.parametrize("nc,n2,cap", [(1, 1000, 16), (1, 4, 4), (17, 1000, 24), (40, 1000, 40),
                                       (20, 23, 23)])
def test_growth_steps(lib, nc, n2, cap):
    assert lib.grow(min(16, n2), n2, 777, 0)      # 16 (or n2) first
    if nc > min(16, n2):
        assert lib.grow(nc, n2, 1234, 0)
    assert lib.now()[4] == cap and lib.laid_out() and lib.now()[7] == 1
