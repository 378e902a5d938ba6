"""Host code of the CUDA library, called from small C++ programs linked against
it.  No GPU: what is called here fills tables or refuses its arguments before
any CUDA call."""
import os
import subprocess

import pytest

import __graft_entry__ as entry

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2003_07720_gb300")


def _run(tmp_path, source):
    from paper_2003_07720_gb300 import build
    entry.build()
    cuda = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source)
    lib = os.path.dirname(build.LIB)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", cuda, "-I", build.INCLUDE, "-I", build.CSRC,
                    str(src), "-o", str(exe), build.LIB, f"-Wl,-rpath,{lib}"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


def test_filling_the_transform_tables_allocates_nothing(tmp_path):
    """rpm_apply_gamma_noalloc fills them in a C entry point that promises not to
    allocate and catches nothing; every supported side is filled."""
    _run(tmp_path, r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include "rpm_internal.h"
static long count = 0;
void* operator new(std::size_t n) {
  ++count;
  void* p = std::malloc(n);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
static rpm::PairTables t;
int main() {
  const int xy[] = {4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 256};
  const int z[] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 256};
  count = 0;
  for (int nx : xy)
    for (int ny : xy)
      for (int nz : z) rpm::pair_tables(nx, ny, nz, &t);
  std::printf("%ld allocations\n", count);
  return count == 0 ? 0 : 1;
}
""")


def test_five_passes_refuse_a_misaligned_spectrum(tmp_path):
    """Their kernels access the spectrum in 16-byte elements; the check comes
    before any launch (the pointers here are not memory)."""
    _run(tmp_path, r"""
#include <cstdio>
#include "rpm_internal.h"
int main() {
  const int sides[][2] = {{8, 4}, {256, 256}, {64, 48}, {16, 16}};
  for (auto& s : sides) {
    rpm::GridDev g{};
    g.nx = s[0];
    g.ny = s[1];
    g.nz = 4;
    g.nxh = g.nx / 2;
    g.n = (long long)g.nx * g.ny * g.nz;
    g.plane = g.ny * (g.nxh + 1);
    g.plane_v = 2;
    const cudaError_t e = rpm::launch_apply_gamma(g, (const float*)0x1000, (float*)0x2000,
                                                  (float2*)0x3008, nullptr, rpm::GM_LINEAR, nullptr);
    if (e != cudaErrorInvalidValue) {
      std::printf("%d x %d: %d\n", g.nx, g.ny, (int)e);
      return 1;
    }
  }
  return 0;
}
""")
