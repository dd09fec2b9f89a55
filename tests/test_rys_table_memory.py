"""The node table's build when memory runs out: an exception for the caller, also from its threads, and a second call
that works."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_01834_gb300", "csrc")
MAIN = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include "mdx_internal.h"
static std::atomic<long> left{-1};
void* operator new(std::size_t n) {
  if (left.load() >= 0 && left.fetch_sub(1) == 0) throw std::bad_alloc();
  if (void* p = std::malloc(n)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
int main(int, char** argv) {
  left = std::atol(argv[1]);
  try {
    mdx::rys_table();
    std::puts("built");
  } catch (const std::bad_alloc&) {
    std::puts("bad_alloc");
  }
  left = -1;
  std::printf("%d\n", (int)(mdx::rys_table().size() == (size_t)mdx::rys_offset(mdx::kRysMax + 1)));
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("rys_memory")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "main")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(d / "main.cpp"), os.path.join(CSRC, "rys_table.cpp"),
                    "-o", exe, "-lpthread"], check=True)
    return exe


@pytest.mark.parametrize("nth,first", [(0, "bad_alloc"), (500, "bad_alloc"), (20000, "bad_alloc"), (10 ** 9, "built")])
def test_allocation_failure_is_an_exception(program, nth, first):
    r = subprocess.run([program, str(nth)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == [first, "1"]
