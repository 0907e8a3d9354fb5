"""Allocation of needed memory with a work space that a problem can do without (csrc/pfc_alloc.h),
compiled for the host with an allocator that fails above a limit."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_04856_gb300", "csrc")
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "pfc_alloc.h"
static size_t g_limit = 0;
static int g_calls = 0;
static void* take(size_t n) { ++g_calls; return n <= g_limit ? std::malloc(n) : nullptr; }
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main()
{
    void *p, *w;
    g_limit = 10000;
    CHECK(pfc::alloc_with_work(take, 1000, 5000, &p, &w) && g_calls == 1);
    CHECK((char*)w - (char*)p == 1024);
    CHECK(pfc::alloc_with_work(take, 1000, 0, &p, &w) && p && !w);
    g_calls = 0;
    g_limit = 1000;                       // the work space is not to be had
    CHECK(pfc::alloc_with_work(take, 1000, 5000, &p, &w) && p && !w && g_calls == 2);
    g_limit = 999;
    CHECK(!pfc::alloc_with_work(take, 1000, 5000, &p, &w) && !p && !w);
    CHECK(!pfc::alloc_with_work(take, 1000, 0, &p, &w) && !p && !w);
    return 0;
}
"""


def test_work_space_is_optional(tmp_path):
    src, exe = tmp_path / "alloc.cpp", tmp_path / "alloc"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
