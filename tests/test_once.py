"""The per-device once flag (csrc/pfc_once.h), compiled for the host: set on each device, again where it
failed, every time on a device past its table, and by several threads."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_04856_gb300", "csrc")
SOURCE = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "pfc_once.h"
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main()
{
    static pfc::OncePerDevice once;
    int calls = 0;
    auto ok = [&] { ++calls; return 0; };
    CHECK(once(0, ok) == 0 && calls == 1 && once(0, ok) == 0 && calls == 1);
    CHECK(once(1, ok) == 0 && calls == 2);               // another device has its own setting
    CHECK(once(2, [] { return 7; }) == 7);               // failed: tried again
    CHECK(once(2, ok) == 0 && calls == 3 && once(2, ok) == 0 && calls == 3);
    CHECK(once(64, ok) == 0 && once(64, ok) == 0 && once(-1, ok) == 0 && calls == 6);
    static pfc::OncePerDevice many;
    std::atomic<int> set[8] = {};
    std::vector<std::thread> t;
    for (int j = 0; j < 8; ++j)
        t.emplace_back([&] { for (int d = 0; d < 8; ++d) many(d, [&] { ++set[d]; return 0; }); });
    for (auto& x : t) x.join();
    for (auto& s : set) CHECK(s >= 1 && s <= 8);
    return 0;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_launchers_opt_in_per_device():
    """No launcher keeps the shared-memory opt-in in a flag of the whole process."""
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        assert not re.search(r"static\s+bool\s+\w+\s*=", text), name
