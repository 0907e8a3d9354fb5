"""The pool that hands out words of one page (csrc/pfc_words.h), compiled for the host with a page of
ordinary memory: distinct words, a bound, words given back are reused, a page that something else
freed is replaced and its words are not given back to the new one, and several threads at once."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_04856_gb300", "csrc")
SOURCE = r"""
#include <set>
#include <thread>
#include <vector>
#include <cstdio>
#include "pfc_words.h"
static bool g_alive = true, g_fail = false;
static int g_made = 0;
struct Page {
    static double* make() { if (g_fail) return nullptr; ++g_made; g_alive = true; return new double[128]; }
    static bool alive(double*) { return g_alive; }
};
using Pool = pfc::WordPool<Page, 128>;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main()
{
    Pool p;
    g_fail = true;
    CHECK(!p.take().p);
    g_fail = false;
    std::vector<Pool::Word> w;
    std::set<double*> seen;
    for (int k = 0; k < 128; ++k) { w.push_back(p.take()); CHECK(w.back().p && seen.insert(w.back().p).second); }
    CHECK(g_made == 1 && !p.take().p);
    p.give(Pool::Word{});
    p.give(w[70]);
    Pool::Word again = p.take();
    CHECK(again.p == w[70].p && !p.take().p);
    g_alive = false;                                     // the page is gone
    Pool::Word fresh = p.take();
    CHECK(g_made == 2 && fresh.p);
    for (auto& x : w) p.give(x);                         // words of the old page
    std::set<double*> now{ fresh.p };
    for (int k = 1; k < 128; ++k) { Pool::Word x = p.take(); CHECK(x.p && now.insert(x.p).second); }
    CHECK(!p.take().p);
    Pool q;
    std::vector<std::thread> t;
    bool bad[4] = {};
    for (int j = 0; j < 4; ++j)
        t.emplace_back([&q, &bad, j] {
            for (int k = 0; k < 20000; ++k) {
                Pool::Word a = q.take(), b = q.take();
                *a.p = j; *b.p = j + 0.5;
                if (a.p == b.p || *a.p != j || *b.p != j + 0.5) bad[j] = true;
                q.give(a); q.give(b);
            }
        });
    for (auto& x : t) x.join();
    for (bool b : bad) CHECK(!b);
    return 0;
}
"""


def test_word_pool(tmp_path):
    src, exe = tmp_path / "words.cpp", tmp_path / "words"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
