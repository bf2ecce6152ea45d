"""The host-side bookkeeping of band launches (csrc/band_host.h, plain C++)
on the CPU: compiled into a small program with fakes for the CUDA side."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1209_0296_gb300", "csrc")
CXX = shutil.which("g++") or shutil.which("c++")


def _run(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "band_host.h"\n#include <cstdio>\n#include <cstdlib>\n#include <set>\n#include <thread>\n'
                   "#define CHECK(x) do { if (!(x)) { std::printf(\"line %d: %s\\n\", __LINE__, #x); std::exit(1); } } while (0)\n"
                   "using namespace lat;\n" + body)
    subprocess.run([CXX, "-std=c++17", "-O1", "-Wall", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


@pytest.mark.skipif(CXX is None, reason="no C++ compiler")
def test_words_are_never_shared(tmp_path):
    _run(tmp_path, r"""
static int pages = 0, queries = 0;
static int *page(size_t n) { ++pages; return new int[n](); }
static bool done(void *e) { ++queries; return *static_cast<bool *>(e); }
static int *none(size_t) { return nullptr; }
int main()
{
    WordPool p(page, done, 8);
    std::set<int *> live;
    for (int i = 0; i < 100; ++i) {       // more owners than a page holds: all words differ
        int *w = p.take();
        CHECK(w != nullptr && *w == 0 && live.insert(w).second);
        *w = 1;
    }
    CHECK(pages == 13);
    bool over = false;
    int *a = *live.begin();
    p.give(a, &over);                     // its launches still run
    for (int i = 0; i < 20; ++i) CHECK(live.insert(p.take()).second);
    CHECK(*a == 1);                       // nobody took it or cleared it
    over = true;
    for (int i = 0; i < 16; ++i) {
        int *w = p.take();
        CHECK(w == a || live.insert(w).second);
        if (w == a) a = nullptr;
    }
    CHECK(a == nullptr);                  // free again
    int *b = p.take();
    *b = 7;
    p.give(b, nullptr);
    CHECK(p.take() == b && *b == 0);
    CHECK(WordPool(none, done, 8).take() == nullptr);
    const int before = pages;             // owners that come and go need no more pages
    for (int i = 0; i < 100000; ++i) {
        static bool yes = true;
        int *w = p.take();
        p.give(w, &yes);
        p.give(p.take(), nullptr);
    }
    CHECK(pages <= before + 1);
    return 0;
}
""")


# function attributes and SM counts belong to a device: found once for each, not once for all
@pytest.mark.skipif(CXX is None, reason="no C++ compiler")
def test_found_once_per_device(tmp_path):
    _run(tmp_path, r"""
#include <atomic>
int main()
{
    PerDevice<int> v;
    std::atomic<int> found[66] = {};
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([&] {
            for (int dev = 0; dev < 64; ++dev)
                for (int rep = 0; rep < 3; ++rep)
                    CHECK(v.get(dev, [&, dev] { ++found[dev]; return 100 + dev; }) == 100 + dev);
        });
    for (auto &x : t) x.join();
    for (int dev = 0; dev < 64; ++dev) CHECK(found[dev] == 1);
    CHECK(v.get(65, [&] { ++found[65]; return 5; }) == 5 && v.get(65, [&] { ++found[65]; return 6; }) == 6);
    CHECK(v.get(-1, [] { return 3; }) == 3);
    return 0;
}
""")
