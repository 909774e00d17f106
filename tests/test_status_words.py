"""The process-wide page of status words (csrc/lbm_pool.h), compiled for the host with a counting fake of
the allocation: words are distinct and come back, the page is one page however many contexts come and go,
a failed allocation is tried again, running out gives nothing, several threads may take and give."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <stdio.h>
#include <stdlib.h>
#include <set>
#include <thread>
#include <vector>
#include "lbm_pool.h"
using namespace gb300lbm;
static int calls = 0, failing = 2;
static int* fake(size_t bytes) { ++calls; return failing-- > 0 ? nullptr : (int*)calloc(1, bytes); }
#define OK(x) if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; }
int main() {
    static StatusWords w(fake);
    OK(w.take() == nullptr && w.take() == nullptr);   // allocation fails twice
    std::set<int*> held;
    for (int k = 0; k < StatusWords::kWords; ++k) { int* p = w.take(); OK(p && held.insert(p).second); }
    OK(w.take() == nullptr && calls == 3);
    int* lo = *held.begin();
    OK(*held.rbegin() - lo == StatusWords::kWords - 1);
    w.give(nullptr);
    w.give(lo + 7);
    OK(w.take() == lo + 7 && w.take() == nullptr);
    for (int* p : held) w.give(p);
    std::vector<std::thread> ts;
    bool bad = false;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&, t] {
            for (int r = 0; r < 2000; ++r) {
                int* p = w.take();
                if (!p) { bad = true; return; }
                *p = t + 1;
                std::this_thread::yield();
                if (*p != t + 1) bad = true;
                w.give(p);
            }
        });
    for (auto& t : ts) t.join();
    OK(!bad && calls == 3);
    return 0;
}
"""


def test_status_words(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    src, exe = tmp_path / "words.cpp", tmp_path / "words"
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_2201_06039_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
