"""The tensor-map encoder is looked up until it is found, then kept (csrc/lbm_pool.h, compiled for the host
with a fake lookup that fails at first): a context made after a failed lookup tries again."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "lbm_pool.h"
using namespace gb300lbm;
typedef int (*Fn)(int);
static int calls = 0;
static int found(int x) { return x + 1; }
static Fn look() { return ++calls < 3 ? nullptr : found; }
int main() {
    static std::atomic<Fn> kept{nullptr};
    if (kept_lookup(kept, look) || kept_lookup(kept, look)) return 1;            // fails, and is tried again
    for (int k = 0; k < 4; ++k) if (kept_lookup(kept, look) != found) return 2;
    return calls == 3 ? 0 : 3;                                                      // kept once found
}
"""


def test_a_failed_lookup_is_made_again(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    src, exe = tmp_path / "look.cpp", tmp_path / "look"
    src.write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2201_06039_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", csrc, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
    # the library's own lookup goes through it
    with open(os.path.join(csrc, "lbm_capi.cu")) as fh:
        text = fh.read()
    body = text[text.index("EncodeTiledFn tensor_map_encoder()"):]
    assert "kept_lookup(kept" in body[:body.index("\n}\n")]
