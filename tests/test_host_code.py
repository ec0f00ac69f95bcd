"""Host code of the library, compiled with the host compiler alone and run on the CPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INCLUDE = os.environ.get("CUDA_HOME", "/usr/local/cuda") + "/include"


def run_cpp(tmp_path, source):
    """Compiles a main() against csrc/ and returns its standard output."""
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(source)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1806_01556_gb300", "csrc"), "-I",
                    CUDA_INCLUDE, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout


def test_status_words_are_kept_per_context(tmp_path):
    """A thread that drives two GPUs in turn keeps one pair of words for each: nothing is allocated twice or lost.
    A context that a reset destroyed keeps its entry unfreed, the table ends, and a failed allocation is not kept."""
    out = run_cpp(tmp_path, r'''
#include "status_words.h"
#include <cstdio>
#include <set>
static int made, failing;
static std::set<unsigned long long> dead;
static std::set<unsigned *> live;
struct Fake {
    static unsigned *allocate() {
        if (failing) return nullptr;
        ++made;
        return *live.insert(new unsigned[2]).first;
    }
    static void release(int, unsigned long long ctx, unsigned *w) {
        if (!dead.count(ctx)) live.erase(w);
    }
};
int main() {
    {
        fdas::StatusWords<Fake> t;
        failing = 1;
        bool ok = t.get(0, 11) == nullptr;
        failing = 0;
        unsigned *a = t.get(0, 11), *b = t.get(1, 12);
        ok = ok && a && b && a != b;
        for (int k = 0; k < 1000; ++k) ok = ok && t.get(0, 11) == a && t.get(1, 12) == b;
        std::printf("%d %d ", ok, made);
        dead.insert(12);  // device 1 is reset: its next context has another id
        unsigned *c = t.get(1, 13);
        std::printf("%d %d ", c && c != a && c != b, made);
        for (unsigned long long ctx = 20; ctx < 40; ++ctx) t.get(0, ctx);
        std::printf("%d %d ", made, t.get(0, 99) == nullptr && t.get(0, 11) == a);
    }
    std::printf("%d\n", (int)live.size());
}
''')
    assert out.split() == ["1", "2", "1", "3", "8", "1", "1"]
