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


def test_the_convolution_work_is_dealt_out_once_and_evenly(tmp_path):
    """Every template of every segment falls to exactly one worker, in every form, length and launch shape; and
    where not every worker group of the tensor-core form has work, no SM gets a second group before each has one
    (its rule for short spectra prices a group alone on its SM)."""
    out = run_cpp(tmp_path, r'''
#include "deal.cuh"
#include <cstdio>
#include <vector>
using namespace fdas;
int main() {
    long checked = 0, spread = 0;
    for (int precision : {FDAS_FP32, FDAS_BF16X3})
        for (int n_temp : {3, 9, 43, 85, 127, 255})
            for (int n_seg : {1, 2, 3, 6, 9, 10, 12, 13, 16, 33, 41, 76, 123, 151, 152, 153, 400, 457, 1289})
                for (int tpi : {0, 1, 2, 17, 43, 44, 85, 1000}) {
                    const int sms = 152, groups = precision == FDAS_FP32 ? 1 : 3;
                    const Geometry g{n_temp, (n_temp - 1) / 2, 421, 210, 2048, 1628, precision};
                    int workers = 0;
                    const Deal d = make_deal(g, n_seg, tpi, sms, 3, &workers);
                    const int grid = groups == 1 || workers < sms ? workers : sms;
                    std::vector<int> seen((size_t)n_seg * n_temp, 0);
                    int most = 0, with_work = 0;
                    for (int b = 0; b < grid; ++b) {
                        int busy = 0;
                        for (int k = 0; k < groups; ++k) {
                            bool any = false;
                            for (int q = -1, t0, t1 = 0;
                                 deal_next(d, groups == 1 ? b : worker(d, b, grid, k, groups), grid * groups, q, t0, t1);) {
                                any = true;
                                if (q < 0 || q >= n_seg || t0 < 0 || t0 >= t1 || t1 > n_temp) return 1;
                                for (int t = t0; t < t1; ++t) ++seen[(size_t)q * n_temp + t];
                            }
                            busy += any;
                        }
                        with_work += busy;
                        most = busy > most ? busy : most;
                    }
                    for (int c : seen)
                        if (c != 1) return 2;
                    if (with_work > workers) return 3;
                    if (groups > 1 && workers <= grid * groups) {
                        ++spread;
                        if (most > (workers + grid - 1) / grid) return 4;
                    }
                    ++checked;
                }
    std::printf("%ld %d\n", checked, spread > 200);
}
''')
    assert out.split() == [str(2 * 6 * 19 * 8), "1"]
