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


def test_the_harmonic_sums_cut_their_work_for_the_device(tmp_path):
    """Columns per unit and rows per CTA follow the number of SMs: the widest unit that leaves 9 per SM (512 columns at
    least), and the same rows for k times the blocks on k times the SMs. 152 SMs keep the widths that were measured."""
    out = run_cpp(tmp_path, r'''
#include "hs_rules.h"
#include <cstdio>
using namespace fdas;
int main() {
    for (int sms : {38, 76, 152, 304})
        for (int rows : {1, 4, 21, 42, 127})
            for (long long total : {1ll, 2050ll, 9125ll, 32769ll, 65536ll, 262144ll, 1048577ll, 16777216ll})
                for (bool hp1 : {false, true}) {
                    const int cols = hs_columns(rows, total, hp1, sms), most = hp1 ? 4096 : 8192;
                    auto units = [&](int c) { return (2 * rows + 1) * ((total + c - 1) / c); };
                    if (cols < 512 || cols > most || (cols & (cols - 1))) return 1;
                    if (cols > 512 && units(cols) < 9ll * sms) return 2;
                    if (cols < most && units(2 * cols) >= 9ll * sms) return 3;
                }
    for (int blocks : {1, 5, 18, 79, 313, 1093, 1249})
        for (int n_temp : {3, 9, 43, 85, 255}) {
            const int r = rows_per_cta(blocks, n_temp, 152);
            if (r < 1 || r > kMaxRows || r > n_temp) return 4;
            if (rows_per_cta(2 * blocks, n_temp, 304) != r || rows_per_cta(4 * blocks, n_temp, 608) != r) return 5;
        }
    for (long long n : {4099, 18248, 65536, 200003, 2097152})
        std::printf("%d %d ", hs_columns(42, n, false, 152), hs_columns(21, (n - 1) / 2 + 1, true, 152));
}
''')
    assert out.split() == "512 512 1024 512 2048 1024 8192 2048 8192 4096".split()
