"""The schedule of the prompt GEMMs (csrc/tc_gemm.cuh: tc_plan, tc_work_next),
on the CPU: its host functions are compiled with nvcc into a small program
that plans random shapes and walks every CTA pair's work.

Checked for each shape: the token tiles cover the rows; every (tile, k block)
is computed exactly once; a segment that starts inside a tile is its pair's
first one (a pair has one workspace slot); and the pair that finalises a tile
counts exactly the pairs that left partial sums of it, which are the next ones
in number (their blocks come before its own, so in the usual order of dispatch it
never waits for a pair that cannot run).
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "tc_gemm.cuh"
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>
using namespace ssd::tc;
static int bad(const char* what, const TcArgs& a, int n_ft) {
    printf("%s: rows %d n_ft %d n_kb %d nt %d tiles %d split %d / %d pairs %d\n", what, a.rows, n_ft, a.n_kb, a.nt,
           a.sched.n_tiles, a.sched.n_split, a.sched.split_pairs, a.sched.pairs);
    return 1;
}
int main(int argc, char** argv) {
    srand(atoi(argv[1]));
    for (int it = 0; it < atoi(argv[2]); ++it) {
        TcArgs a{};
        a.rows = rand() % 3 ? 17 + rand() % 2032 : 17 + rand() % 300;
        const int n_ft = 1 + rand() % (rand() % 4 ? 64 : 450), P = rand() % 5 ? 76 : 1 + rand() % 80;
        const int K = 16 * (4 + rand() % (rand() % 2 ? 80 : 1800));
        a.n_kb = (K + kBK - 1) / kBK;
        tc_plan(a, n_ft, P, K);
        const TcSched& s = a.sched;
        if (a.nt % 32 || a.nt < 32 || a.nt > kMaxTok || s.n_tt * a.nt < a.rows || (s.n_tt - 1) * a.nt >= a.rows)
            return bad("token tiles", a, n_ft);
        if (a.stages < 4 || a.stages > kMaxStages || a.stages * (kATile + a.nt * 128) > kRingBytes)
            return bad("ring", a, n_ft);
        if (s.n_tiles != n_ft * s.n_tt || s.pairs < 1 || s.pairs > P || s.split_pairs > P) return bad("grid", a, n_ft);
        if ((long)s.n_tiles * a.n_kb > 200000) continue;
        std::vector<char> seen((size_t)s.n_tiles * a.n_kb, 0);
        std::vector<int> partial_of(s.pairs, -1), fin(s.n_tiles, -1), contrib(s.n_tiles, 0);
        for (int p = 0; p < s.pairs; ++p) {
            TcWork w;
            tc_work_init(w, s, a.n_kb, p);
            for (bool first = true; tc_work_next(w, s, a.n_kb, p); first = false) {
                if (w.tile < 0 || w.tile >= s.n_tiles || w.kb0 >= w.kb1 || w.kb1 > a.n_kb) return bad("segment", a, n_ft);
                for (int k = w.kb0; k < w.kb1; ++k)
                    if (seen[(size_t)w.tile * a.n_kb + k]++) return bad("twice", a, n_ft);
                if (w.partial) {
                    if (!first) return bad("second partial of a pair", a, n_ft);
                    partial_of[p] = w.tile;
                } else {
                    if (fin[w.tile] >= 0) return bad("two finalisers", a, n_ft);
                    fin[w.tile] = p;
                    contrib[w.tile] = w.contributors;
                }
            }
        }
        for (char c : seen)
            if (!c) return bad("missing", a, n_ft);
        for (int t = 0; t < s.n_tiles; ++t) {
            int n = 0;
            for (int p = 0; p < s.pairs; ++p) n += partial_of[p] == t;
            if (fin[t] < 0 || n != contrib[t]) return bad("contributors", a, n_ft);
            for (int c = 1; c <= n; ++c)
                if (partial_of[fin[t] + c] != t) return bad("order", a, n_ft);
        }
    }
    printf("ok\n");
    return 0;
}
"""


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    d = tmp_path_factory.mktemp("sched")
    src, exe = d / "check.cu", d / "check"
    src.write_text(SOURCE)
    subprocess.check_call(["nvcc", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "paper_2309_08168_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)])
    return str(exe)


@pytest.mark.parametrize("seed", [1, 2])
def test_every_block_once(checker, seed):
    r = subprocess.run([checker, str(seed), "8000"], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
