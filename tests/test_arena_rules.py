"""The bounds that the checked build holds publications, chunks, records and
viewpoints to (vcm_internal.h), compiled for the host: the last place inside each
buffer passes, the first one outside does not, whatever the other fields say.
"""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1310_7297_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = r"""
#include <climits>
#include <cstdio>
#include "vcm_internal.h"
using namespace vcm;
static int bad = 0;
static void expect(bool got, bool want, const char *what) { if (got != want) { printf("%s\n", what); ++bad; } }
#define YES(x) expect(x, true, #x)
#define NO(x) expect(x, false, #x)
int main()
{
    Arena d;   // the default one
    Arena a;   // a small one
    a.chunk_cap = 7; a.rec_cap = 3; a.pool_ints = 100;
    for (const Arena &r : {a, d}) {
        const int C = r.chunk_cap, K = r.rec_cap, P = r.pool_ints;
        YES(publication_in_bounds(r, 0, 0, 1, 0, P));
        YES(publication_in_bounds(r, K - 1, C - 1, 1, P - 1, 1));
        YES(publication_in_bounds(r, 0, 0, C, P, 0));
        NO(publication_in_bounds(r, K, 0, 1, 0, 1));
        NO(publication_in_bounds(r, -1, 0, 1, 0, 1));
        NO(publication_in_bounds(r, 0, C, 1, 0, 1));
        NO(publication_in_bounds(r, 0, 1, C, 0, 1));
        NO(publication_in_bounds(r, 0, -1, 1, 0, 1));
        NO(publication_in_bounds(r, 0, INT_MAX, 1, 0, 1));
        NO(publication_in_bounds(r, 0, 0, 1, P, 1));
        NO(publication_in_bounds(r, 0, 0, 1, 1, P));
        NO(publication_in_bounds(r, 0, 0, 1, INT_MAX, 1));
        NO(publication_in_bounds(r, 0, 0, 1, 0, INT_MAX));
        NO(publication_in_bounds(r, 0, 0, 1, -1, 1));
        YES(chunk_in_bounds(r, (K - 1) * 32 + kChunkVp));
        YES(chunk_in_bounds(r, 0));
        NO(chunk_in_bounds(r, (K - 1) * 32 + kChunkVp + 1));
        NO(chunk_in_bounds(r, K * 32 + 1));
        NO(chunk_in_bounds(r, -1));
        NO(chunk_in_bounds(r, INT_MIN));
        DevRequest reqs[2] = {};
        reqs[0].nl = 4; reqs[1].nl = 1;
        const int n_boxes = 50;
        auto rec = [&](int req, int count, int off, int layer) {
            const int x[kRecInts] = {req, count, off, layer};
            return record_in_bounds(r, x, reqs, 2, n_boxes);
        };
        YES(rec(0, 50, P - 50, 3));
        YES(rec(1, 0, P, 0));
        NO(rec(2, 1, 0, 0));
        NO(rec(-1, 1, 0, 0));
        NO(rec(0, 51, 0, 0));
        NO(rec(0, -1, 0, 0));
        NO(rec(0, 50, P - 49, 0));
        NO(rec(0, 1, -1, 0));
        NO(rec(0, 1, INT_MAX, 0));
        NO(rec(0, 1, 0, 4));
        NO(rec(1, 1, 0, 1));
        NO(rec(0, 1, 0, -1));
    }
    DevRequest R = {};
    R.nx = 5; R.ny = 9;
    YES(viewpoint_in_bounds(R, 4, 8));
    YES(viewpoint_in_bounds(R, 0, 0));
    NO(viewpoint_in_bounds(R, 5, 0));
    NO(viewpoint_in_bounds(R, 0, 9));
    NO(viewpoint_in_bounds(R, -1, 0));
    NO(viewpoint_in_bounds(R, 0, -1));
    return bad != 0;
}
"""


def test_rules_at_the_ends_of_the_buffers(tmp_path):
    cxx = shutil.which("g++")
    if not cxx or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "rules.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "rules")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, "-I", os.path.join(CUDA, "include"), str(src), "-o", exe], check=True)
    run = subprocess.run([exe], stdout=subprocess.PIPE, text=True)
    assert run.returncode == 0, run.stdout
