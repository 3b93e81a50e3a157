"""The order of the Ritz values is a permutation whatever the values are: the
rank of every column is taken once.  The kernel that gathers the Ritz vectors
reads the columns that this order names, so a rank that nothing writes would
be an index out of whatever the scratch memory held."""

import itertools
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "ritz.h"
// pairs of sums (x^T C x, x^T x) in, the rank of every column out
int main(int n, char** a) {
    const int l = (n - 1) / 2;
    float d[64];
    for (int j = 0; j < l; ++j) d[j] = moara::ritz_value(strtof(a[1 + 2 * j], nullptr), strtof(a[2 + 2 * j], nullptr));
    for (int j = 0; j < l; ++j) {
        int rank = 0;
        for (int i = 0; i < l; ++i) rank += moara::ritz_before(d[i], i, d[j], j);
        printf("%d ", rank);
    }
}
"""


@pytest.fixture(scope="module")
def ranks(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    tmp = tmp_path_factory.mktemp("ritz")
    (tmp / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-I", inc, "-I", os.path.join(ROOT, "paper_2609_15037_gb300", "csrc"),
                    str(tmp / "t.cpp"), "-o", str(tmp / "t")], check=True)

    def run(pairs):
        args = [str(x) for p in pairs for x in p]
        return [int(x) for x in subprocess.run([str(tmp / "t")] + args, capture_output=True, text=True, check=True).stdout.split()]
    return run


def test_descending_with_ties(ranks):
    assert ranks([(2, 1), (3, 1), (2, 1), (0, 0), (-1, 1)]) == [1, 0, 2, 3, 4]


@pytest.mark.parametrize("col", list(itertools.product([("nan", "1"), ("inf", "inf"), ("1", "nan"), ("inf", "1"), ("-inf", "1")],
                                                       [1, 2, 4])))
def test_permutation_with_non_finite_values(ranks, col):
    bad, count = col
    for where in itertools.combinations(range(5), count):
        r = ranks([bad if j in where else (j + 1, 1) for j in range(5)])
        assert sorted(r) == list(range(5)), (where, r)
        good = [j for j in range(4, -1, -1) if j not in where]
        if bad[0] in ("nan", "-inf") or bad == ("inf", "inf"):      # behind every number
            assert [r[j] for j in good] == list(range(len(good)))
