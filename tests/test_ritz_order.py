"""The order of the Ritz values (csrc/rank.h, compiled here with g++): the ranks are a
permutation for any values, and numpy's stable order by magnitude for finite ones."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_11989_gb300", "csrc")
SRC = r"""
#include "rank.h"
#include <math.h>
extern "C" void ranks(const double *v, int k, int *out)
{
    for (int i = 0; i < k; ++i) {
        out[i] = 0;
        for (int j = 0; j < k; ++j) out[i] += qs_abs_before(fabs(v[j]), j, fabs(v[i]), i);
    }
}
"""


@pytest.fixture(scope="module")
def ranks(tmp_path_factory):
    d = tmp_path_factory.mktemp("rank")
    (d / "rank.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "rank.cpp"), "-o", str(d / "rank.so")], check=True)
    lib = ctypes.CDLL(str(d / "rank.so"))

    def f(v):
        v = np.ascontiguousarray(v, dtype=np.float64)
        out = np.full(len(v), -1, dtype=np.int32)
        lib.ranks(v.ctypes.data_as(ctypes.c_void_p), len(v), out.ctypes.data_as(ctypes.c_void_p))
        return out
    return f


@pytest.mark.parametrize("k", [2, 16, 64])
def test_ranks_are_a_permutation_whatever_the_values(ranks, k):
    rng = np.random.default_rng(k)
    pool = np.array([np.nan, -np.nan, np.inf, -np.inf, 0.0, -0.0, 5e-324, 1.0, -1.0, 1e308])
    for n_nan in range(k + 1):
        v = rng.choice(pool, k)
        v[rng.permutation(k)[:n_nan]] = np.nan
        r = ranks(v)
        assert sorted(r) == list(range(k)), (v, r)
        finite = ~np.isnan(v)
        assert not finite.any() or r[finite].max() == finite.sum() - 1   # NaN behind every number


@pytest.mark.parametrize("k", [2, 32, 64])
def test_ranks_of_numbers_are_the_stable_order_by_magnitude(ranks, k):
    v = np.random.default_rng(k).integers(-5, 6, k) * 0.25
    order = np.argsort(np.abs(v), kind="stable")
    assert np.array_equal(ranks(v)[order], np.arange(k))
