"""The order of ChooseNBestExpansions' candidates (csrc/rank_order.h): total, so that every place of the kept list is written by
exactly one candidate, also where the approximate logarithm gives neighbours of a row the other order."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WIDTH = 16                                  # entries of a row's list

SOURCE = """
#include "rank_order.h"
// what hyp_step_kernel does with the scores of `rows` lists of `n` entries: ranks[i] of the candidate at place i
extern "C" void rank_lists(double* score, int rows, int n, int* ranks) {
  for (int h = 0; h < rows; ++h) tw::settle_row(score + h * %(w)d, n);
  for (int i = 0; i < rows * %(w)d; ++i) {
    ranks[i] = 0;
    for (int j = 0; j < rows * %(w)d; ++j)
      ranks[i] += tw::ranks_before(tw::order_key(score[j]), j, tw::order_key(score[i]), i);
  }
}
""" % {"w": WIDTH}


@pytest.fixture(scope="module")
def rank_lists(tmp_path_factory):
    cc = shutil.which("g++") or shutil.which("c++")
    if cc is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("rank_order")
    (d / "rank.cpp").write_text(SOURCE)
    subprocess.run([cc, "-O2", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2302_14357_b200", "csrc"), str(d / "rank.cpp"),
                    "-o", str(d / "rank.so")], check=True)
    lib = ctypes.CDLL(str(d / "rank.so"))

    def call(lists, n):
        scores = np.full((len(lists), WIDTH), -np.inf)
        for h, row in enumerate(lists):
            scores[h, :len(row)] = row
        ranks = np.empty(scores.shape, dtype=np.int32)
        lib.rank_lists(scores.ctypes.data_as(ctypes.c_void_p), len(lists), n, ranks.ctypes.data_as(ctypes.c_void_p))
        return scores, ranks
    return call


CASES = [
    [[-2.0000005, -2.0], [-2.00000025]],                     # neighbours inverted, another row's entry between them
    [[-2.0000005, -2.0], [-2.0]],                            # ... equal to the better one
    [[-2.0000005, -2.0], [-2.0000005, -2.0]],                # the same inversion in two rows
    [[-1.0, -3.0 - 1e-6, -3.0, -3.0 + 1e-6, -5.0], [-3.0, -3.0 - 5e-7, -3.0 + 1e-7], [-3.0 + 5e-7]],
    [[0.0, -0.0, 0.0], [-0.0, 0.0]],
]


@pytest.mark.parametrize("lists", CASES)
def test_each_rank_is_taken_once(rank_lists, lists):
    scores, ranks = rank_lists(lists, WIDTH)
    assert sorted(ranks.ravel()) == list(range(ranks.size))
    for row in ranks:
        assert (np.diff(row) > 0).all()                      # a row's candidates keep the row's order
    order = sorted(range(scores.size), key=lambda i: (-scores.flat[i], i))
    assert [int(ranks.flat[i]) for i in order] == list(range(scores.size))
    for row, raw in zip(scores, lists):
        np.testing.assert_array_equal(row[:len(raw)], np.minimum.accumulate(raw))


def test_random_near_ties(rank_lists):
    rng = np.random.default_rng(3)
    for _ in range(200):
        lists = [np.sort(rng.integers(-4, 1, rng.integers(1, WIDTH + 1)))[::-1] * 1e-6 + rng.integers(-3, 4) * 5e-7 for _ in range(rng.integers(1, 17))]
        lists = [row + rng.integers(-2, 3, len(row)) * 7e-7 for row in lists]
        scores, ranks = rank_lists(lists, WIDTH)
        assert sorted(ranks.ravel()) == list(range(ranks.size))
        assert (np.diff(ranks, axis=1) > 0).all()
