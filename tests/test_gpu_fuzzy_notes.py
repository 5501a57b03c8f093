"""Tolerance 1 on large prompts: the positions that the counting scan notes, at the edges of the room for notes."""
import numpy as np
import pytest

from harness import Pair
from paper_2503_05330_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L,V,k", [(9, 700, 60, 3), (5, 1501, 12, 4), (130, 64, 300, 2)])
def test_match_lists_that_hold_the_notes_just_so_and_not_quite(N, L, V, k):
    # m matches in all: slices and notes side by side take 3 m + 1 entries, the slices alone m
    tokens, lps = synth.small_random(N, L, V, 12000 + L)
    lens = (L - 3 - (np.arange(N) * 7) % (L // 3)).astype(np.int32)
    from oracle import Oracle
    o = Oracle(1, N, L, V, 5, eps=1)
    o.append(tokens[:, :L - 3], lps[:, :L - 3], lens)
    o.build_all(k)
    m = sum(len(o.matches(i)) for i in range(N))
    assert 100 < 3 * m + 8 < N * N * L                                  # (less than that: not the single-launch build)
    for cap in (m, m + 1, 2 * m, 3 * m - 3, 3 * m - 1, 3 * m, 3 * m + 1, 3 * m + 2, 3 * m + 3, 3 * m + 8):
        pair = Pair(1, N, L, V, 4, 5, eps=1, match_capacity=cap)
        pair.append(tokens[:, :L - 3], lps[:, :L - 3], lens, expect_status=0)
        pair.build_and_compare(k)
        pair.build_and_compare(k)


def test_back_off_rounds_whose_slices_reach_into_the_notes():
    N, L, V = 8, 600, 40
    tokens, lps = synth.small_random(N, L, V, 12700)
    lens = (590 - np.arange(N) * 11).astype(np.int32)
    from oracle import Oracle
    o = Oracle(1, N, L, V, 5, eps=1)
    o.append(tokens[:, :590], lps[:, :590], lens)
    total = 0
    for i in range(N):                                                  # what the rounds' slices hold in all
        for k in (4, 3, 2):
            o.build_path(k, i)
            if len(o.matches(i)):
                total += len(o.matches(i))
                break
    for cap in (total, total + 9, 2 * total, 3 * total, 4 * total):
        pair = Pair(1, N, L, V, 4, 5, eps=1, match_capacity=cap)
        pair.append(tokens[:, :590], lps[:, :590], lens, expect_status=0)
        pair.backoff_and_compare(4)
