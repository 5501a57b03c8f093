"""Indexes of 16 MiB and more chain their n-gram lengths (a position is listed under the shortest n-gram that still had a place):
phrases that occur around and beyond the six places of a bucket, at every suffix length, by every way of appending."""
import numpy as np
import pytest

from harness import Pair, run_step_protocol

pytestmark = pytest.mark.gpu

TIMES = [1, 2, 5, 6, 7, 8, 11, 12, 13, 14, 18, 19, 24, 25, 31, 40, 60]


def phrases(G, N, L, V, seed):
    """Streams of V everyday tokens with phrases of 20 tokens of their own planted in them: phrase c of a prompt TIMES[c] times, and
    begun at the end of a path's first n tokens."""
    rng = np.random.default_rng(seed)
    tokens = rng.integers(0, V, size=(G * N, L)).astype(np.int32)
    lps = (-rng.exponential(0.5, size=tokens.shape)).astype(np.float32)
    start = (L - 100 - (np.arange(G * N) * 37) % 300).astype(np.int32)
    for g in range(G):
        for c, times in enumerate(TIMES):
            phrase = V + 20 * c + np.arange(20)
            phrase[7] = phrase[3]                                     # a 1-gram of it is commoner than the longer ones
            for _ in range(times):
                p, x = g * N + rng.integers(N), rng.integers(0, start.min() - 60)
                tokens[p, x:x + 20] = phrase
    for i in range(G * N):
        c, n = i % len(TIMES), 1 + (i // len(TIMES) + i) % 19
        tokens[i, start[i] - n:start[i] + 20 - n] = V + 20 * c + np.arange(20)
    return tokens, lps, start, V + 20 * len(TIMES)


@pytest.mark.parametrize("G,N,L,k_max,index_max_n,match_capacity", [
    (1, 64, 2048, 16, 0, 0),              # the single-launch build
    (1, 64, 2048, 16, 0, 600000),         # probe, scan, dag
    (1, 64, 2048, 7, 3, 600000),
    (1, 64, 2048, 5, 2, 0),
    (8, 16, 1024, 5, 0, 0),               # one launch per step
])
@pytest.mark.parametrize("V", [200, 20000])
def test_phrases_around_the_places_of_a_bucket(G, N, L, k_max, index_max_n, match_capacity, V):
    tokens, lps, start, vocab = phrases(G, N, L, V, 31 * k_max + V)
    pair = Pair(G, N, L, vocab, k_max, 6, index_max_n=index_max_n, match_capacity=match_capacity, max_append=6)
    first = np.minimum(start, 400 + np.arange(G * N) % 50).astype(np.int32)
    pair.append(tokens[:, :first.max()], lps[:, :first.max()], first, expect_status=0)          # wide rows
    for _ in range(2):                                                                          # narrow rows
        at = pair.o.lengths()[:, None] + np.arange(40)
        pair.append(np.take_along_axis(tokens, at, 1), np.take_along_axis(lps, at, 1), np.full(G * N, 40), expect_status=0)
    rest = start - pair.o.lengths()
    at = np.minimum(pair.o.lengths()[:, None] + np.arange(rest.max()), L - 1)
    pair.append(np.take_along_axis(tokens, at, 1), np.take_along_axis(lps, at, 1), rest, expect_status=0)
    for k in range(1 if V > 200 else 2, k_max + 1):
        pair.build_and_compare(k)
    pair.backoff_and_compare(k_max)
    pair.trim(np.where(np.arange(G * N) % 3 == 0, start - 300, L))                              # tables emptied and filled again
    for k in (2, min(k_max, 4)):
        pair.build_and_compare(k)


@pytest.mark.parametrize("G,N,L,match_capacity", [(8, 16, 1024, 0), (1, 64, 2048, 0), (1, 64, 2048, 600000)])
def test_steps_that_commit_into_full_and_half_full_buckets(G, N, L, match_capacity):
    # paths that say the same at the same time: commits of one launch meet in the same buckets
    tokens, lps, start, vocab = phrases(G, N, L, 3000, 77)
    lens = (start - 90).astype(np.int32)
    for i in range(G * N):
        phrase = vocab + (i % 5) * 30 + np.arange(30)
        tokens[i, lens[i] + 2:lens[i] + 32] = phrase
        tokens[i, lens[i] + 40:lens[i] + 70] = phrase
    pair = Pair(G, N, L, vocab + 150, 5, 6, match_capacity=match_capacity, max_append=6)
    st = run_step_protocol(pair, tokens, lps, [5, 2, 3, 4, 1], steps=20, warm=0, start_lens=lens, check_every=2)
    assert st["steps"] == 20 and st["accepted"] > 0


def test_rows_whose_chunks_count_full_buckets_for_themselves():
    # more chunks than run at once, by the append and by the trim: common 1- and 2-grams are added up per chunk
    G, N, L, V, k_max = 8, 64, 1600, 3000, 5
    tokens, lps, start, vocab = phrases(G, N, L, V, 78)
    rng = np.random.default_rng(79)
    common = (tokens < V) & (rng.random(tokens.shape) < 0.3)
    tokens[common] = rng.integers(0, 3, common.sum())
    pair = Pair(G, N, L, vocab, k_max, 6)
    pair.append(tokens, lps, start, expect_status=0)
    some = range(0, G * N, 7)
    for k in (2, 3, k_max):
        pair.build_and_compare(k, paths=some)
    pair.trim(np.where(np.arange(G * N) % 3 == 0, start - 200, L))
    for k in (2, 4):
        pair.build_and_compare(k, paths=some)
