"""The single-launch build hands queries with many matches to the launch that all SMs share (k = 1 on prompts of 65536 tokens and
more, k <= 2 with tolerance 1 from 16384): match counts around its limits, its fallbacks, and builds that follow one another."""
import numpy as np
import pytest

from harness import Pair, run_step_protocol

pytestmark = pytest.mark.gpu

COUNTS = [0, 1, 127, 128, 129, 300, 511, 512, 513, 900]


def planted(G, N, L, seed):
    """Path i of a prompt ends in a token of its own that the prompt's other paths hold COUNTS[i % 10] times; followers are half from a
    small heavy-tailed alphabet."""
    rng = np.random.default_rng(seed)
    V = 5000
    tokens = np.minimum((rng.random((G * N, L)) ** 3 * 48).astype(np.int32), 47)
    tokens = np.where(rng.random(tokens.shape) < 0.5, rng.integers(0, V, tokens.shape), tokens).astype(np.int32)
    lps = (-rng.exponential(0.5, tokens.shape)).astype(np.float32)
    lens = (L - 20 - (np.arange(G * N) * 7) % 13).astype(np.int32)
    for g in range(G):
        spots = rng.permutation(N * (L - 40))                          # (path, position), each once
        at = 0
        for n in range(N):
            for _ in range(COUNTS[n % len(COUNTS)]):
                while spots[at] % N == n:                               # (never in the query's own path)
                    at += 1
                tokens[g * N + spots[at] % N, spots[at] // N] = V + n
                at += 1
        for n in range(N):
            tokens[g * N + n, lens[g * N + n] - 1] = V + n
    return tokens, lps, lens, V + N


@pytest.mark.parametrize("G,N,L,kw", [
    (1, 32, 2051, {}),
    (1, 32, 2048, dict(alpha=0.5)),
    (1, 32, 2048, dict(mode=1)),
    (1, 32, 2048, dict(max_matches=9)),
    (1, 32, 2048, dict(wide_table_bytes=16 * 6 * 700)),                 # room for the first few
    (1, 32, 2048, dict(wide_table_bytes=64)),                           # room asked for in vain only
    (1, 32, 2048, dict(wide_table_bytes=-1)),
    (1, 32, 2047, {}),                                                  # below the limit
    (9, 40, 1640, {}),                                                  # 360 paths: CTAs with others behind them, and a last round
    (15, 40, 1640, {}),                                                 # 600: too many
])
def test_counts_around_the_limits(G, N, L, kw):
    tokens, lps, lens, V = planted(G, N, L, 9000 + L)
    pair = Pair(G, N, L, V, 2, 6, B=2, Ke=2, **kw)
    pair.append(tokens, lps, lens, expect_status=0)
    for k in (1, 2, 1, 1):
        pair.build_and_compare(k, check_dag=G == 1)


@pytest.mark.parametrize("eps", [0, 1])
def test_steps_of_one_launch_and_one_for_the_heavy_queries(eps):
    N, L = (16, 4100) if eps == 0 else (16, 1026)
    rng = np.random.default_rng(88)
    tokens = np.minimum((rng.random((N, L)) ** 3 * 150).astype(np.int32), 149)
    lps = (-rng.exponential(0.5, tokens.shape)).astype(np.float32)
    pair = Pair(1, N, L, 150, 3, 7, eps=eps, max_append=7)
    assert pair.g.step_is_single_launch()
    start = (L - 90 - (np.arange(N) * 5) % 31).astype(np.int32)
    st = run_step_protocol(pair, tokens, lps, [1, 2, 3, 1, 2], steps=14, warm=0, start_lens=start, check_every=3)
    assert st["steps"] > 10
    assert max(len(pair.o.matches(i)) for i in range(N)) > 0


def test_tolerance_one_at_its_shortest_suffixes():
    G, N, L, V = 2, 16, 1024, 90
    rng = np.random.default_rng(89)
    tokens = np.minimum((rng.random((G * N, L)) ** 2 * V).astype(np.int32), V - 1)
    lps = (-rng.exponential(0.5, tokens.shape)).astype(np.float32)
    pair = Pair(G, N, L, V, 3, 5, eps=1, B=2, Ke=2)
    pair.append(tokens, lps, (L - 3 - (np.arange(G * N) * 3) % 29).astype(np.int32), expect_status=0)
    for k in (2, 1, 3, 2, 1):
        pair.build_and_compare(k)
