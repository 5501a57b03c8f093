"""The single-launch build hands queries with many matches to the launch that all SMs share (k = 1 on prompts of 65536 tokens and
more, k <= 2 with tolerance 1 from 16384): match counts around its limits, its fallbacks, and builds that follow one another."""
import numpy as np
import pytest
import torch

from harness import Pair, run_step_protocol, t32
from oracle import Oracle
from paper_2503_05330_b200 import binding, synth

pytestmark = pytest.mark.gpu

COUNTS = [0, 1, 127, 128, 129, 300, 511, 512, 513, 900]


def planted(G, N, L, seed, counts=COUNTS):
    """Path i of a prompt ends in a token of its own that the prompt's other paths hold counts[i % 10] times; followers are half from a
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
            for _ in range(counts[n % len(counts)]):
                while spots[at] % N == n:                               # (never in the query's own path)
                    at += 1
                tokens[g * N + spots[at] % N, spots[at] // N] = V + n
                at += 1
        for n in range(N):
            tokens[g * N + n, lens[g * N + n] - 1] = V + n
    return tokens, lps, lens, V + N


def worked_off(pair, area, build):
    """Whether build() made the launch for heavy queries lay any out: the table area, the last `area` bytes of the workspace, is written by it alone."""
    tail = pair.g.workspace[pair.g.workspace_bytes - area:]
    tail.fill_(0xa5)
    build()
    return bool((tail != 0xa5).any().item())


AREA = 32 << 20
# one query that makes it worth its while, the others around the limits
FAR = [0, 1, 127, 128, 129, 400, 511, 512, 513, 3600]
FEW = [0, 1, 127, 128, 129, 400, 511, 512, 513] + 10 * [3] + [3600]


@pytest.mark.parametrize("G,N,L,kw", [
    (1, 32, 2051, {}),
    (1, 32, 2048, dict(alpha=0.5)),
    (1, 32, 2048, dict(mode=1)),
    (1, 32, 2048, dict(max_matches=100)),
    (9, 40, 1640, {}),                                                  # 360 paths: CTAs with others behind them, and a last round
    (1, 32, 2051, dict(eps=1)),                                         # tolerance 1: any k <= 2
])
def test_heavy_queries_are_handed_over(G, N, L, kw):
    tokens, lps, lens, V = planted(G, N, L, 9300 + L, FAR if G == 1 else FEW)
    pair = Pair(G, N, L, V, 3, 12, B=2, Ke=2, wide_table_bytes=AREA, **kw)
    pair.append(tokens, lps, lens, expect_status=0)
    for _ in range(2):
        assert worked_off(pair, AREA, lambda: pair.build_and_compare(2 if kw.get("eps") else 1, check_dag=G == 1))
        assert not worked_off(pair, AREA, lambda: pair.build_and_compare(3, check_dag=False))
    if not kw.get("eps"):
        assert worked_off(pair, AREA, lambda: pair.backoff_and_compare(1))


def test_steps_hand_over_when_one_prompt_has_reason_enough():
    G, N, L = 5, 16, 4100
    tokens, lps, lens, V = planted(G, N, L, 9350, FAR)
    tokens[:N], lps[:N], lens[:N] = planted(1, N, L, 9351)[:3]          # prompt 0 has none
    pair = Pair(G, N, L, V, 2, 12, max_append=1, wide_table_bytes=AREA)
    assert pair.g.step_is_single_launch()
    pair.append(tokens, lps, lens - 1, expect_status=0)
    pair.backoff_and_compare(2)
    assert worked_off(pair, AREA, lambda: backoff_step_and_compare(pair, *synth.sampled_window(tokens, lps, lens - 1, 13)))
    assert not worked_off(pair, AREA, lambda: pair.build_and_compare(2))
    assert worked_off(pair, AREA, lambda: pair.build_and_compare(1))


@pytest.mark.parametrize("N,L,counts,area,handed", [
    (32, 2051, [0, 1, 127, 129, 300, 511, 513, 900, 1000, 1100], AREA, False),          # a walk of 1100 matches costs less than the launch
    (32, 2051, FAR, AREA, True),
    (72, 1800, [1400] * 10, AREA, False),                              # more work for the pass than walks by all SMs
    (32, 2051, FAR, 16 * 12 * 6400, False),                            # not enough room for all of them
])
def test_what_makes_it_worth_its_while(N, L, counts, area, handed):
    tokens, lps, lens, V = planted(1, N, L, 9400 + N, counts)
    pair = Pair(1, N, L, V, 2, 12, wide_table_bytes=area)
    pair.append(tokens, lps, lens, expect_status=0)
    assert worked_off(pair, area, lambda: pair.build_and_compare(1)) == handed
    assert worked_off(pair, area, lambda: pair.build_and_compare(1)) == handed


@pytest.mark.parametrize("G,N,L,eps,kw,launches", [
    (1, 32, 2048, 0, {}, 2),
    (1, 32, 2047, 0, {}, 1),                                            # a prompt below the limit
    (15, 40, 1640, 0, {}, 1),                                           # 600 paths
    (1, 32, 2048, 0, dict(wide_table_bytes=-1), 1),
    (1, 16, 1024, 1, {}, 2),
    (1, 16, 1023, 1, {}, 1),
])
def test_which_builds_have_a_second_launch(G, N, L, eps, kw, launches):
    tokens, lps = synth.small_random(G * N, L, 3000, 9600)
    pair = Pair(G, N, L, 3000, 3, 4, eps=eps, **kw)
    last = 2 if eps else 1                                              # the longest suffix that hands over

    def count(k):
        n0 = binding.sdms_launch_count(pair.g.ctx)
        pair.g.build_drafts(k)
        return binding.sdms_launch_count(pair.g.ctx) - n0

    lens = np.full(G * N, L // 3, np.int32)
    pair.append(tokens[:, :L // 3], lps[:, :L // 3], lens, expect_status=0)
    assert count(last) == 1                                             # so far the prompt can hold no more than that
    pair.append(tokens[:, L // 3:L - 8], lps[:, L // 3:L - 8], L - 8 - lens, expect_status=0)
    assert count(last) == launches and count(last + 1) == 1
    pair.build_and_compare(last)


def test_a_graph_of_a_build_serves_longer_histories():
    N, L = 32, 2051
    tokens, lps, lens, V = planted(1, N, L, 9700, FAR)
    pair = Pair(1, N, L, V, 2, 12, wide_table_bytes=AREA)
    pair.append(tokens[:, :300], lps[:, :300], np.full(N, 300, np.int32), expect_status=0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pair.g.build_drafts(1)
    pair.append(tokens[:, 300:], lps[:, 300:], lens - 300, expect_status=0)
    pair.o.build_all(1)
    assert worked_off(pair, AREA, graph.replay)
    tok, ln, sc, ew = pair.o.drafts()
    assert np.array_equal(pair.g.draft_len.cpu().numpy(), ln) and np.array_equal(pair.g.draft_tok.cpu().numpy(), tok)
    np.testing.assert_allclose(pair.g.draft_edge_w.cpu().numpy(), ew, rtol=1e-5, atol=0)


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


def backoff_step_and_compare(pair, sampled, sampled_lp):
    """sdms_step_backoff with k_hi = 1 on both sides."""
    tok, ln, _, _ = pair.o.drafts()
    tau_o, st_o = pair.o.accept_commit(tok, ln, sampled, sampled_lp, pair.max_append)
    pair.o.build_all(1)
    pair.g.draft_score.fill_(7.0)
    tau, gt, gl, gk = pair.g.step_backoff(1, t32(sampled, pair.dev), t32(sampled_lp, pair.dev))
    assert pair.g.status() == st_o
    tok, ln, sc, ew = pair.o.drafts()
    assert np.array_equal(tau.cpu().numpy(), tau_o)
    assert np.array_equal(gl.cpu().numpy(), ln) and np.array_equal(gt.cpu().numpy(), tok)
    assert np.array_equal(gk.cpu().numpy(), [int(len(pair.o.matches(i)) > 0) for i in range(pair.P)])
    np.testing.assert_allclose(pair.g.draft_score.cpu().numpy(), sc, rtol=1e-5, atol=0)
    np.testing.assert_allclose(pair.g.draft_edge_w.cpu().numpy(), ew, rtol=1e-5, atol=0)


@pytest.mark.parametrize("G,N,L,eps", [(1, 32, 2048, 0), (9, 40, 1640, 0), (1, 16, 4100, 0), (1, 16, 1026, 1)])
def test_back_off_that_starts_at_one_token(G, N, L, eps):
    # k_hi = 1 is a build of one suffix length: what its launch hands over is worked off behind it, and nothing of it is left for later builds
    tokens, lps, lens, V = planted(G, N, L, 9100 + L)
    if eps:                                                            # (every position matches: few enough for the wide pass)
        lens = lens - L // 3
    pair = Pair(G, N, L, V, 3, 6, eps=eps, max_append=6)
    for again in range(2):
        if again:
            pair.g.reset()
            pair.o = Oracle(G, N, L, V, 6, eps=eps)
        pair.append(tokens, lps, lens - 40 * again, expect_status=0)
        pair.g.draft_len.fill_(77)
        pair.backoff_and_compare(1)
        heavy = sum(len(pair.o.matches(i)) > 128 for i in range(G * N))
        assert heavy > 0 if again == 0 else True
        pair.build_and_compare(1)
        pair.g.draft_len.fill_(77)
        pair.backoff_and_compare(1)
        pair.backoff_and_compare(3)
        pair.build_and_compare(1)
        for _ in range(3):
            backoff_step_and_compare(pair, *synth.sampled_window(tokens, lps, pair.o.lengths(), 7))
        pair.build_and_compare(2)
        pair.g.draft_len.fill_(77)
        pair.backoff_and_compare(1)                                    # (its list is what the reset finds)


def test_steps_of_prompts_whose_lengths_share_a_sector():
    # the launch for the heavy queries is resident while the step in front of it commits lengths, tokens and probabilities
    G, N, L = 2, 12, 5500
    rng = np.random.default_rng(90)
    tokens = np.minimum((rng.random((G * N, L)) ** 3 * 150).astype(np.int32), 149)
    lps = (-rng.exponential(0.5, tokens.shape)).astype(np.float32)
    pair = Pair(G, N, L, 150, 3, 7, max_append=7)
    assert pair.g.step_is_single_launch()
    start = (L - 80 - (np.arange(G * N) * 5) % 31).astype(np.int32)
    st = run_step_protocol(pair, tokens, lps, [1, 1, 2], steps=20, warm=0, start_lens=start, check_every=5)
    assert st["steps"] > 10
