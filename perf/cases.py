"""The workloads whose speed counts: what a serving loop asks of the library, from the smallest prompt to the largest.

Sizes are those of ``synth.WORKLOADS`` (4 x 256 up to 256 x 8192 paths x tokens, vocabularies of 32000 to 151936),
with odd ones between them.  The token streams follow the same recipe as ``synth.make_streams`` (paths that repeat
segments of a common pool, separated by private tokens), drawn on the GPU.  Every pass starts from an emptied
context or leaves the histories as they are, so that it can be repeated.

Kinds of pass
  decode   a session: reset, append what the paths hold already, first drafts, then `steps` decode steps, each of
           which checks the drafts, commits the sampled tokens and builds the next drafts (sdms_step)
  host     the same with every step's inputs and results in page-locked host memory, waited for step by step
  prefill  a batch of sessions is taken in: reset, append, first drafts
  window   a session that outgrows its capacity: reset, append, trim to the newer half, append, drafts
  beams    drafts by best-path search and several beams per path from the same pools, for every suffix length
"""
import math

import numpy as np
import torch

from paper_2503_05330_b200 import binding

DEVICE = "cuda:0"
BEAMS = 4


def _case(name, kind, G, N, L, V, k_lo, k_max, D, segments, seg_lo, seg_hi, overlap, start, steps, zipf=1.1, seg_zipf=0.0,
          lp_mean=0.5, eps=0, backoff=False, alpha=1.0, cap=0):
    c = dict(kind=kind, G=G, N=N, L=L, V=V, k_lo=k_lo, k_max=k_max, D=D, segments=segments, seg_lo=seg_lo, seg_hi=seg_hi,
             overlap=overlap, start=start, steps=steps, zipf=zipf, seg_zipf=seg_zipf, lp_mean=lp_mean, eps=eps,
             backoff=backoff, alpha=alpha, cap=cap)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest prompt, whole decode from the warm start: every microsecond is latency
        _case("decode_4x256", "decode", 1, 4, 256, 32000, 1, 3, 4, 20, 8, 32, 0.70, 3, 50),
        # one prompt of 16 paths (the benchmark's), driven by a loop that reads each step's result on the host
        _case("host_16x1024", "host", 1, 16, 1024, 128256, 1, 4, 8, 60, 8, 64, 0.40, 512, 48),
        # the same prompt with edit-distance tolerance 1, the setting of the paper's experiments
        _case("decode_16x1024_fuzzy", "decode", 1, 16, 1024, 128256, 2, 4, 8, 60, 8, 64, 0.40, 700, 24, eps=1),
        # odd sizes (rows that are no multiple of 16 bytes), suffix length backing off, mixed edge weights
        _case("decode_11x1501_backoff", "decode", 1, 11, 1501, 100003, 1, 5, 7, 60, 8, 64, 0.40, 1100, 40, backoff=True, alpha=0.5),
        # one prompt of 64 paths
        _case("decode_64x2048", "decode", 1, 64, 2048, 128256, 1, 4, 8, 120, 8, 64, 0.25, 1500, 32),
        # batched serving: 32 prompts of 16 paths with long histories
        _case("decode_32x16x4096", "decode", 32, 16, 4096, 151936, 1, 5, 12, 100, 16, 96, 0.35, 3400, 20, zipf=1.2, lp_mean=0.4),
        # one very wide prompt, popular segments: some suffixes occur thousands of times
        _case("decode_256x8192", "decode", 1, 256, 8192, 151936, 1, 8, 16, 200, 8, 64, 0.10, 7800, 16, seg_zipf=1.0, lp_mean=1.0),
        # wide prompts served in a batch: the largest store, hundreds of queries with hundreds of matches
        _case("decode_16x128x4096", "decode", 16, 128, 4096, 151936, 1, 4, 16, 200, 8, 64, 0.25, 3900, 4),
        # sessions taken in whole (a preempted batch comes back): index construction
        _case("prefill_32x16x4096", "prefill", 32, 16, 4096, 151936, 5, 5, 12, 100, 16, 96, 0.35, 3900, 0, zipf=1.2, lp_mean=0.4),
        # tolerance 1 on a prompt too large for the single-launch build
        _case("decode_96x3001_fuzzy", "decode", 1, 96, 3001, 128256, 3, 4, 8, 120, 8, 64, 0.25, 2500, 6, eps=1),
        # best-path search and four drafts per path, for tree verification
        _case("beams_16x1024", "beams", 1, 16, 1024, 128256, 1, 4, 8, 60, 8, 64, 0.40, 1000, 0),
        # a batch of sessions reaches the end of its window
        _case("window_8x16x1024", "window", 8, 16, 1024, 128256, 4, 4, 8, 60, 8, 64, 0.40, 1000, 0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "decode", "host", "prefill", "beams", "window"])
    eps = int(kind == "decode" and rng.random() < 0.25)
    backoff = kind == "decode" and not eps and rng.random() < 0.25
    while True:
        G, N, L = _log_int(rng, 1, 32), _log_int(rng, 2, 256), _log_int(rng, 200, 8192)
        tokens = G * N * L
        most = {"beams": 1 << 15, "window": 1 << 20, "host": 1 << 17}.get(kind, 1 << 19 if eps else 1 << 23)
        if G * N <= (64 if kind == "beams" else 2048) and (1 << 10) <= tokens <= most and tokens * N <= 1 << 30:
            break
    k_max = rng.randint(3, 8)
    D = rng.randint(4, 16)
    steps = rng.randint(4, 24) if kind in ("decode", "host") else 0
    if tokens > 1 << 20:
        steps = min(steps, 4)
    lo = rng.choice([8, 16])
    start = min(L - 16, max(k_max, int(rng.uniform(0.4, 0.97) * (L - 8 - 2 * steps))))
    big = N * L > 1 << 17
    k_lo = k_max if kind in ("prefill", "window") else (3 if big else 2) if eps else 1
    return _case(None, kind, G, N, L, rng.choice([32000, 100003, 128256, 151936]), k_lo, k_max, D, rng.randint(20, 200), lo,
                 rng.choice([32, 64, 96]), round(rng.uniform(0.1, 0.7) if not big else rng.uniform(0.1, 0.25), 3), start, steps,
                 zipf=rng.choice([1.1, 1.2]), seg_zipf=rng.choice([0.0, 0.0, 1.0]), lp_mean=rng.choice([0.4, 0.5, 1.0]), eps=eps, backoff=backoff,
                 alpha=rng.choice([1.0, 1.0, 0.5]), cap=rng.choice([0, 0, 0, 64]) if kind == "decode" else 0)


# ---- inputs -------------------------------------------------------------------------------------------------
def _zipf_cdf(n, s):
    c = torch.cumsum(torch.arange(1, n + 1, dtype=torch.float64, device=DEVICE) ** -s, 0)
    return c / c[-1]


def _pick(cdf, u):
    return torch.searchsorted(cdf, u, right=True).clamp_(max=cdf.numel() - 1)


def _streams(c, seed):
    """Tokens int32 [P][L] and logprobs float32 [P][L]: per prompt a pool of segments (Zipf token ids); a path is a row
    of runs, each a segment of the pool (with probability `overlap`) or private uniform tokens."""
    G, N, L, V, lo, hi, S = (c[x] for x in ("G", "N", "L", "V", "seg_lo", "seg_hi", "segments"))
    P, runs = G * N, L // lo + 1
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(1 + 7919 * seed)
    rand = lambda *shape: torch.rand(shape, generator=gen, device=DEVICE, dtype=torch.float64)  # noqa: E731
    ints = lambda a, b, *shape: torch.randint(a, b, shape, generator=gen, device=DEVICE)  # noqa: E731
    pool = _pick(_zipf_cdf(V, c["zipf"]), rand(G, S, hi))
    pool_len = ints(lo, hi + 1, G, S)
    shared = rand(P, runs) < c["overlap"]
    seg = _pick(_zipf_cdf(S, c["seg_zipf"]), rand(P, runs)) if c["seg_zipf"] > 0 else ints(0, S, P, runs)
    seg += (torch.arange(P, device=DEVICE) // N * S)[:, None]                # row of the pool of all prompts
    length = torch.where(shared, pool_len.view(-1)[seg], ints(lo, hi + 1, P, runs))
    ends = torch.cumsum(length, 1)
    x = torch.arange(L, device=DEVICE).expand(P, L).contiguous()
    run = torch.searchsorted(ends, x, right=True)
    off = x - (ends - length).gather(1, run)
    tok = torch.where(shared.gather(1, run), pool.view(G * S, hi)[seg.gather(1, run), off], ints(0, V, P, L))
    lp = c["lp_mean"] * torch.log1p(-torch.rand((P, L), generator=gen, device=DEVICE))
    counts = c["start"] - ints(0, max(1, (c["start"] - c["k_max"]) // 8 + 1), P)   # paths of one prompt differ in length
    return tok.to(torch.int32), lp, counts.to(torch.int32)


def _window(tok, lp, lens, width):
    """The next `width` stream entries of every path after position lens (-1 past the stream's end)."""
    at = lens[:, None].long() + torch.arange(width, device=DEVICE)[None]
    ok, at = at < tok.shape[1], at.clamp(max=tok.shape[1] - 1)
    return torch.where(ok, tok.gather(1, at), -1), torch.where(ok, lp.gather(1, at), 0.0)


def _context(c):
    return binding.Sdms(c["G"], c["N"], c["L"], c["V"], c["k_max"], c["D"], device=DEVICE, max_append=c["D"], epsilon=c["eps"],
                        alpha=c["alpha"], max_matches_per_path=c["cap"], host_io=c["kind"] == "host",
                        **(dict(search_mode=2, max_beams=BEAMS) if c["kind"] == "beams" else {}))


def _ks(c):
    span = c["k_max"] - c["k_lo"] + 1
    return [c["k_lo"] + t % span for t in range(c["steps"] + 1)]


def _start(st):
    """Reset, append and first drafts of a session."""
    s = st["s"]
    s.reset()
    s.append(st["tok"], st["lp"], st["counts"])
    if st["c"]["backoff"]:
        s.build_drafts_backoff(st["c"]["k_max"])
    else:
        s.build_drafts(st["ks"][0])


def prepare(case, seed):
    c = dict(case)
    tok, lp, counts = _streams(c, seed)
    s = _context(c)
    n, P, D = c["start"], s.P, s.D
    st = dict(c=c, s=s, counts=counts, tok=tok[:, :n].contiguous(), lp=lp[:, :n].contiguous(), ks=_ks(c))
    if c["kind"] in ("decode", "host"):
        # what the model will answer: play the session once and note the sampled tokens of every step
        answers, lens = [], counts.clone()
        _start(st)
        for t in range(c["steps"]):
            w_tok, w_lp = _window(tok, lp, lens, D + 1)
            answers.append((w_tok, w_lp))
            s.accept(w_tok, w_lp)
            torch.cuda.current_stream().synchronize()
            gained = (s.accept_len.to(DEVICE) + 1).clamp(max=D)
            lens = torch.minimum(lens + gained, torch.full_like(lens, c["L"]))
            if c["backoff"]:
                s.build_drafts_backoff(c["k_max"])
            else:
                s.build_drafts(st["ks"][t + 1])
        st["answers"] = answers
        if c["kind"] == "host":
            st["host_in"] = [torch.cat([a.flatten(), b.flatten().view(torch.int32)]).cpu().numpy() for a, b in answers]
            st["step_in"], st["accept_np"] = s.step_in.numpy(), s.accept_len.numpy()
            st["accepts"] = np.zeros((c["steps"], P), np.int32)
        else:
            st["accepts"] = torch.zeros((c["steps"], P), dtype=torch.int32, device=DEVICE)
            st["accept_rows"] = list(st["accepts"])
    elif c["kind"] == "beams":
        s.append(st["tok"], st["lp"], counts)
        i32, f32 = dict(dtype=torch.int32, device=DEVICE), dict(dtype=torch.float32, device=DEVICE)
        st["out"] = {k: [torch.empty((P, D), **i32), torch.empty(P, **i32), torch.empty((P, D), **f32), torch.empty((P, D), **f32),
                         torch.empty((P, BEAMS, D), **i32), torch.empty((P, BEAMS), **i32), torch.empty((P, BEAMS), **f32)]
                     for k in range(c["k_lo"], c["k_max"] + 1)}
    if c["kind"] == "window":
        half = c["L"] // 2
        st["keep"] = torch.full((P,), half, dtype=torch.int32, device=DEVICE)
        more = c["L"] - half - 16                                                 # the window fills again
        at = (torch.arange(more, device=DEVICE) + n - half) % c["L"]               # the stream goes on (around its end)
        st["more"] = (tok[:, at].contiguous(), lp[:, at].contiguous(), torch.full((P,), more, dtype=torch.int32, device=DEVICE))
    st["history"] = [torch.empty((P, c["L"]), dtype=torch.int32, device=DEVICE) for _ in range(2)]
    st["lens"] = torch.empty(P, dtype=torch.int32, device=DEVICE)
    return st


def run(st):
    c, s, kind = st["c"], st["s"], st["c"]["kind"]
    if kind == "decode":
        _start(st)
        for t, (sampled, lp) in enumerate(st["answers"]):
            if c["backoff"]:
                binding.sdms_step_backoff(s.ctx, c["k_max"], sampled, lp, st["accept_rows"][t], s.draft_tok, s.draft_len,
                                          s.draft_score, s.draft_edge_w, s.used_k)
            else:
                binding.sdms_step(s.ctx, st["ks"][t + 1], sampled, lp, st["accept_rows"][t], s.draft_tok, s.draft_len,
                                  s.draft_score, s.draft_edge_w)
        more = [s.used_k] if c["backoff"] else []
        return [st["accepts"], s.draft_tok, s.draft_len, s.draft_score, s.draft_edge_w, *more, *_history(st)]
    if kind == "host":
        stream = torch.cuda.current_stream()
        handle = stream.cuda_stream
        _start(st)
        for t, answer in enumerate(st["host_in"]):
            np.copyto(st["step_in"], answer)            # the model's answer arrives in the mapped buffer ...
            s.step_own_buffers(st["ks"][t + 1], handle)
            stream.synchronize()                        # ... and the caller reads the result before its next step
            np.copyto(st["accepts"][t], st["accept_np"])
        return [st["accepts"], s.draft_tok, s.draft_len, s.draft_score, s.draft_edge_w, *_history(st)]
    if kind == "beams":
        for k, (tok, ln, score, edge, b_tok, b_len, b_val) in st["out"].items():
            binding.sdms_build_drafts(s.ctx, k, tok, ln, score, edge)
            binding.sdms_get_beams(s.ctx, BEAMS, b_tok, b_len, b_val)
        return {str(k): v for k, v in st["out"].items()}
    if kind == "window":
        s.reset()
        s.append(st["tok"], st["lp"], st["counts"])
        s.trim(st["keep"])
        s.append(*st["more"])
        s.build_drafts(c["k_max"])
    else:
        _start(st)
    return [s.draft_tok, s.draft_len, s.draft_score, s.draft_edge_w, *_history(st)]


def _history(st):
    """The state after the pass, as a caller saves it: stored tokens and probabilities (no path was ever longer than it is
    now: zeros behind) and lengths."""
    binding.sdms_debug_read_history(st["s"].ctx, *st["history"], st["lens"])
    return [*st["history"], st["lens"]]


# ---- what a pass cannot do without ------------------------------------------------------------------------------
def work(case):
    """Bytes: the appended tokens and probabilities in and into the store, per step the sampled tokens and logprobs in, the
    drafts (token, score, edge weight, length) and accept lengths out, and one 32-byte look-up per query.  The followers
    of the matches depend on the streams and are not counted.  No floating-point work worth counting."""
    c = case
    P, D = c["G"] * c["N"], c["D"]
    held = P * c["start"]
    draft = P * (12 * D + 4 + 32 + 4 * c["k_max"])
    b = 16 * held + draft + c["steps"] * (draft + 4 * P + P * (D + 1) * 8 + 16 * P)
    if c["kind"] == "window":
        b += P * c["L"] * 16                             # the kept half moved, as much appended again
    if c["kind"] != "beams":
        b += 2 * 2 * 4 * P * c["L"]                      # the history handed back: read and written
    if c["kind"] == "beams":
        b = (c["k_max"] - c["k_lo"] + 1) * (draft + P * BEAMS * (4 * D + 8))
    return {"bytes": b, "flops": 0}


def tolerance(case):
    """Sums are integers, every choice has a tie rule and every weight is rounded in a stated order: all outputs are the
    same bits in any correct implementation."""
    return "exact"
