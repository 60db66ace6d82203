"""Performance cases of the search library: what its users have it do, through its public entry points.

Every case is a dict of plain values.  ``kind`` says which entry point it goes through:

  search    walks already admitted to a context advance by ``moves`` steps (``Context.step``) and their
            results are read back: the body of every long run
  fitness   the same for the merit-factor objective (alpha = 2 in both phases), whose result is the lowest
            energy and its sequence
  serve     a burst of requests of mixed length through ``serving.serve``: submission, admission,
            initialisation, steps, readback and release
  rounds    restart-from-best rounds (``rounds.restart_rounds``)
  autocorr  ``psl_autocorr`` of host sequences

Walk budgets are far beyond what is measured (a walk that reached its budget would stop working).
"""
import math
import random

import numpy as np
import torch

import paper_2107_09801_gb300 as P
from paper_2107_09801_gb300.rounds import restart_rounds
from paper_2107_09801_gb300.serving import serve
from psl_workloads import FLIP_LMT, LS_LMT, N_LMT, Request, WalkSpec, random_pm1

BUDGET = 1 << 40


def _search(name, L, walks, moves, alpha1=4, alpha2=13, n_lmt=N_LMT, ls_lmt=LS_LMT, flip_lmt=FLIP_LMT, topk=1,
            graph=0, hot_threads=0, hot_tile_sb=0, form="batched", kind="search"):
    return dict(name=name, kind=kind, L=L, walks=walks, moves=moves, alpha1=alpha1, alpha2=alpha2, n_lmt=n_lmt,
                ls_lmt=ls_lmt, flip_lmt=flip_lmt, topk=topk, graph=graph, hot_threads=hot_threads,
                hot_tile_sb=hot_tile_sb, form=form)


def listed():
    tuned = dict(hot_threads=896, hot_tile_sb=32)  # what the autotuner picks for batches of long walks
    return [
        # one short walk with its full neighbourhood: nothing to fill the GPU with, so the latency of a
        # step's launches and serial phases is the whole time
        _search("one_walk_1023", 1023, 1, 500, n_lmt=1023, graph=50),
        # one long walk on the whole GPU: a single sequence of record length
        _search("one_walk_131071", 131071, 1, 200, graph=50),
        # many short walks with both exponents: parameter studies, the short end of the length range
        _search("batch_1023", 1023, 4096, 200, graph=50),
        # the merit-factor batch, run for its budget of 2000 moves
        _search("labs_1023", 1023, 4096, 2000, alpha1=2, alpha2=2, graph=100, kind="fitness"),
        # a setting of the LS_lmt x FLIP_lmt study that switches phase every few moves: the general update
        # pass (several flips at once, partner windows rebuilt) runs all the time; a length that is not
        # a power of two less one
        _search("switching_4093", 4093, 256, 200, ls_lmt=3, graph=50),
        # the batch of medium length with the exact re-check of the four best-ranked neighbours
        _search("batch_16383", 16383, 1024, 60, topk=4, graph=20, **tuned),
        # the headline batch
        _search("batch_131071", 131071, 1024, 24, graph=12, **tuned),
        # the longest walks
        _search("batch_1048575", 1048575, 148, 8, alpha2=10, graph=8, **tuned),
        # one walk per launch with selection on the host: the execution model of the paper
        _search("plain_16383", 16383, 1, 20, form="plain"),
        # a burst of serving requests of mixed length and exponents (short budgets, so that admission,
        # readback and release count)
        dict(name="serve_mixed", kind="serve", requests=64, m_min=10, m_max=17, budget_min=10, budget_max=100,
             steps_per_round=16, graph=8),
        # restart rounds: every walk of a round starts from the best sequence of the last
        dict(name="rounds_8191", kind="rounds", L=8191, walks=64, rounds=3, budget=30, alpha1=4, alpha2=13),
        # autocorrelation of sequences in host memory: scoring a set of candidates from elsewhere
        dict(name="autocorr_65535", kind="autocorr", L=65535, nseq=32),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng: random.Random):
    kind = rng.choices(["search", "fitness", "serve", "rounds", "autocorr", "plain"], [6, 2, 1, 1, 1, 1])[0]
    if kind == "autocorr":
        L = _log_int(rng, 257, 131071)
        return dict(kind="autocorr", L=L, nseq=_log_int(rng, 1, max(1, min(64, (1 << 21) // L))))
    if kind == "rounds":
        a1 = rng.randint(2, 6)
        return dict(kind="rounds", L=_log_int(rng, 300, 16383), walks=_log_int(rng, 8, 64), rounds=rng.randint(2, 3),
                    budget=rng.randint(8, 30), alpha1=a1, alpha2=rng.randint(a1 + 4, 13))
    if kind == "serve":
        m = rng.randint(10, 13)
        return dict(kind="serve", requests=_log_int(rng, 12, 64), m_min=m, m_max=rng.randint(m + 1, 17),
                    budget_min=rng.randint(5, 20), budget_max=rng.randint(30, 100), steps_per_round=16, graph=8)
    if kind == "plain":
        c = _search("", _log_int(rng, 511, 65535), 1, rng.randint(4, 12), form="plain")
    else:
        fitness = kind == "fitness"
        L = _log_int(rng, 200, 8191 if fitness else 1 << 19)
        # walks and moves so that the (neighbour, shift) terms of a pass stay within an eighth of the headline's
        n_lmt = rng.choice([N_LMT, N_LMT, N_LMT, max(64, L // 3)])
        per_move = min(n_lmt, L) * (L - 1)
        room = 24 * 1024 * N_LMT * 131070 // 8
        walks = _log_int(rng, 1, max(1, min(2048, room // (8 * per_move))))
        moves = max(4, min(200, room // (walks * per_move)))
        a1 = 2 if fitness else rng.randint(2, 6)
        c = _search("", L, walks, moves, alpha1=a1, alpha2=2 if fitness else rng.randint(a1 + 4, 13), n_lmt=n_lmt,
                    ls_lmt=rng.choice([LS_LMT, LS_LMT, 5]), topk=rng.choice([1, 1, 4]), graph=min(20, moves), kind=kind)
    del c["name"]
    return c


class _Walks:
    """A context with its admitted walks, closed when the last reference goes."""

    def __init__(self, ctx, arena, ids=()):
        self.ctx, self.arena, self.ids = ctx, arena, list(ids)

    def __del__(self):
        self.ctx.close()


def _context(nbytes, **kw):
    arena = torch.empty(int(nbytes * 1.1) + (64 << 20), dtype=torch.uint8, device="cuda")
    return P.Context(arena_tensor=arena, **kw), arena


def _host_sequences(case, seed):
    gen = np.random.Generator(np.random.PCG64(seed))
    return (1 - 2 * gen.integers(0, 2, size=(case["nseq"], case["L"]))).astype(np.int8)


def prepare(case, seed):
    rng = random.Random(seed)
    kind = case["kind"]
    if kind in ("search", "fitness"):
        plain = case["form"] == "plain"
        need = case["walks"] * P.psl_walk_bytes(case["L"], case["n_lmt"], 0)
        ctx, arena = _context(need, form=case["form"], max_walks=case["walks"], steps_per_graph=case["graph"],
                              hot_threads=case["hot_threads"], hot_tile_sb=case["hot_tile_sb"])
        state = _Walks(ctx, arena)
        for _ in range(case["walks"]):
            state.ids.append(ctx.submit_ex(case["L"], rng.getrandbits(63), case["alpha1"], case["alpha2"], BUDGET,
                                           n_lmt=case["n_lmt"], ls_lmt=case["ls_lmt"], flip_lmt=case["flip_lmt"],
                                           topk=case["topk"]))
        ctx.step(1)  # admission, initialisation and the first move
        if not plain:
            ctx.set_steps_per_graph(case["graph"])  # the step graph is captured once
        return case, state
    if kind == "serve":
        trace = []
        mix = random.Random(case["requests"])  # the same lengths for every seed: other seeds are other walks
        for _ in range(case["requests"]):
            m = mix.randint(case["m_min"], case["m_max"])
            L = (1 << m) - 1 - (mix.randrange(1 << (m - 2)) if mix.random() < 0.5 else 0)  # half of them odd sizes
            a1 = mix.randint(2, 6)
            trace.append(Request(0.0, WalkSpec(L=L, seed=rng.getrandbits(63), alpha1=a1, alpha2=mix.randint(a1 + 4, 13),
                                               budget=mix.randint(case["budget_min"], case["budget_max"]))))
        need = sum(P.psl_walk_bytes(r.spec.L, r.spec.n_lmt, 0) for r in trace)
        ctx, arena = _context(need, max_walks=len(trace), steps_per_graph=case["graph"])
        return case, _Walks(ctx, arena), trace
    if kind == "rounds":
        ctx, arena = _context(case["walks"] * P.psl_walk_bytes(case["L"], N_LMT, 0), max_walks=case["walks"])
        return case, _Walks(ctx, arena), random_pm1(case["L"], seed), rng.getrandbits(62)
    ctx, arena = _context(0, max_walks=1)
    return case, _Walks(ctx, arena), _host_sequences(case, seed)


def run(state):
    case, walks = state[0], state[1]
    ctx, kind = walks.ctx, case["kind"]
    if kind == "search":
        ctx.step(case["moves"])
        psl_best, seqs = ctx.best_many(walks.ids)
        st = [ctx.poll(w) for w in walks.ids]
        return {"psl_best": psl_best, "best": seqs, "F": np.array([s["F"] for s in st]),
                "progress": np.array([[s["state"], s["moves"], s["flip_evals"], s["switches"], s["psl"], s["alpha"],
                                       s["unimproved"]] for s in st], dtype=np.int64)}
    if kind == "fitness":
        ctx.step(case["moves"])
        found = [ctx.best_fitness(w) for w in walks.ids]
        return {"energy": np.array([e for e, _ in found], dtype=np.int64), "best": np.stack([s for _, s in found])}
    if kind == "serve":
        res = serve(ctx, state[2], steps_per_round=case["steps_per_round"], keep_sequences=True)
        order = sorted(res.psl_best)
        return {"psl_best": np.array([res.psl_best[r][0] for r in order], dtype=np.int32),
                "best": np.concatenate([res.psl_best[r][1] for r in order]), "flip_evals": res.flip_evals,
                "errors": res.errors}
    if kind == "rounds":
        hist = restart_rounds(ctx, case["L"], case["walks"], case["rounds"], case["budget"], case["alpha1"],
                              case["alpha2"], seed0=state[3], start=state[2])
        return {"psl_best": np.array([h.psl_best for h in hist]), "walk": np.array([h.walk for h in hist]),
                "best": np.stack([h.sequence for h in hist])}
    return {"C": ctx.autocorr(state[2])}


def _terms(L, n_lmt=N_LMT):
    """(neighbour, shift) terms of one move."""
    return min(n_lmt, L) * (L - 1)


def work(case):
    """Two lane operations per (neighbour, shift) term of every move; every move reads and writes its walk's
    autocorrelation once (4 bytes a shift each way); a start costs two operations per 32 products."""
    kind = case["kind"]
    if kind in ("search", "fitness"):
        n = case["walks"] * case["moves"]
        return {"bytes": 8 * case["L"] * n + case["L"] * case["walks"], "flops": 2 * n * _terms(case["L"], case["n_lmt"])}
    if kind == "serve":
        n = case["requests"] * (case["budget_min"] + case["budget_max"]) / 2
        Ls = [1 << m for m in range(case["m_min"], case["m_max"] + 1)]  # the mean over the lengths
        return {"bytes": 8 * n * sum(Ls) / len(Ls), "flops": 2 * n * sum(_terms(L) for L in Ls) / len(Ls)}
    if kind == "rounds":
        n = case["walks"] * case["rounds"] * case["budget"]
        return {"bytes": 8 * case["L"] * n, "flops": 2 * n * _terms(case["L"])}
    L, n = case["L"], case["nseq"]
    return {"bytes": 5 * L * n, "flops": n * L * L / 32}


def exact(case, seed):
    """The autocorrelations by FFT in 64 bits, rounded to the integers they are.  The searches return integers,
    bytes and F, the correctly rounded value of an exact integer; an independent search would take minutes."""
    if case["kind"] != "autocorr":
        return None
    s = _host_sequences(case, seed).astype(np.float64)
    n = 1 << (2 * case["L"] - 1).bit_length()
    f = np.fft.rfft(s, n, axis=1)
    return {"C": np.rint(np.fft.irfft(f * np.conj(f), n, axis=1)[:, :case["L"]])}
