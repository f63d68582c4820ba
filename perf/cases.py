"""The work that users of this library have it do, as timed cases.

Twelve cases over the public entry points of ``paper_2205_07610_gb300``: short
DNA reads (device batches, a captured plan, host buffers), protein database
search and protein pairs, long DNA pairs (a handful, thousands, a single one),
banded alignment, the training of the band predictor and the serving loop.
Inputs are synthetic, drawn on the GPU from the seed alone, with the shapes of
the library's benchmark and tests:

  reads    |Q| uniform in [lmin, lmax]; S = Q with 5 % substitutions and 1 %
           indels (``mutated``), or an unrelated sequence of the same length
  search   queries uniform in [100, 1000], targets LogNormal(300, 0.6) in
           [10, 5000], BLOSUM62 background residues
  protein  pairs of LogNormal length, S an 85 %-identity copy of Q
  long     |Q| uniform in [lmin, lmax], divergence 1..15 %, 10..40 % of the
           events indels
  serve    lengths LogNormal(1000, 1.2) in [100, 50000], 60 % DNA / 40 %
           protein, half local and half global
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2205_07610_gb300 as ga

_BLOSUM62 = np.array([[int(v) for v in row.split()] for row in """
4 -1 -2 -2 0 -1 -1 0 -2 -1 -1 -1 -1 -2 -1 1 0 -3 -2 0 -2 -1 0 -4
-1 5 0 -2 -3 1 0 -2 0 -3 -2 2 -1 -3 -2 -1 -1 -3 -2 -3 -1 0 -1 -4
-2 0 6 1 -3 0 0 0 1 -3 -3 0 -2 -3 -2 1 0 -4 -2 -3 3 0 -1 -4
-2 -2 1 6 -3 0 2 -1 -1 -3 -4 -1 -3 -3 -1 0 -1 -4 -3 -3 4 1 -1 -4
0 -3 -3 -3 9 -3 -4 -3 -3 -1 -1 -3 -1 -2 -3 -1 -1 -2 -2 -1 -3 -3 -2 -4
-1 1 0 0 -3 5 2 -2 0 -3 -2 1 0 -3 -1 0 -1 -2 -1 -2 0 3 -1 -4
-1 0 0 2 -4 2 5 -2 0 -3 -3 1 -2 -3 -1 0 -1 -3 -2 -2 1 4 -1 -4
0 -2 0 -1 -3 -2 -2 6 -2 -4 -4 -2 -3 -3 -2 0 -2 -2 -3 -3 -1 -2 -1 -4
-2 0 1 -1 -3 0 0 -2 8 -3 -3 -1 -2 -1 -2 -1 -2 -2 2 -3 0 0 -1 -4
-1 -3 -3 -3 -1 -3 -3 -4 -3 4 2 -3 1 0 -3 -2 -1 -3 -1 3 -3 -3 -1 -4
-1 -2 -3 -4 -1 -2 -3 -4 -3 2 4 -2 2 0 -3 -2 -1 -2 -1 1 -4 -3 -1 -4
-1 2 0 -1 -3 1 1 -2 -1 -3 -2 5 -1 -3 -1 0 -1 -3 -2 -2 0 1 -1 -4
-1 -1 -2 -3 -1 0 -2 -3 -2 1 2 -1 5 0 -2 -1 -1 -1 -1 1 -3 -1 -1 -4
-2 -3 -3 -3 -2 -3 -3 -3 -1 0 0 -3 0 6 -4 -2 -2 1 3 -1 -3 -3 -1 -4
-1 -2 -2 -1 -3 -1 -1 -2 -2 -3 -3 -1 -2 -4 7 -1 -1 -4 -3 -2 -2 -1 -2 -4
1 -1 1 0 -1 0 0 0 -1 -2 -2 0 -1 -2 -1 4 1 -3 -2 -2 0 0 0 -4
0 -1 0 -1 -1 -1 -1 -2 -2 -1 -1 -1 -1 -2 -1 1 5 -2 -2 0 -1 -1 0 -4
-3 -3 -4 -4 -2 -2 -3 -2 -2 -3 -2 -3 -1 1 -4 -3 -2 11 2 -3 -4 -3 -2 -4
-2 -2 -2 -3 -2 -1 -2 -3 2 -1 -1 -2 -1 3 -3 -2 -2 2 7 -1 -3 -2 -1 -4
0 -3 -3 -3 -1 -2 -2 -3 -3 3 1 -2 1 -1 -2 -2 0 -3 -1 4 -3 -2 -1 -4
-2 -1 3 4 -3 0 1 -1 0 -3 -4 0 -3 -3 -2 0 -1 -4 -3 -3 4 1 -1 -4
-1 0 0 1 -3 3 4 -2 0 -3 -3 1 -1 -3 -1 0 -1 -3 -2 -2 1 4 -1 -4
0 -1 -1 -1 -2 -1 -1 -1 -1 -1 -1 -1 -1 -1 -2 0 0 -2 -1 -1 -1 -1 -1 -4
-4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 1
""".strip().splitlines()], dtype=np.int8)
# background frequencies of the first 20 residues
_BACKGROUND = [0.07805, 0.05129, 0.04487, 0.05364, 0.01925, 0.04264, 0.06295, 0.07377, 0.02199, 0.05142,
               0.09019, 0.05744, 0.02243, 0.03856, 0.05203, 0.07120, 0.05841, 0.01330, 0.03216, 0.06441]
_DNA = (np.where(np.eye(4, dtype=bool), 2, -3).astype(np.int8), 5, 2)  # match +2 / mismatch -3, open 5, extend 2
_PROTEIN = (_BLOSUM62, 11, 1)


# ---- the cases --------------------------------------------------------------

def listed():
    return [
        # one request's worth of sequencing reads: the smallest call, all latency
        {"name": "reads_small", "kind": "reads", "entry": "batch", "npairs": 1000, "lmin": 150, "lmax": 150,
         "mutated": False, "modes": "local"},
        # the same size in a loop that keeps a plan and replays its graph
        {"name": "reads_plan", "kind": "reads", "entry": "plan", "npairs": 1000, "lmin": 100, "lmax": 300,
         "mutated": True, "modes": "global"},
        # a lane of reads against their candidate sites, two modes in one call
        {"name": "reads_modes", "kind": "reads", "entry": "modes", "npairs": 1_000_000, "lmin": 100, "lmax": 300,
         "mutated": True, "modes": "global,semiglobal"},
        # reads in pinned host memory, scores back in host memory
        {"name": "reads_host", "kind": "reads", "entry": "host", "npairs": 400_000, "lmin": 100, "lmax": 300,
         "mutated": True, "modes": "local"},
        # database search: the largest case
        {"name": "search", "kind": "search", "nq": 96, "nt": 40_000, "mode": "local"},
        # rescoring the hits of a search: protein pairs
        {"name": "protein_pairs", "kind": "protein", "npairs": 10_000, "median": 300, "mode": "local"},
        # overlaps of one long read with its candidates
        {"name": "long_few", "kind": "long", "npairs": 48, "lmin": 5000, "lmax": 20_000, "mode": "semiglobal"},
        # a batch of long reads against their references
        {"name": "long_many", "kind": "long", "npairs": 2000, "lmin": 1000, "lmax": 20_000, "mode": "global"},
        # one long pair, where the answer is waited for
        {"name": "long_single", "kind": "single", "m": 20_000, "n": 20_000, "protein": False, "mode": "local"},
        # exact global scores by band doubling, from the best constant start
        {"name": "banded", "kind": "banded", "npairs": 1500, "lmin": 1000, "lmax": 20_000, "w0": 1024},
        # training of the band predictor
        {"name": "predictor_train", "kind": "train", "samples": 4000, "steps": 300, "batch": 256},
        # a burst of requests of every size through the alignment server
        {"name": "serve_burst", "kind": "serve", "requests": 4000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["reads", "reads", "reads", "search", "protein", "long", "long", "single", "banded", "train", "serve"])
    mode = rng.choice(["local", "global", "semiglobal"])
    if kind == "reads":
        lmin, lmax = rng.choice([(100, 300), (150, 150), (rng.randint(40, 120), rng.randint(121, 600)),
                                 (rng.randint(200, 400), rng.randint(401, 1000))])
        entry = rng.choice(["batch", "plan", "modes", "host"])
        most = min({"plan": 50_000, "host": 400_000}.get(entry, 1_000_000), int(2e8 / lmax))
        return {"kind": kind, "entry": entry, "npairs": _log_int(rng, 100, most), "lmin": lmin, "lmax": lmax,
                "mutated": rng.random() < 0.75, "modes": "global,semiglobal" if entry == "modes" else mode}
    if kind == "search":
        # mostly local; whole-sequence modes for sets of domains
        local = rng.random() < 0.7
        return {"kind": kind, "nq": _log_int(rng, 4, 90 if local else 16), "nt": _log_int(rng, 500, 40_000 if local else 8000),
                "mode": "local" if local else mode}
    if kind == "protein":
        return {"kind": kind, "npairs": _log_int(rng, 300, 12_000), "median": rng.randint(120, 600), "mode": mode}
    if kind == "long":
        lmax = rng.randint(3000, 20_000)
        return {"kind": kind, "npairs": _log_int(rng, 8, 1800), "lmin": rng.randint(700, 2500), "lmax": lmax, "mode": mode}
    if kind == "single":
        return {"kind": kind, "m": _log_int(rng, 700, 40_000), "n": _log_int(rng, 700, 40_000),
                "protein": rng.random() < 0.4, "mode": mode}
    if kind == "banded":
        return {"kind": kind, "npairs": _log_int(rng, 30, 1400), "lmin": rng.randint(300, 1500),
                "lmax": rng.randint(2000, 20_000), "w0": _log_int(rng, 16, 2048)}
    if kind == "train":
        return {"kind": kind, "samples": _log_int(rng, 500, 8000), "steps": _log_int(rng, 20, 300),
                "batch": _log_int(rng, 16, 512)}
    return {"kind": kind, "requests": _log_int(rng, 100, 4000)}


# ---- inputs -----------------------------------------------------------------

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    return g


def _offsets(lens):
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device=lens.device)
    torch.cumsum(lens, 0, out=off[1:])
    return off


def _uniform_lengths(g, n, lo, hi):
    return torch.randint(lo, hi + 1, (n,), generator=g, device=_device())


def _lognormal_lengths(g, n, median, sigma, lo, hi):
    z = torch.randn(n, generator=g, device=_device(), dtype=torch.float64)
    return (z * sigma).exp().mul(median).round().clamp(lo, hi).to(torch.int64)


def _residues(g, n, protein):
    if not protein:
        return torch.randint(0, 4, (n,), generator=g, device=_device(), dtype=torch.uint8)
    cdf = torch.tensor(_BACKGROUND, dtype=torch.float64, device=_device()).cumsum(0)
    cdf = (cdf / cdf[-1]).to(torch.float32)[:-1].contiguous()
    u = torch.rand(n, generator=g, device=_device())
    return torch.searchsorted(cdf, u, right=True).to(torch.uint8)


def _mutate(g, codes, off, p_event, indel_frac, protein):
    """A copy of every sequence: per position an event with probability
    p_event, an indel (half insertions, half deletions, lengths geometric with
    mean 2) with probability indel_frac, else a substitution."""
    dev, N, nseq, A = codes.device, codes.numel(), off.numel() - 1, 20 if protein else 4
    seq = torch.repeat_interleave(torch.arange(nseq, device=dev, dtype=torch.int32), off[1:] - off[:-1], output_size=N)
    p = p_event[seq.long()] if isinstance(p_event, torch.Tensor) else p_event
    at = torch.nonzero(torch.rand(N, generator=g, device=dev) < p).squeeze(1)
    f = indel_frac[seq[at].long()] if isinstance(indel_frac, torch.Tensor) else indel_frac
    indel = torch.rand(at.numel(), generator=g, device=dev) < f
    ins = torch.rand(at.numel(), generator=g, device=dev) < 0.5
    sub, ipos, dpos = at[~indel], at[indel & ins], at[indel & ~ins]
    out = codes.clone()
    out[sub] = ((out[sub].long() + torch.randint(1, A, (sub.numel(),), generator=g, device=dev)) % A).to(torch.uint8)

    def geometric(n):
        return torch.rand(n, generator=g, device=dev, dtype=torch.float64).clamp_min(1e-9).log().div(math.log(0.5)).floor().long() + 1

    edge = torch.zeros(N + 1, dtype=torch.int32, device=dev)
    ends = torch.minimum(dpos + geometric(dpos.numel()), off[seq[dpos].long() + 1])
    one = torch.ones(1, dtype=torch.int32, device=dev)
    edge.index_add_(0, dpos, one.expand(dpos.numel()))
    edge.index_add_(0, ends, -one.expand(ends.numel()))
    new = torch.zeros(N, dtype=torch.int64, device=dev)
    new[ipos] = geometric(ipos.numel())
    kept = (torch.cumsum(edge[:N], 0) == 0).long() + new
    start = _offsets(kept)
    total = int(start[-1])
    src = torch.repeat_interleave(torch.arange(N, device=dev), kept, output_size=total)
    fresh = torch.arange(total, device=dev) - start[src] < new[src]
    res = out[src]
    res[fresh] = _residues(g, int(fresh.sum()), protein)
    return res, start[off]


def _pairs(g, lens, protein, p_event, indel_frac):
    off = _offsets(lens)
    q = _residues(g, int(off[-1]), protein)
    t, toff = _mutate(g, q, off, p_event, indel_frac, protein)
    return q, off, t, toff


def _long_pairs(g, case):
    n = case["npairs"]
    lens = _uniform_lengths(g, n, case["lmin"], case["lmax"])
    d = torch.rand(n, generator=g, device=_device()) * 0.14 + 0.01
    f = torch.rand(n, generator=g, device=_device()) * 0.3 + 0.1
    return _pairs(g, lens, False, d, f)


def _inputs(case, seed):
    """The sequences of a case as device tensors (q, q_off, t, t_off)."""
    g, kind = _generator(seed), case["kind"]
    if kind == "reads":
        lens = _uniform_lengths(g, case["npairs"], case["lmin"], case["lmax"])
        if case["mutated"]:
            return _pairs(g, lens, False, 0.06, 1 / 6)
        off = _offsets(lens)
        return _residues(g, int(off[-1]), False), off, _residues(g, int(off[-1]), False), off.clone()
    if kind == "search":
        qo = _offsets(_uniform_lengths(g, case["nq"], 100, 1000))
        to = _offsets(_lognormal_lengths(g, case["nt"], 300, 0.6, 10, 5000))
        return _residues(g, int(qo[-1]), True), qo, _residues(g, int(to[-1]), True), to
    if kind == "protein":
        return _pairs(g, _lognormal_lengths(g, case["npairs"], case["median"], 0.6, 20, 3000), True, 0.15, 0.1)
    if kind in ("long", "banded"):
        return _long_pairs(g, case)
    raise ValueError(kind)


def _single_inputs(case, seed):
    """Two related sequences: T a mutated copy of Q, cut or extended to n residues."""
    g, m, n, protein = _generator(seed), case["m"], case["n"], case["protein"]
    q = _residues(g, m, protein)
    off = torch.tensor([0, m], dtype=torch.int64, device=_device())
    t, _ = _mutate(g, q, off, 0.08, 0.2, protein)
    if t.numel() < n:
        t = torch.cat([t, _residues(g, n - t.numel(), protein)])
    return q, t[:n].contiguous()


def _train_inputs(case, seed):
    """Features in [0, 1], targets log2(1 + w), He-uniform weights, minibatches."""
    g, dev, n = _generator(seed), _device(), case["samples"]
    x = torch.rand(n, 32, generator=g, device=dev)
    y = 3 + 6 * x[:, 4] + 2 * x[:, 20] * x[:, 2] + 0.1 * torch.randn(n, generator=g, device=dev)
    u = torch.rand(6337, generator=g, device=dev) * 2 - 1
    w = torch.zeros(6337, device=dev)
    w[:2048] = u[:2048] * math.sqrt(6 / 32)
    w[2112:6208] = u[2112:6208] * math.sqrt(6 / 64)
    w[6272:6336] = u[6272:6336] * math.sqrt(3 / 64)
    idx = torch.randint(0, n, (case["steps"], case["batch"]), generator=g, device=dev, dtype=torch.int32)
    return {"x": x, "y": y, "master": w, "idx": idx}


def _serve_inputs(case, seed):
    """Requests in arrival order, on the host: CSR codes, mode and scoring index (0 DNA, 1 protein)."""
    g, n = _generator(seed), case["requests"]
    parts = []
    for protein, k in ((False, n - (2 * n) // 5), (True, (2 * n) // 5)):
        lens = _lognormal_lengths(g, k, 1000, 1.2, 100, 50_000)
        q, qo, t, to = _pairs(g, lens, protein, 0.15 if protein else 0.06, 0.1 if protein else 1 / 6)
        parts.append([a.cpu().numpy() for a in (q, qo, t, to)])
    rng = np.random.default_rng(seed)
    order = rng.permutation(n)
    split = len(parts[0][1]) - 1

    def arranged(c):
        seqs = []
        for r in order:
            codes, off = parts[int(r >= split)][c], parts[int(r >= split)][c + 1]
            k = r - split if r >= split else r
            seqs.append(codes[off[k]:off[k + 1]])
        return np.concatenate(seqs), np.concatenate([[0], np.cumsum([len(s) for s in seqs])]).astype(np.int64)

    (q, qo), (t, to) = arranged(0), arranged(2)
    return {"q": q, "qo": qo, "t": t, "to": to, "modes": rng.integers(0, 2, n).astype(np.int32),
            "scorings": (order >= split).astype(np.int32)}


# ---- the server that the process keeps --------------------------------------
_SERVER = {}


def _server():
    """One server per process, as a service keeps it.  Its kernel gives the GPU
    back after 0.2 ms without work, so that other work of the process runs."""
    if not _SERVER:
        s = ga.Server(idle_us=200)
        _SERVER["ids"] = [s.add_scoring(*_DNA), s.add_scoring(*_PROTEIN)]
        _SERVER["server"] = s
    return _SERVER["server"], _SERVER["ids"]


# ---- preparation and one pass -----------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "single":
        q, t = _single_inputs(case, seed)
        return {"case": case, "q": q, "t": t, "scoring": _PROTEIN if case["protein"] else _DNA}
    if kind == "train":
        return {"case": case, **_train_inputs(case, seed)}
    if kind == "serve":
        s = _serve_inputs(case, seed)
        server, ids = _server()
        return {"case": case, "server": server, **s, "scorings": np.asarray(ids, dtype=np.int32)[s["scorings"]]}
    seqs = _inputs(case, seed)
    state = {"case": case, "seqs": seqs, "scoring": _PROTEIN if kind in ("search", "protein") else _DNA}
    if kind == "reads" and case["entry"] == "host":
        state["seqs"] = tuple(a.cpu().pin_memory() for a in seqs)
        state["scores"] = torch.empty(case["npairs"], dtype=torch.int32).pin_memory()
    if kind == "reads" and case["entry"] == "plan":
        # capacity of the loop's batches, not of this one batch
        longest = case["lmax"] + case["lmax"] // 4 + 32
        plan = ga.Plan(*_DNA, case["modes"], case["npairs"], case["npairs"] * longest, longest)
        state["scores"] = torch.empty(case["npairs"], dtype=torch.int32, device=_device())
        plan.capture(*seqs, state["scores"])
        state["plan"] = plan
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "reads":
        entry = case["entry"]
        if entry == "plan":
            state["plan"].launch()
            return state["scores"]
        if entry == "modes":
            return ga.align_batch_modes(*state["seqs"], *state["scoring"], case["modes"].split(","))
        if entry == "host":
            return ga.align_batch_host(*state["seqs"], *state["scoring"], case["modes"], scores=state["scores"])
        return ga.align_batch(*state["seqs"], *state["scoring"], case["modes"])
    if kind == "search":
        return ga.align_cross(*state["seqs"], *state["scoring"], case["mode"])
    if kind in ("protein", "long"):
        return ga.align_batch(*state["seqs"], *state["scoring"], case["mode"])
    if kind == "single":
        return ga.align_long(state["q"], state["t"], *state["scoring"], case["mode"])
    if kind == "banded":
        return list(ga.align_banded(*state["seqs"], *state["scoring"], default_w0=case["w0"]))
    if kind == "train":
        master = state["master"].clone()
        m, v = torch.zeros_like(master), torch.zeros_like(master)
        bf16 = ga.mlp_cast(master)
        losses = ga.mlp_train(master, bf16, m, v, state["x"], state["y"], state["idx"], lr=2e-3)
        return {"master": master, "bf16": bf16.view(torch.bfloat16), "m": m, "v": v, "losses": losses}
    server = state["server"]
    first = server.submit(state["q"], state["qo"], state["t"], state["to"], state["modes"], state["scorings"])
    server.drain()
    got = server.poll()
    scores = np.empty(case["requests"], dtype=np.int32)
    status = np.empty(case["requests"], dtype=np.int32)
    scores[got["id"] - first], status[got["id"] - first] = got["score"], got["status"]
    return {"scores": scores, "status": status}


# ---- what a pass cannot do without ------------------------------------------

def _ops_per_cell(mode):
    """Adds and maxima of the recurrence for one cell; local mode also clamps
    at zero and keeps a maximum."""
    return 9 if mode == "local" else 7


def work(case):
    kind = case["kind"]
    if kind == "reads":
        a, b, n = case["lmin"], case["lmax"], case["npairs"]
        mean, square = (a + b) / 2, (a * a + a * b + b * b) / 3
        modes = case["modes"].split(",")
        return {"bytes": n * (2 * mean + 16 + 4 * len(modes)), "flops": n * square * sum(map(_ops_per_cell, modes))}
    if kind == "search":
        q, t = case["nq"] * 550.0, case["nt"] * 359.0
        return {"bytes": q + t + 4.0 * case["nq"] * case["nt"], "flops": q * t * _ops_per_cell(case["mode"])}
    if kind == "protein":
        n, mean, square = case["npairs"], case["median"] * math.exp(0.18), case["median"] ** 2 * math.exp(0.72)
        return {"bytes": n * (2 * mean + 20), "flops": n * square * _ops_per_cell(case["mode"])}
    if kind == "single":
        return {"bytes": case["m"] + case["n"] + 4, "flops": case["m"] * float(case["n"]) * _ops_per_cell(case["mode"])}
    if kind in ("long", "banded"):
        a, b, n = case["lmin"], case["lmax"], case["npairs"]
        mean, square = (a + b) / 2, (a * a + a * b + b * b) / 3
        if kind == "long":
            return {"bytes": n * (2 * mean + 20), "flops": n * square * _ops_per_cell(case["mode"])}
        band = min(square, mean * (2 * case["w0"] + 1))  # cells of the starting band
        return {"bytes": n * (2 * mean + 24), "flops": n * band * 7}
    if kind == "train":
        k = case["steps"]
        per_sample = 2 * 6337 * 2 + 2 * 64 * 65  # forward, weight gradients, input gradients of layer 2 and the head
        return {"bytes": 4.0 * (3 * 2 * 6337 + case["samples"] * 33 + k * case["batch"]),
                "flops": float(k) * (case["batch"] * per_sample + 6337 * 12)}
    n = case["requests"]
    return {"bytes": n * (2 * 2050.0 + 24), "flops": n * 1000.0 ** 2 * math.exp(2 * 1.44) * 0.75 * 8}  # half local, half global


# ---- the same results in plain 64-bit torch -----------------------------------

def _padded(codes, off):
    lens = off[1:] - off[:-1]
    at = off[:-1, None] + torch.arange(int(lens.max()), device=codes.device)
    return codes.long()[at.clamp_max(codes.numel() - 1)].clamp(0, 23), lens


def _dp(seqs, scoring, mode):
    """Scores of the pairs by the plain affine-gap recurrence, a row at a time.
    Along a row, F(j) = max over k < j of X(k) - open - extend (j - 1 - k),
    X being H before F: a running maximum of X(k) + extend k."""
    q, m = _padded(seqs[0], seqs[1])
    t, n = _padded(seqs[2], seqs[3])
    dev, (B, N) = q.device, t.shape
    sigma = torch.tensor(scoring[0].astype(np.int64), device=dev)
    alpha, beta = scoring[1], scoring[2]
    k = torch.arange(N + 1, device=dev)
    H = torch.where(k == 0, 0, -alpha - beta * (k - 1)) if mode == "global" else torch.zeros_like(k)
    H = H.expand(B, N + 1).clone()
    E = H[:, 1:] - alpha
    real = k[1:] <= n[:, None]
    best = torch.zeros(B, dtype=torch.int64, device=dev)
    for i in range(1, q.shape[1] + 1):
        X = torch.maximum(H[:, :-1] + sigma[q[:, i - 1, None], t], E)
        if mode == "local":
            X = X.clamp_min(0)
        edge = torch.full((B, 1), -alpha - beta * (i - 1) if mode == "global" else 0, dtype=torch.int64, device=dev)
        run_max = torch.cummax(torch.cat([edge, X], 1) + beta * k, 1).values[:, :-1]
        X = torch.maximum(X, run_max - alpha - beta * k[:-1])
        H = torch.cat([edge, X], 1)
        E = torch.maximum(E - beta, X - alpha)
        inside = i <= m
        if mode == "local":
            best = torch.where(inside, torch.maximum(best, X.masked_fill(~real, 0).amax(1)), best)
            continue
        last = torch.gather(H, 1, n[:, None]).squeeze(1)
        if mode == "global":
            best = torch.where(i == m, last, best)
        else:
            best = torch.where(inside, torch.maximum(best, last), best)
            best = torch.where(i == m, torch.maximum(best, X.masked_fill(~real, 0).amax(1)), best)
    return best.to(torch.int32)


def _train(s):
    """Adam on the mean squared error of the 32-64-64-1 network: float64
    weights and state, the forward and backward passes on their bfloat16 copy.
    The first moment has no value here: near the minimum it is a sum of
    gradients that cancel, so a weight that rounds to the other neighbour of
    its bfloat16 copy early on changes most of it."""
    w = s["master"].double()
    m, v, losses = torch.zeros_like(w), torch.zeros_like(w), []
    lr, b1, b2, eps = 2e-3, 0.9, 0.999, 1e-8
    x, y, idx = s["x"].double(), s["y"].double(), s["idx"].long()
    for k in range(idx.shape[0]):
        c = w.to(torch.bfloat16).double()
        W1, c1, W2, c2, w3, c3 = c[:2048].view(64, 32), c[2048:2112], c[2112:6208].view(64, 64), c[6208:6272], c[6272:6336], c[6336]
        xb, B = x[idx[k]], idx.shape[1]
        h1 = (xb @ W1.T + c1).clamp_min(0)
        h2 = (h1 @ W2.T + c2).clamp_min(0)
        r = h2 @ w3 + c3 - y[idx[k]]
        losses.append((r * r).sum() / (2 * B))
        d = r / B
        d2 = d[:, None] * w3 * (h2 > 0)
        d1 = (d2 @ W2) * (h1 > 0)
        grad = torch.cat([(d1.T @ xb).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), d @ h2, d.sum()[None]])
        m = b1 * m + (1 - b1) * grad
        v = b2 * v + (1 - b2) * grad * grad
        w = w - lr * (m / (1 - b1 ** (k + 1))) / ((v / (1 - b2 ** (k + 1))).sqrt() + eps)
    return {"master": w, "bf16": w.to(torch.bfloat16).double(), "m": None, "v": v, "losses": torch.stack(losses)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _train(_train_inputs(case, seed))
    if kind not in ("reads", "protein"):
        return None
    side = case["lmax"] * 1.1 if kind == "reads" else 3000
    if case["npairs"] * side * side > 4e10:
        return None
    seqs = _inputs(case, seed)
    modes = (case["modes"] if kind == "reads" else case["mode"]).split(",")
    scores = [_dp(seqs, _PROTEIN if kind == "protein" else _DNA, md) for md in modes]
    return torch.stack(scores) if kind == "reads" and case["entry"] == "modes" else scores[0].cpu()
