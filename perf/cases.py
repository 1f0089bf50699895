"""The matching work a user of this framework has it do, as cases to be timed:
single texts from the paper's size up to 1 GiB through every output (dense ids,
count, compacted list, every occurrence), host buffers, a batch of texts
against several automata, and the request server.

A case is a dict of plain values; ``prepare`` makes what a program has in hand
before the call (texts on the GPU, compiled automata, output buffers, a plan or
a server), ``run`` is one pass through the public entry points, ``work`` the
bytes that pass cannot do without.  Every output is whole numbers (keyword ids,
positions, counts), which are equal or wrong, so there is no ``exact``.

Keyword sets and texts follow ``paper_1412_7789_gb300/workloads.py`` (same
recipes, made on the GPU so that large texts are quick):

* ``sweep``   ACGT, keywords of 16-64 letters, half copied from the first 4 KiB
* ``single``  ACGT, keywords of 8-32 letters, half copied from all of the text
* ``zipf``    Zipf(1.1) bytes, keywords of 4-100 bytes, 30% copied
* ``paper``   the alphabet repeated, keywords permutations of its 26 letters
"""
import numpy as np
import torch

from paper_1412_7789_gb300 import api, workloads

KIB, MIB, GIB = 1 << 10, 1 << 20, 1 << 30


def listed():
    return [
        # the paper's own workload at its largest text: a call's fixed cost
        {"name": "paper_53710_dense", "kind": "text", "set": "paper", "out": "dense", "n": 53_710, "keywords": 5},
        # the input-size sweep's smallest text, where every position matches
        {"name": "acgt_4k_dense", "kind": "text", "set": "sweep", "out": "dense", "n": 4 * KIB, "keywords": 10_000},
        # one ordinary text, few keywords
        {"name": "acgt_1m_single_dense", "kind": "text", "set": "single", "out": "dense", "n": MIB, "keywords": 100},
        # the sweep's middle at a ragged length, the text at an odd address
        {"name": "acgt_16m_odd_dense", "kind": "text", "set": "sweep", "out": "dense", "n": 16 * MIB + 4_099,
         "keywords": 10_000, "shift": 5},
        # the headline: the sweep's largest text
        {"name": "acgt_1g_dense", "kind": "text", "set": "sweep", "out": "dense", "n": GIB, "keywords": 10_000},
        # a genome-like text with runs of N, as a list of its matches
        {"name": "acgt_256m_gaps_compact", "kind": "text", "set": "sweep", "out": "compact", "n": 256 * MIB,
         "keywords": 10_000, "gaps": True},
        # byte text at a ragged length: how many positions match
        {"name": "zipf_24m_odd_count", "kind": "text", "set": "zipf", "out": "count", "n": 24 * MIB + 777,
         "keywords": 20_000, "shift": 3},
        # every occurrence, sub-patterns included
        {"name": "zipf_128m_full", "kind": "text", "set": "zipf", "out": "full", "n": 128 * MIB, "keywords": 20_000},
        # the byte workload at full size
        {"name": "zipf_1g_compact", "kind": "text", "set": "zipf", "out": "compact", "n": GIB, "keywords": 20_000},
        # host buffers in and out
        {"name": "acgt_48m_host", "kind": "host", "set": "sweep", "n": 48 * MIB + 321, "keywords": 10_000},
        # texts of uneven length against several automata at once
        {"name": "batch_1024", "kind": "batch", "texts": 1024, "sets": 6, "longest": 4 * MIB},
        # requests of every size through the server
        {"name": "serve_64", "kind": "serve", "requests": 64, "longest": 16 * MIB},
    ]


def _log(rng, lo, hi):
    """A whole number of [lo, hi], uniform over its logarithm."""
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["acgt", "acgt", "zipf", "zipf", "paper", "host", "batch", "serve"])
    if kind == "acgt":
        return {"kind": "text", "set": rng.choice(["sweep", "single"]),
                "out": rng.choice(["dense", "count", "compact", "full"]), "n": _log(rng, 4 * KIB, GIB),
                "keywords": _log(rng, 100, 10_000), "shift": rng.randrange(16), "gaps": rng.random() < 0.3}
    if kind == "zipf":
        return {"kind": "text", "set": "zipf", "out": rng.choice(["dense", "count", "compact", "full"]),
                "n": _log(rng, 4 * KIB, 512 * MIB), "keywords": _log(rng, 1_000, 20_000), "shift": rng.randrange(16)}
    if kind == "paper":
        return {"kind": "text", "set": "paper", "out": rng.choice(["dense", "compact"]), "n": _log(rng, 1_310, MIB),
                "keywords": rng.choice([5, 10]), "shift": rng.randrange(16)}
    if kind == "host":
        return {"kind": "host", "set": rng.choice(["sweep", "zipf"]), "n": _log(rng, 64 * KIB, 64 * MIB),
                "keywords": _log(rng, 1_000, 10_000)}
    if kind == "batch":
        return {"kind": "batch", "texts": _log(rng, 16, 1024), "sets": rng.randint(2, 6),
                "longest": _log(rng, 64 * KIB, 4 * MIB)}
    return {"kind": "serve", "requests": _log(rng, 8, 64), "longest": _log(rng, 64 * KIB, 16 * MIB)}


# ---- inputs ------------------------------------------------------------------
_CHUNK = 64 * MIB
_ZIPF = workloads.zipf_table(1.1)


def _text(alphabet, n, g):
    """n random letters on the GPU: uniform ACGT, or Zipf(1.1) bytes."""
    lut = torch.from_numpy(workloads.ACGT.copy() if alphabet == "acgt" else _ZIPF).cuda()
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    for lo in range(0, n, _CHUNK):
        m = min(n, lo + _CHUNK) - lo
        at = torch.randint(0, lut.numel(), (m,), generator=g, device="cuda", dtype=torch.int32)
        torch.index_select(lut, 0, at, out=out[lo:lo + m])
    return out


def _cut(flat, lens):
    ends = np.cumsum(lens)
    data = flat.tobytes()
    return [data[e - m:e] for e, m in zip(ends.tolist(), lens.tolist())]


def _random_keywords(alphabet, r, lens):
    total = int(lens.sum())
    lut = workloads.ACGT if alphabet == "acgt" else _ZIPF
    return _cut(lut[r.integers(0, lut.size, size=total)], lens)


def _copied_keywords(text, r, lens, window):
    """Keywords copied from the first `window` bytes of a text on the GPU."""
    window = min(window, text.numel())
    lens = np.minimum(lens, window)
    offs = r.integers(0, window - lens + 1)
    longest = int(lens.max())
    at = torch.from_numpy(offs).cuda()[:, None] + torch.arange(longest, device="cuda")[None, :]
    rows = text[at.clamp_(max=text.numel() - 1)].cpu().numpy()
    return [row[:m].tobytes() for row, m in zip(rows, lens.tolist())]


def _keywords(which, count, text, r):
    lo, hi, copied, window = {"sweep": (16, 64, 0.5, 4 * KIB), "single": (8, 32, 0.5, text.numel()),
                              "zipf": (4, 100, 0.3, text.numel())}[which]
    alphabet = "zipf" if which == "zipf" else "acgt"
    lens = r.integers(lo, hi + 1, size=count)
    k = int(round(count * copied))
    pats = _copied_keywords(text, r, lens[:k], window) + _random_keywords(alphabet, r, lens[k:])
    return [pats[i] for i in r.permutation(count)]


def _text_and_keywords(case, seed):
    """(the text at the case's offset from an aligned address, its keyword set)."""
    n, which, shift = case["n"], case["set"], case.get("shift", 0)
    r = workloads.rng(seed + 1)
    if which == "paper":
        # the alphabet repeated from a seeded letter on; keyword order seeded
        at = int(r.integers(0, 26))
        letters = torch.from_numpy(workloads.paper_text(n + 26)[at:at + n].copy()).cuda()
        pats = workloads.paper_keywords(case["keywords"], seed)
        pats = [pats[i] for i in r.permutation(len(pats))]
    else:
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        letters = _text("zipf" if which == "zipf" else "acgt", n, g)
        pats = _keywords(which, case["keywords"], letters, r)
        if case.get("gaps"):
            # runs of 200 N, about one in 256 KiB
            starts = torch.randint(0, n, (max(1, n >> 18),), generator=g, device="cuda")
            letters[(starts[:, None] + torch.arange(200, device="cuda")).clamp_(max=n - 1)] = ord("N")
    if shift:
        moved = torch.empty(n + shift, dtype=torch.uint8, device="cuda")
        moved[shift:] = letters
        letters = moved[shift:]
    return letters, pats


def _sets(count, lo, hi, least, most, seed):
    """Keyword sets of growing size, ACGT and Zipf in turn, with random keywords."""
    sizes = np.geomspace(least, most, count).astype(np.int64)
    out = []
    for j, k in enumerate(sizes.tolist()):
        r = workloads.rng(seed + 1000 + j)
        out.append(_random_keywords("acgt" if j % 2 == 0 else "zipf", r, r.integers(lo, hi + 1, size=k)))
    return out


def _filled(n, dtype=torch.int32):
    return torch.full((max(1, n),), -1, dtype=dtype, device="cuda")


def _prepare_text(case, seed):
    text, pats = _text_and_keywords(case, seed)
    s = {"case": case, "automaton": api.Automaton(pats), "text": text, "n": case["n"]}
    if case["out"] == "dense":
        s["ids"] = _filled(case["n"])
    elif case["out"] == "count":
        s["count"] = _filled(1, torch.int64)
    else:
        s["cap"] = case["n"] // 64 + 8 * KIB
        s["pos"], s["ids"], s["count"] = _filled(s["cap"]), _filled(s["cap"]), _filled(1, torch.int64)
    return s


def _prepare_host(case, seed):
    text, pats = _text_and_keywords(case, seed)
    host = torch.empty(case["n"], dtype=torch.uint8, pin_memory=True)
    host.copy_(text)
    ids = torch.empty(case["n"], dtype=torch.int32, pin_memory=True)
    return {"case": case, "automaton": api.Automaton(pats), "text": host, "ids": ids}


def _log_lengths(r, count, lo, hi):
    """Lengths spread evenly over the logarithm of [lo, hi], in a seeded order."""
    at = (np.arange(count) + 0.5) / count
    return r.permutation(np.exp(np.log(lo) + at * np.log(hi / lo)).astype(np.int64))


def _prepare_batch(case, seed):
    r = workloads.rng(seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    sets = case["sets"]
    automata = [api.Automaton(p) for p in _sets(sets, 8, 64, 1_000, 16_500, seed)]
    lens = _log_lengths(r, case["texts"], KIB, case["longest"])
    which = r.integers(0, sets, size=case["texts"])
    offs = np.concatenate([[0], np.cumsum(lens)[:-1]])
    total = int(lens.sum())
    # texts back to back, each in its automaton's alphabet
    texts = torch.empty(total, dtype=torch.uint8, device="cuda")
    acgt, zipf = _text("acgt", total, g), _text("zipf", total, g)
    for o, m, a in zip(offs.tolist(), lens.tolist(), which.tolist()):
        texts[o:o + m] = (acgt if a % 2 == 0 else zipf)[o:o + m]
    plan = api.BatchPlan([a.handle for a in automata], case["texts"])
    plan.reserve_lists(total)
    items = api.items_to_device(api.batch_items(offs, lens, offs, which))
    return {"case": case, "automata": automata, "plan": plan, "texts": texts, "items": items, "ids": _filled(total)}


def _prepare_serve(case, seed):
    r = workloads.rng(seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    automata = [api.Automaton(p) for p in _sets(4, 4, 100, 1_000, 8_000, seed)]
    count = case["requests"]
    lens = _log_lengths(r, count, 256, case["longest"])
    which = r.integers(0, 4, size=count)
    size = 32 * MIB
    pools = [_text("acgt", size, g), _text("zipf", size, g)]
    offs = (r.random(count) * (size - lens + 1)).astype(np.int64)
    caps = np.maximum(1, lens // 64)
    at = np.concatenate([[0], np.cumsum(caps)[:-1]])
    pos, ids, counts = _filled(int(caps.sum())), _filled(int(caps.sum())), _filled(count, torch.int64)
    reqs = np.zeros(count, dtype=api.SERVER_REQUEST)
    reqs["automaton"] = which
    base = np.array([p.data_ptr() for p in pools], dtype=np.uint64)
    reqs["d_text"] = base[which % 2] + offs.astype(np.uint64)
    reqs["n"] = lens
    reqs["d_pos"] = np.uint64(pos.data_ptr()) + 4 * at.astype(np.uint64)
    reqs["d_ids"] = np.uint64(ids.data_ptr()) + 4 * at.astype(np.uint64)
    reqs["cap"] = caps
    reqs["d_count"] = np.uint64(counts.data_ptr()) + 8 * np.arange(count, dtype=np.uint64)
    torch.cuda.current_stream().synchronize()  # the server's streams read what was made here
    server = api.Server([a.handle for a in automata], hbm_budget=8 << 30)
    return {"case": case, "automata": automata, "server": server, "pools": pools, "reqs": reqs,
            "arrivals": np.zeros(count), "pos": pos, "ids": ids, "counts": counts}


def prepare(case, seed):
    return {"text": _prepare_text, "host": _prepare_host, "batch": _prepare_batch,
            "serve": _prepare_serve}[case["kind"]](case, seed)


# ---- one pass ------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "text":
        out, a = case["out"], state["automaton"]
        if out == "dense":
            return a.match(state["text"], out=state["ids"])
        if out == "count":
            return a.count(state["text"], out=state["count"])
        call = api.ac_match_compact if out == "compact" else api.ac_match_full
        call(a.handle, state["text"], state["n"], state["pos"], state["ids"], state["cap"], state["count"])
        return state["pos"], state["ids"], state["count"]
    if kind == "host":
        return state["automaton"].match_host(state["text"], out=state["ids"])
    if kind == "batch":
        state["plan"].run(state["texts"], state["items"], case["texts"], state["ids"])
        return state["ids"]
    server = state["server"]
    server.replay(state["reqs"], state["arrivals"])
    server.drain()
    server.poll(case["requests"])
    return state["pos"], state["ids"], state["counts"]


# ---- the bytes of a pass -------------------------------------------------------
def _mean_length(lo, hi):
    return (hi - lo) / np.log(hi / lo)


def work(case):
    """Every text byte read once and every output written once: 4 bytes of id a
    position (dense), or 8 bytes a match -- about the copied windows' 4,096 with
    ACGT text, one position in 500 with Zipf text."""
    kind = case["kind"]
    if kind == "batch":
        total = case["texts"] * _mean_length(KIB, case["longest"])
        return {"bytes": float(5 * total), "flops": 0.0}
    if kind == "serve":
        total = case["requests"] * _mean_length(256, case["longest"])
        return {"bytes": float(total + 8 * total / 64), "flops": 0.0}
    n = case["n"]
    if kind == "host" or case["out"] == "dense":
        return {"bytes": float(5 * n), "flops": 0.0}
    if case["out"] == "count":
        return {"bytes": float(n + 8), "flops": 0.0}
    matches = n / 500 if case["set"] == "zipf" else n / 26 if case["set"] == "paper" else min(n, 4_096)
    return {"bytes": float(n + 8 * matches), "flops": 0.0}
