"""The forms a single text takes with the tuning left as built, against the
oracle, where they can go wrong: the short-text form (one thread per position,
up to 2 MiB) at warp and CTA edges, the streaming form (tiles of 2,048
positions, longer texts) at tile edges, texts and outputs off 16-byte
boundaries, every filter it can have, bytes in no keyword, and texts with more
walks than the walk list holds."""
import numpy as np
import pytest

import oracle
from paper_1412_7789_gb300 import api, workloads
from tests import _gpu

pytestmark = pytest.mark.gpu

AT_MAX = 2 << 20  # the short-text form's longest text


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1412_7789_gb300 import build

    build.build()
    api.lib()
    yield
    assert api.ac_device_status() == api.AC_OK


def _letters(n, alphabet, seed):
    a = np.frombuffer(alphabet, dtype=np.uint8)
    return a[workloads.rng(seed).integers(0, a.size, size=n)]


def _cut(text, seed, count, lmin, lmax):
    """Half copied from the text, half random over its letters."""
    r = workloads.rng(seed)
    out = []
    for i in range(count):
        m = int(r.integers(lmin, lmax + 1))
        if i % 2:
            at = int(r.integers(0, text.size - m))
            out.append(bytes(text[at:at + m]))
        else:
            out.append(bytes(r.permutation(text[:4 * m])[:m]))
    return out


# name: (alphabet, keywords, shortest, longest)
SETS = {
    "dna16": (b"ACGT", 600, 16, 40),    # every 4th position looked up, a second filter
    "dna8": (b"ACGT", 300, 8, 32),      # every 2nd
    "dna4": (b"ACGT", 200, 4, 40),      # every one
    "dna4dense": (b"ACGT", 1500, 4, 12),  # a third of the positions match
    "dna4lines": (b"ACGT", 1500, 4, 12),  # ... with a line break after every 60
    "dna1": (b"ACGT", 60, 1, 30),       # keywords shorter than any window
    "iupac": (b"ACGTNRYKM", 200, 6, 20),  # 4-bit codes: no streaming form
    "bytes4": (bytes(range(256)), 4000, 4, 30),
    "bytes5": (bytes(range(256)), 4000, 5, 30),
    "bytes9": (bytes(range(256)), 4000, 9, 30),
    "bytes2": (bytes(range(256)), 3000, 2, 12),  # keywords shorter than the hashed window
    "words4": (b"abcdefghijklmnopqrstuvwxyz ", 400, 4, 12),  # classes, not bytes
    "words7": (b"abcdefghijklmnopqrstuvwxyz ", 400, 7, 20),
}


def _workload(name, n):
    alphabet, count, lmin, lmax = SETS[name]
    if len(alphabet) == 256:
        text = workloads.zipf_text(n, 11)
    else:
        text = _letters(n, alphabet, 11)
    pats = _cut(text, 12, count, lmin, lmax)
    text = text.copy()
    if len(alphabet) < 256:  # bytes in no keyword, alone and in a run
        r = workloads.rng(13)
        text[r.integers(0, n, size=n // 500 + 1)] = ord("#")
        text[n // 3:n // 3 + 40] = ord("#")
    if name.endswith("lines"):
        text[60::61] = ord("\n")
    return text, pats


def _check(a, text, want, shift, out_shift):
    import torch

    n = text.size
    buf = torch.zeros(n + shift, dtype=torch.uint8, device="cuda")
    buf[shift:] = torch.from_numpy(text)
    t = buf[shift:]
    out = torch.full((n + out_shift + 8,), -7, dtype=torch.int32, device="cuda")
    api.ac_match(a.handle, t, n, out[out_shift:])
    got = out.cpu().numpy()
    assert np.array_equal(got[out_shift:out_shift + n], want)
    assert (got[:out_shift] == -7).all() and (got[out_shift + n:] == -7).all()  # nothing beside it
    _gpu.check_all_modes(a.handle, text, want, t=t, modes=("count", "compact"))


@pytest.mark.parametrize("name", sorted(SETS))
def test_short_texts(name):
    text, pats = _workload(name, 5000)
    with api.Automaton(pats) as a:
        for n in (1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 127, 128, 129, 2047, 2048, 2049, 5000):
            want = oracle.pfac_ids(pats, text[:n])
            for shift in (0, 7):
                _check(a, text[:n], want, shift, 0)


@pytest.mark.parametrize("name", sorted(SETS))
def test_streaming_edges(name):
    """Lengths on both sides of the short-text limit and of tile edges, text
    and output at several offsets from a 16-byte boundary."""
    top = AT_MAX + 6144
    text, pats = _workload(name, top)
    want_all = oracle.pfac_ids(pats, text)
    longest = max(len(p) for p in pats)
    with api.Automaton(pats) as a:
        for n, shift, out_shift in ((AT_MAX, 0, 0), (AT_MAX + 1, 0, 0), (AT_MAX + 2047, 1, 0), (AT_MAX + 2048, 0, 1),
                                    (AT_MAX + 2049, 15, 3), (AT_MAX + 4096 + 13, 3, 2), (top, 8, 0)):
            want = want_all[:n].copy()
            tail = max(0, n - longest)  # a keyword may not reach past n
            want[tail:] = oracle.pfac_ids(pats, text[tail:n])
            _check(a, text[:n], want, shift, out_shift)


@pytest.mark.parametrize("name", ["dna16", "dna8", "dna4", "dna4lines", "bytes4", "bytes9", "words7"])
def test_full_list(name):
    for n in (3000, AT_MAX + 777):
        text, pats = _workload(name, n)
        ends, ids = oracle.full_occurrences(pats, text)
        import torch

        cap = len(ends) + 1
        t = torch.from_numpy(text).cuda()
        with api.Automaton(pats) as a:
            e, i, c = a.match_full(t, cap=cap)
        assert int(c.item()) == len(ends)
        got = np.stack([e.cpu().numpy()[:len(ends)], i.cpu().numpy()[:len(ends)]], axis=1)
        want = np.stack([np.asarray(ends), np.asarray(ids)], axis=1).astype(got.dtype)
        assert np.array_equal(got[np.lexsort((got[:, 1], got[:, 0]))], want[np.lexsort((want[:, 1], want[:, 0]))])


def test_full_list_of_many_dense_tiles():
    """160 MiB in which every tile has more than 256 matches: more such tiles a
    CTA than it notes (64), so that some are done by the CTA and some by a warp.
    The text repeats 16 letters, so the list follows from their period."""
    import torch

    unit, n = b"ACGTTGCAACCGGTTA", 160 << 20
    pats = [unit[:4], unit[:8], unit[5:9], unit[9:13], (unit * 2)[14:19], unit[5:9]]
    starts = [(o, len(p), i) for o in range(16) for i, p in enumerate(pats) if (unit * 3)[o:o + len(p)] == p]
    starts.sort()
    assert 16 // 8 < len({o for o, _, _ in starts}) and len(starts) >= 6
    text = torch.tensor(list(unit), dtype=torch.uint8, device="cuda").repeat(n // 16)
    first = torch.arange(0, n, 16, dtype=torch.int64, device="cuda")
    ends = (first[:, None] + torch.tensor([o + m - 1 for o, m, _ in starts], device="cuda")[None, :]).flatten()
    ids = torch.tensor([i for _, _, i in starts], dtype=torch.int32, device="cuda").repeat(n // 16)
    inside = ends < n
    ends, ids = ends[inside].int(), ids[inside]
    with api.Automaton(pats) as a:
        e, i, c = a.match_full(text, cap=ends.numel())
        assert int(c.item()) == ends.numel()
        assert bool((e.int() == ends).all()) and bool((i.int() == ids).all())


def test_full_counts_past_32_bits():
    """2^21 equal keywords: a tile of 2,048 of their matches holds 2^32
    occurrences, which only units of half a tile can count in 32 bits."""
    import torch

    copies, run = 1 << 21, 2 * 2048 + 100
    pats = [b"A"] * copies + [b"CGTCGTCCGGTTCC"]
    with api.Automaton(pats) as a:
        for n in (run, AT_MAX + 4096):
            text = _letters(n, b"CGT", 17).copy()
            at = (n - run) // 2  # the matches: one run, two whole tiles of it at least at most offsets
            text[at:at + run] = ord("A")
            other = text.tobytes().count(pats[-1])
            cap = 4
            t = torch.from_numpy(text).cuda()
            e, i, c = a.match_full(t, cap=cap)
            assert int(c.item()) == run * copies + other
            if not other:  # the first start's occurrences come first, ids ascending
                assert e.cpu().tolist() == [at] * cap and i.cpu().tolist() == list(range(cap))


@pytest.mark.parametrize("letters,lens", [(b"A", (16, 20, 60)), (b"A", (4, 33)), (b"x", (6, 9, 40)), (b"x", (4, 50))])
def test_more_walks_than_listed(letters, lens):
    """A text of one letter: every position is a survivor and a long walk, far
    more than the walk list holds; the rest are settled where they are found."""
    n = AT_MAX + 3000
    text = np.full(n, letters[0], dtype=np.uint8)
    text[5000] = ord("C") if letters == b"A" else ord("y")
    others = [b"ACGT" * 10, b"TTGACCA" * 3] if letters == b"A" else [bytes(range(40, 120)), b"xyzw" * 3]
    pats = [letters * m for m in lens] + others
    want = oracle.pfac_ids(pats, text)
    assert (want >= 0).sum() > n // 2
    with api.Automaton(pats) as a:
        _check(a, text, want, 3, 0)


def _event_us(f):
    """Median of five timings of three calls."""
    import torch

    f()
    torch.cuda.synchronize()
    out = []
    for _ in range(5):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        for _ in range(3):
            f()
        t1.record()
        torch.cuda.synchronize()
        out.append(t0.elapsed_time(t1) * 1000 / 3)
    return sorted(out)[2]


@pytest.mark.parametrize("kind,block", [("one letter", 640), ("repeat of 1009", 640), ("one byte", 512), ("phrase", 512)])
def test_repetitive_texts_are_no_slower(kind, block):
    """Texts where most positions walk far: as built, dense ids take no longer
    than in the filter kernel with its own best block (a quarter more allowed
    for the spread of the timings)."""
    import torch

    n = 8 << 20
    if kind == "one letter":
        unit, pats = b"A", [b"A" * m for m in (16, 20, 60)] + [b"ACGT" * 10, b"TTGACCA" * 3]
    elif kind == "repeat of 1009":
        unit = bytes(_letters(1009, b"ACGT", 6))
        at = workloads.rng(2).integers(0, 1009, size=500)
        lens = workloads.rng(3).integers(16, 65, size=500)
        pats = [(unit * 2)[o:o + m] for o, m in zip(at.tolist(), lens.tolist())]
    elif kind == "one byte":
        unit, pats = b"x", [b"x" * m for m in (6, 9, 40)] + [bytes(range(40, 120)), b"xyzw" * 3]
    else:
        unit = b"the quick brown fox jumps over the lazy dog while the cat sleeps in the sun. "
        at = workloads.rng(4).integers(0, len(unit), size=200)
        lens = workloads.rng(5).integers(4, 41, size=200)
        pats = [(unit * 2)[o:o + m] for o, m in zip(at.tolist(), lens.tolist())]
    text = torch.from_numpy(np.tile(np.frombuffer(unit, dtype=np.uint8), n // len(unit) + 1)[:n].copy()).cuda()
    ids = torch.empty(n, dtype=torch.int32, device="cuda")
    with api.Automaton(pats) as a, api.Automaton(pats) as b:
        b.set_tuning(block=block)
        built, tuned = _event_us(lambda: a.match(text, out=ids)), _event_us(lambda: b.match(text, out=ids))
    assert built <= 1.25 * tuned, (built, tuned)


@pytest.mark.parametrize("kind", ["alphabet", "words"])
def test_short_texts_with_scattered_walks(kind):
    """Byte texts of 1.5 MiB where a lane or two of every warp walk: dense ids
    take no longer as built than in the filter kernel (a quarter more allowed,
    as above), and every output is right."""
    import torch

    n = (3 << 19) + 77
    if kind == "alphabet":
        text, pats = workloads.paper_text(n), workloads.paper_keywords(10, 0)
    else:
        r = workloads.rng(31)
        pats = [bytes(r.integers(97, 123, size=int(m)).astype(np.uint8)) for m in r.integers(4, 12, size=2000)]
        text = np.frombuffer(b" ".join(pats[min(1999, int(x))] for x in r.zipf(1.3, size=n // 5)), dtype=np.uint8)[:n].copy()
        assert text.size == n
    t = torch.from_numpy(text).cuda()
    ids = torch.empty(n, dtype=torch.int32, device="cuda")
    with api.Automaton(pats) as a, api.Automaton(pats) as b:
        _check(a, text, oracle.pfac_ids(pats, text), 5, 1)
        b.set_tuning(block=512)
        built, tuned = _event_us(lambda: a.match(t, out=ids)), _event_us(lambda: b.match(t, out=ids))
    assert built <= 1.25 * tuned, (built, tuned)


@pytest.mark.parametrize("letters,shortest", [(b"ACGT", 16), (b"ACGT", 8), (b"ACGT", 4),
                                              (b"abcdefghijklmnopqrstuvwxyz", 6)])
def test_walks_fill_the_list_part_way(letters, shortest):
    """A repeat of 40 letters where a run of 12 starts walks 26 letters or more:
    few enough for a tile to be resolved in its warp, and more walks than the
    list holds, so that later tiles are listed whole (dense ids, count and the
    compacted list; the last tile ends inside the text)."""
    n = (12 << 20) + 1234
    unit = bytes(_letters(40, letters, 21))
    text = np.tile(np.frombuffer(unit, dtype=np.uint8), n // 40 + 1)[:n].copy()
    text[(3 << 20):(3 << 20) + 3000] = ord("#")
    pats = [(unit * 3)[o:o + 26 + o] for o in range(12)] + [b"".join(bytes([letters[(i * j) % 4]]) for i in range(shortest))
                                                         for j in range(1, 4)]
    want = oracle.pfac_ids(pats, text)
    assert n // 5 < (want >= 0).sum() < n // 2
    with api.Automaton(pats) as a:
        assert a.info()["min_len"] == shortest
        _check(a, text, want, 5, 1)


def test_list_capacity_is_kept():
    """A compacted list longer than its capacity: the first entries and the
    whole count, and nothing written past the capacity."""
    import torch

    for n in (4096, AT_MAX + 4096):
        text, pats = _workload("dna4", n)
        wpos, wids = oracle.compact(oracle.pfac_ids(pats, text))
        t = torch.from_numpy(text).cuda()
        with api.Automaton(pats) as a:
            for cap in (0, 1, wpos.size // 2):
                pos = torch.full((wpos.size,), -7, dtype=torch.int32, device="cuda")
                ids = torch.full((wpos.size,), -7, dtype=torch.int32, device="cuda")
                c = torch.zeros(1, dtype=torch.int64, device="cuda")
                api.ac_match_compact(a.handle, t, n, pos, ids, cap, c)
                assert int(c.item()) == wpos.size
                assert np.array_equal(pos[:cap].cpu().numpy(), wpos[:cap])
                assert np.array_equal(ids[:cap].cpu().numpy(), wids[:cap])
                assert bool((pos[cap:] == -7).all()) and bool((ids[cap:] == -7).all())


@pytest.mark.parametrize("names", [("dna16", "bytes4"), ("dna8", "dna4", "dna4lines", "bytes9", "words7"),
                                   ("dna16", "iupac", "bytes2", "bytes5", "dna1")])
@pytest.mark.parametrize("reserve", [1 << 22, 64])
def test_batch_streams(names, reserve):
    """A plan with lists: automata the streaming form serves, next to ones it
    does not; texts from 1 byte to several tiles, packed back to back (most
    start off a 16-byte boundary), some empty; also with a walk list too small
    for the batch."""
    import torch

    r = workloads.rng(len(names))
    lens = [0, 1, 2, 15, 17, 2047, 2048, 2049, 4096 + 5, 70_000] + [int(x) for x in r.integers(1, 12_000, size=30)]
    which = [int(x) for x in r.integers(0, len(names), size=len(lens))]
    which[9] = 0
    loads = [_workload(n, 80_000) for n in names]
    texts = [loads[a][0][s:s + n] for a, n, s in zip(which, lens, r.integers(0, 5_000, size=len(lens)))]
    offs = np.concatenate([[0], np.cumsum(lens)[:-1]]) + 3
    total = int(sum(lens)) + 3
    buf = np.zeros(total, dtype=np.uint8)
    for t, o in zip(texts, offs):
        buf[o:o + t.size] = t
    autos = [api.Automaton(p) for _, p in loads]
    try:
        d = torch.from_numpy(buf).cuda()
        out = torch.full((total + 8,), -7, dtype=torch.int32, device="cuda")
        items = api.items_to_device(api.batch_items(offs, lens, offs + 1, which))
        with api.BatchPlan([a.handle for a in autos], len(lens)) as plan:
            plan.reserve_lists(reserve)
            for run in range(2):
                out.fill_(-7)
                if run == 0:
                    plan.run(d, items, len(lens), out)
                else:
                    plan.capture(d, items, len(lens), out)
                    plan.replay()
                got = out.cpu().numpy()
                want = np.full(total + 8, -7, dtype=np.int32)
                for t, o, a in zip(texts, offs, which):
                    if t.size:
                        want[o + 1:o + 1 + t.size] = oracle.pfac_ids(loads[a][1], t)
                assert np.array_equal(got, want)
    finally:
        for a in autos:
            a.close()


@pytest.mark.parametrize("reserve", [1 << 22, 1 << 13])
def test_batch_of_texts_dense_in_walks(reserve):
    """Texts of one letter in a plan with lists: tiles listed whole, and (the
    smaller plan) more of them than the tile list holds."""
    import torch

    lens = [300_001, 5, 2048, 700_003, 4096 + 7]
    sets = [[b"A" * m for m in (16, 20, 60)] + [b"ACGT" * 10], [b"A" * m for m in (4, 33)] + [b"ACGTTGCA" * 3],
            [b"x" * m for m in (6, 9, 40)] + [bytes(range(40, 120))]]
    which = [0, 1, 2, 2, 1, 0, 1, 2, 0, 1]
    lens = lens + lens
    offs = np.concatenate([[0], np.cumsum(lens)[:-1]]) + 1
    total = int(sum(lens)) + 1
    buf = np.zeros(total, dtype=np.uint8)
    for o, m, a in zip(offs, lens, which):
        buf[o:o + m] = sets[a][0][0]
        buf[o + m // 2] = ord("C") if a < 2 else ord("y")
    autos = [api.Automaton(p) for p in sets]
    try:
        out = torch.full((total,), -7, dtype=torch.int32, device="cuda")
        items = api.items_to_device(api.batch_items(offs, lens, offs, which))
        with api.BatchPlan([a.handle for a in autos], len(lens)) as plan:
            plan.reserve_lists(reserve)
            plan.run(torch.from_numpy(buf).cuda(), items, len(lens), out)
        got = out.cpu().numpy()
        for o, m, a in zip(offs, lens, which):
            assert np.array_equal(got[o:o + m], oracle.pfac_ids(sets[a], buf[o:o + m]))
    finally:
        for a in autos:
            a.close()


def _tables(autos):
    return sum(a.info()["table_bytes"] for a in autos)


def test_request_charge_is_kept():
    """What a request is charged does not depend on the form its wave takes:
    text, output and the slot form's scratch per tile of 992 positions.  A
    budget of exactly that serves it, one byte less refuses it."""
    import torch

    n, cap = (6 << 20) + 1, 4096
    text, pats = _workload("dna16", n)
    wpos, wids = oracle.compact(oracle.pfac_ids(pats, text))
    assert wpos.size <= cap
    d = torch.from_numpy(text).cuda()
    pos = torch.full((cap,), -7, dtype=torch.int32, device="cuda")
    ids = torch.full((cap,), -7, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    req = np.zeros(1, dtype=api.SERVER_REQUEST)
    for f, v in (("d_text", d.data_ptr()), ("n", n), ("d_pos", pos.data_ptr()), ("d_ids", ids.data_ptr()),
                 ("cap", cap), ("d_count", cnt.data_ptr())):
        req[f] = v
    charge = n + 8 * cap + -(-n // 992) * (4 + 8 + 8 * 32 + 4 * 1024) + 64
    with api.Automaton(pats) as a:
        with api.Server([a.handle], hbm_budget=_tables([a]) + charge - 1) as srv:
            with pytest.raises(api.AcError) as e:
                srv.submit(req)
            assert e.value.status == api.AC_ERR_BUDGET
        with api.Server([a.handle], hbm_budget=_tables([a]) + charge) as srv:
            srv.submit(req)
            srv.drain()
            assert srv.poll(4)["status"].tolist() == [api.AC_OK]
    m = int(cnt.item())
    assert m == wpos.size
    assert np.array_equal(pos[:m].cpu().numpy(), wpos) and np.array_equal(ids[:m].cpu().numpy(), wids)


@pytest.mark.parametrize("names,lens", [
    (("dna16",), [(0, (4 << 20) + 5)]),
    (("dna4", "dna16"), [(0, 3_000_000), (1, 5_000_001), (0, 777), (1, 2047)]),
    (("bytes5", "dna8"), [(0, 3_000_000), (1, 4_000_001), (1, 1)]),
    (("iupac", "dna16"), [(0, 5 << 20), (1, 40)]),  # 40 bytes of it for the streaming form
])
def test_wave_scratch_is_charged(names, lens):
    """The device scratch of a wave stays within what its requests were charged
    for their tiles (and lists), the wave's plan (a head and a counter an
    automaton, 64 bytes a request, the scan's 256 partial sums) and a kilobyte
    of rounding for each of its parts; every request is served."""
    import torch

    loads = [_workload(name, 5 << 20) for name in names]
    blocks = {}

    def alloc(nbytes):
        t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        blocks[t.data_ptr()] = t
        sizes.append(nbytes)
        return t.data_ptr()

    sizes, reqs, outs, charge = [], [], [], 0
    autos = [api.Automaton(p) for _, p in loads]
    try:
        for a, n in lens:
            text = loads[a][0][:n]
            d = torch.from_numpy(text.copy()).cuda()
            want = oracle.compact(oracle.pfac_ids(loads[a][1], text))
            cap = max(1, want[0].size)
            pos = torch.full((cap,), -7, dtype=torch.int32, device="cuda")
            ids = torch.full((cap,), -7, dtype=torch.int32, device="cuda")
            cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
            reqs.append(api.Server.request(a, d, n, pos, ids, cap, cnt))
            outs.append((d, pos, ids, cnt, want))
            charge += -(-n // 992) * (4 + 8 + 8 * 32 + 4 * 1024) + 64
            if autos[a].info()["code_bits"] == 8:
                charge += 32 * (n // 8) + 32
        torch.cuda.synchronize()
        with api.Server([a.handle for a in autos], waves_in_flight=1, dev_alloc=alloc,
                        dev_free=lambda p: blocks.pop(p)) as srv:
            srv.replay(np.concatenate(reqs), np.zeros(len(reqs)))
            srv.drain()
            done = srv.poll(len(reqs) + 1)
            assert done["status"].tolist() == [api.AC_OK] * len(reqs)
            waves = len(sizes)
        assert waves and not blocks
        assert sum(sizes) <= charge + waves * (32 * len(autos) + 8 * 256 + 12 * 1024), (sizes, charge)
        for _, pos, ids, cnt, (wpos, wids) in outs:
            m = int(cnt.item())
            assert m == wpos.size
            assert np.array_equal(pos[:m].cpu().numpy(), wpos) and np.array_equal(ids[:m].cpu().numpy(), wids)
    finally:
        for a in autos:
            a.close()


def test_wave_past_32_bits_of_text():
    """Waves that hold more text than 32 bits can number: every request is
    served, each as ac_match_compact alone."""
    import torch

    n, cap, k = 1 << 30, 1 << 16, 8
    letters = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")
    torch.manual_seed(5)
    d = letters[torch.randint(0, 4, (n,), dtype=torch.uint8, device="cuda").int()]
    _, pats = _workload("dna16", 100_000)
    pats = pats + [bytes(d[x:x + 20].cpu().numpy()) for x in range(0, n - 64, n // 40)]
    new = lambda: (torch.full((cap,), -7, dtype=torch.int32, device="cuda"),
                   torch.full((cap,), -7, dtype=torch.int32, device="cuda"),
                   torch.zeros(1, dtype=torch.int64, device="cuda"))
    with api.Automaton(pats) as a:
        wpos, wids, wcnt = new()
        api.ac_match_compact(a.handle, d, n, wpos, wids, cap, wcnt)
        assert 0 < int(wcnt.item()) <= cap
        bufs = [new() for _ in range(k)]
        torch.cuda.synchronize()
        with api.Server([a.handle], hbm_budget=64 << 30, waves_in_flight=1) as srv:
            for pos, ids, cnt in bufs:
                req = np.zeros(1, dtype=api.SERVER_REQUEST)
                for f, v in (("d_text", d.data_ptr()), ("n", n), ("d_pos", pos.data_ptr()),
                             ("d_ids", ids.data_ptr()), ("cap", cap), ("d_count", cnt.data_ptr())):
                    req[f] = v
                srv.submit(req)
            srv.drain()
            assert srv.poll(2 * k)["status"].tolist() == [api.AC_OK] * k
        for pos, ids, cnt in bufs:
            assert int(cnt.item()) == int(wcnt.item())
            assert bool((pos == wpos).all()) and bool((ids == wids).all())


@pytest.mark.parametrize("kind", ["dense", "count", "compact"])
def test_scratch_of_dna_texts(kind):
    """2-bit codes: lists of half a byte per text byte (8 bytes for every
    sixteenth, with a bit and an id a position for the compacted list: 4.7 in
    all) and a few MB; in a captured graph, whose memory no other form could do
    without, no more for the lists than those few MB."""
    import torch

    n, few = 128 << 20, 8 << 20
    text = _letters(n, b"ACGT", 9)
    pats = [bytes(text[x:x + 20]) for x in range(1000, n - 64, n // 300)]
    t = torch.from_numpy(text).cuda()
    m = n if kind == "dense" else 4096
    out, ids = torch.empty(m, dtype=torch.int32, device="cuda"), torch.empty(4096, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    per_byte = 4 * (1 + 1 / 32) + 12 / 2048 if kind == "compact" else 0

    def call(a, stream=None, n=n):
        if kind == "dense":
            api.ac_match(a.handle, t, n, out, stream)
        elif kind == "count":
            api.ac_count(a.handle, t, n, cnt, stream)
        else:
            api.ac_match_compact(a.handle, t, n, out, ids, 4096, cnt, stream)

    def captured(a, n):
        g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(g, stream=side):
            call(a, side, n)
        g.replay()
        torch.cuda.synchronize()
        return g

    def check():
        torch.cuda.synchronize()
        if kind == "dense":
            at = torch.nonzero(out >= 0).flatten()
            assert int((out < -1).sum()) == 0 and out[at].tolist() == list(range(len(pats)))
        else:
            assert int(cnt.item()) == len(pats)
            at = out[:len(pats)].long() if kind == "compact" else None
        if at is not None:
            assert at.tolist() == list(range(1000, n - 64, n // 300))

    with api.Automaton(pats) as a:
        call(a)  # code loaded
        torch.cuda.synchronize()
        base, _ = api.ac_scratch_pool_usage(reset_high=True)
        call(a)
        check()
        assert api.ac_scratch_pool_usage()[1] - base <= (per_byte + 0.5) * n + few
        captured(a, AT_MAX + 1)  # what a process's first graph takes
        out.fill_(-7)
        cnt.zero_()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()  # as the capture will
        free, _ = torch.cuda.mem_get_info()
        g = captured(a, n)
        taken = free - torch.cuda.mem_get_info()[0]
        check()
        assert taken <= per_byte * n + (64 << 20)  # (mapped in pieces of up to 32 MB)
        del g


_NO_ROOM = """
import sys
import numpy as np
import torch
from paper_1412_7789_gb300 import api, workloads
kind, free_mib = sys.argv[1], int(sys.argv[2])
n = 128 << 20
text = np.frombuffer(b"ACGT", dtype=np.uint8)[workloads.rng(9).integers(0, 4, size=n)]
pats = [bytes(text[x:x + 20]) for x in range(1000, n - 64, n // 300)]
t = torch.from_numpy(text).cuda()
out = torch.full((n if kind == "dense" else 4096,), -7, dtype=torch.int32, device="cuda")
ids = torch.full((4096,), -7, dtype=torch.int32, device="cuda")
cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
def call(a, m):
    if kind == "dense":
        api.ac_match(a.handle, t, m, out)
    else:
        api.ac_match_compact(a.handle, t, m, out, ids, 4096, cnt)
    torch.cuda.synchronize()
with api.Automaton(pats) as a, api.Automaton(pats) as b:
    b.set_tuning(block=256)  # the filter kernel: its code is loaded before the memory goes
    call(b, 1 << 20)
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - (free_mib << 20), dtype=torch.uint8, device="cuda")
    call(a, n)
    del hold
if kind == "dense":
    pos = torch.nonzero(out >= 0).flatten()
    assert int((out < -1).sum()) == 0
    val = out[pos]
else:
    pos, val = out[:int(cnt.item())], ids[:int(cnt.item())]
at = list(range(1000, n - 64, n // 300))
assert pos.tolist() == at and val.tolist() == list(range(len(pats)))
assert api.ac_device_status() == api.AC_OK
"""


@pytest.mark.parametrize("kind,free_mib", [("dense", 40), ("compact", 600)])
def test_no_room_for_the_streaming_scratch(kind, free_mib):
    """Where the device has no room for the walk list (about a byte per text
    byte) or the bits and ids (5.2 bytes), the call takes the form that needs
    less (16 bytes; 4.4 per text byte) and still succeeds."""
    import os
    import subprocess
    import sys

    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _NO_ROOM, kind, str(free_mib)], cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("name", ["dna16", "dna4", "iupac", "bytes4"])
@pytest.mark.parametrize("part", [4, 16])
def test_other_table_depths(name, part):
    """Root tables rebuilt for a smaller filter: the short-text form reads them
    at the new window, longer texts leave the streaming form."""
    for n in (5001, AT_MAX + 5001):
        text, pats = _workload(name, n)
        want = oracle.pfac_ids(pats, text)
        with api.Automaton(pats) as a:
            a.set_tuning(filter_bytes=max(4, a.tuning()["filter_bytes"] // part))
            _check(a, text, want, 3, 0)
