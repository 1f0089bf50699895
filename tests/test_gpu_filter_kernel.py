"""The filter kernel, which every tuning but the one as built keeps (and a call
for whose other forms' scratch there is no room): the sizes, alphabets and
outputs that single texts take elsewhere as built -- ragged ends, unaligned
texts, tiles dense in matches, slots and the dense fallback, full output, the
largest text that needs no tile counter -- against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1412_7789_gb300 import api, workloads
from tests import _gpu
from tests.test_gpu_full import SIZES as FULL_SIZES
from tests.test_gpu_full import check as check_full
from tests.test_gpu_full import nested, planted_text
from tests.test_gpu_parity import ALPHABETS, SIZES, random_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1412_7789_gb300 import build

    build.build()
    api.lib()
    yield
    assert api.ac_device_status() == api.AC_OK


@pytest.mark.parametrize("tuning", [{"block": 512}, {"survivor_list": 2}], ids=["block", "list"])
@pytest.mark.parametrize("alpha", sorted(ALPHABETS))
def test_random_sizes(alpha, tuning):
    g = np.random.Generator(np.random.PCG64(sorted(ALPHABETS).index(alpha) + 2000))
    for n in SIZES:
        text, pats = random_case(g, ALPHABETS[alpha], max(n, 40), 50, 24)
        text = text[:n]
        want = oracle.pfac_ids(pats, text)
        with api.Automaton(pats) as a:
            a.set_tuning(**tuning)
            _gpu.check_all_modes(a.handle, text, want)
            if n > 20:
                t = _gpu.to_dev(text)
                _gpu.check_all_modes(a.handle, text[3:], oracle.pfac_ids(pats, text[3:]), t=t[3:])


@pytest.mark.parametrize("n", [4096, 65536, 1 << 20])
def test_sweep_keywords(n):
    """The first 4 KiB all match: heavy tiles, shared within the CTA."""
    text, pats = workloads.sweep_acgt(n)
    with api.Automaton(pats) as a:
        a.set_tuning(block=640)
        _gpu.check_all_modes(a.handle, text, oracle.pfac_ids(pats, text))


@pytest.mark.parametrize("alpha", ["acgt", "bytes"])
def test_tiles_dense_in_matches(alpha):
    """More matches a tile than slots: the list comes from the dense fallback."""
    g = np.random.Generator(np.random.PCG64(78))
    text, pats = random_case(g, ALPHABETS[alpha], 300_001, 60, 12)
    pats += [bytes([b]) for b in ALPHABETS[alpha][::3]]
    want = oracle.pfac_ids(pats, text)
    assert (want >= 0).mean() > 0.2
    with api.Automaton(pats) as a:
        a.set_tuning(block=512)
        _gpu.check_all_modes(a.handle, text, want)


@pytest.mark.parametrize("alpha", [b"ACGT", b"abcdefghijklmnopqrstuvwxyz"])
def test_counter_free_boundary(alpha):
    """Texts just below and above the largest whose tiles of 992 positions all go
    to the first claims of 16 warps an SM, launched without a tile counter."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = np.random.Generator(np.random.PCG64(len(alpha) + 9))
    a = np.frombuffer(alpha, dtype=np.uint8)
    edge = sms * 16 * 992
    base = a[g.integers(0, a.size, size=edge + 4096)]
    pats = [bytes(base[o:o + int(L)]) for o, L in zip(g.integers(0, 1 << 20, size=300), g.integers(3, 20, size=300))]
    with api.Automaton(pats) as h:
        h.set_tuning(block=512)
        for n in (edge - 4096, edge - 1, edge, edge + 1, edge + 4096):
            text = base[:n]
            _gpu.check_all_modes(h.handle, text, oracle.pfac_ids(pats, text), modes=("dense", "count"))


@pytest.mark.parametrize("alpha,kw", [(b"ACGT", {}), (b"abcdefghijkl", {}), (bytes(range(40, 120)), {}),
                                      (bytes(range(256)), {"class_compress": False})])
def test_full_output(alpha, kw):
    g = np.random.Generator(np.random.PCG64(len(alpha) * 11 + len(kw)))
    pats, stems = nested(g, alpha, 300, 40)
    with api.Automaton(pats, **kw) as a:
        a.set_tuning(block=512)
        for n in FULL_SIZES:
            text = planted_text(g, alpha, n + 5, stems)
            t = _gpu.to_dev(text)
            check_full(a.handle, pats, text[:n], t=t[:n])
            check_full(a.handle, pats, text[3:3 + n], t=t[3:3 + n])


def test_full_output_of_dense_tiles():
    """Every string of one to three letters is a keyword: every tile has more
    results than slots; also with room for some of the occurrences only."""
    import itertools

    pats = [bytes(p) for m in (1, 2, 3) for p in itertools.product(b"ACGT", repeat=m)]
    text = workloads.acgt_text(50_000, 5)
    with api.Automaton(pats) as a:
        a.set_tuning(block=512)
        check_full(a.handle, pats, text)
        check_full(a.handle, pats, text[7:7 + 30_001], cap=1000)
