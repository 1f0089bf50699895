"""Rules and tables on the host that no entry point shows, through a small
program linked against the library (no GPU needed)."""
import os
import subprocess

import numpy as np
import pytest

from paper_1412_7789_gb300 import build, workloads


def compile_cpp(directory, source: str) -> str:
    """A program compiled against the internal header and the library."""
    lib = build.build()
    src, exe = directory / "prog.cpp", directory / "prog"
    src.write_text(source)
    subprocess.run([build._nvcc(), "-O1", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o", str(exe),
                    lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True)
    return str(exe)


def output(*command: str) -> str:
    return subprocess.run(command, capture_output=True, text=True, check=True).stdout


def test_full_counts_fit_32_bits(tmp_path):
    """Full output goes tile by tile (2,048 results) while 2,048 results with
    the set's longest chain fit 32 bits, by half tiles while 1,024 do."""
    out = output(compile_cpp(tmp_path, r'''
#include <cstdio>
#include "pfac_internal.h"
int main() {
    for (unsigned c : {1u, (1u << 21) - 1, 1u << 21, (1u << 22) - 1, 1u << 22, 0xFFFFFFFFu})
        std::printf("%d%d ", pfac::full_fits(c, pfac::kStreamTile), pfac::full_fits(c, pfac::kDenseStride));
}'''))
    assert out.split() == ["11", "11", "01", "01", "00", "00"]


_FILTERS = r'''
#include <cstdio>
#include <cstring>
#include <string>
#include "pfac_internal.h"
int main(int argc, char **argv) {  // keywords in hex
    std::vector<std::string> p;
    for (int i = 1; i < argc; ++i) {
        std::string s;
        for (const char *c = argv[i]; *c; c += 2) { unsigned v; std::sscanf(c, "%2x", &v); s += static_cast<char>(v); }
        p.push_back(s);
    }
    std::vector<const uint8_t *> ps;
    std::vector<uint32_t> ls;
    for (auto &s : p) { ps.push_back(reinterpret_cast<const uint8_t *>(s.data())); ls.push_back(static_cast<uint32_t>(s.size())); }
    pfac::HostTables h;
    if (pfac::build_tables(ps.data(), ls.data(), static_cast<uint32_t>(p.size()), pfac::BuildOptions(), &h) != 0) return 1;
    const pfac::StreamTables &t = h.stream;
    const std::vector<uint32_t> &F1 = h.stream_F1.empty() ? h.F : h.stream_F1;
    std::printf("%u %u %u %u %u %u\n", t.form, t.step, h.k, t.win2, t.m1, t.m2);
    for (uint32_t w : F1) std::printf("%x ", w);
    std::printf("\n");
    for (uint32_t w : h.stream_F2) std::printf("%x ", w);
    std::printf("\n");
}'''

_MASK = (1 << 32) - 1
_MUL, _STATE_MUL, _MUL2, _SHORT = 0x9E3779B1, 0x85EBCA77, 0xC2B2AE35, 4096


def _word(b, o):
    return int.from_bytes(b[o:o + 4].ljust(4, b"\0"), "little")


# name: (alphabet, keywords, shortest, longest, form, step)
_FILTER_SETS = {
    "dna16": (b"ACGT", 300, 16, 40, 2, 4),
    "dna8": (b"ACGT", 1500, 8, 32, 2, None),
    "dna4": (b"ACGT", 200, 4, 20, 2, 1),
    "bytes4": (bytes(range(256)), 1500, 4, 30, 8, 1),
    "bytes5": (bytes(range(256)), 1500, 5, 12, 8, 1),
    "bytes9": (bytes(range(256)), 1500, 9, 30, 8, 1),
    "words4": (b"abcdefghijklmnopqrstuvwxyz ", 400, 4, 12, 8, 1),
    "iupac": (b"ACGTNRYKM", 100, 6, 20, 0, None),
    "bytes2": (bytes(range(256)), 300, 2, 12, 0, None),
}


@pytest.fixture(scope="module")
def filters(tmp_path_factory):
    return compile_cpp(tmp_path_factory.mktemp("filters"), _FILTERS)


@pytest.mark.parametrize("name", sorted(_FILTER_SETS))
def test_streaming_filters_hold_every_keyword(name, filters):
    """Looked up as the kernels do, the streaming form's filters pass every
    keyword at every offset at which it may be sampled, whatever bytes follow
    it; and they have no more bits than those windows (with the completions of
    the keywords that end inside one)."""
    alphabet, count, lmin, lmax, form, step = _FILTER_SETS[name]
    a, r = np.frombuffer(alphabet, dtype=np.uint8), workloads.rng(41)
    pats = sorted({bytes(a[r.integers(0, a.size, size=int(m))]) for m in r.integers(lmin, lmax + 1, size=count)} |
                  {bytes(a[r.integers(0, a.size, size=lmin)])})
    out = output(filters, *[p.hex() for p in pats]).split("\n")
    got_form, S, k, win2, m1, m2 = (int(x) for x in out[0].split())
    F1, F2 = ([int(x, 16) for x in line.split()] for line in out[1:3])
    assert got_form == form
    if form == 0:
        return
    assert len(F1) == 1 << 15 and (step is None or S == step)
    tails = [bytes(a[r.integers(0, a.size, size=24)]) for _ in range(4)] + [bytes(24), b"\xff" * 24]
    bits = 0
    if form == 2:
        codes = lambda b, m: sum(((c >> 1) & 3) << (2 * j) for j, c in enumerate(b[:m]))
        for p in pats:
            for o in range(S):
                bits += 4 ** (k - min(k, len(p) - o))
                for t in tails:
                    b = (p + t)[o:]
                    w = codes(b, k)
                    assert (F1[w >> 5] >> (31 - (w & 31))) & 1
                    if F2:
                        x = (codes(b, 16) << (32 - 2 * win2) & _MASK) * _MUL & _MASK
                        assert (F2[x * len(F2) >> 32] >> ((x >> 12) & 31)) & 1
        if F2:
            assert sum(bin(w).count("1") for w in F2) <= len(pats) * S
    else:
        words2 = len(F2) - _SHORT // 4
        win = 32 if m2 == 0 else 65 - (m2 & -m2).bit_length()  # bits of the window: m2 is odd << (64 - win)
        for p in pats:
            bits += 2 ** max(0, win - 8 * len(p))
            for t in tails:
                b = p + t
                w0, w1 = _word(b, 0), _word(b, 4)
                h = w0 * m1
                i = ((h + w1 * m2) & _MASK) >> 17
                assert (F1[i] >> (31 - ((h >> 32) & 31))) & 1
                if F2:
                    hs, h6 = w0 * _STATE_MUL & _MASK, (w0 * _MUL + (w1 << 16 & _MASK) * _MUL2) & _MASK
                    short = F2[words2 + (hs >> 22)] >> ((hs >> 17) & 31)
                    six = F2[h6 * words2 >> 32] >> ((h6 >> 12) & 31)
                    assert (short | six) & 1
        if F2:
            assert sum(bin(w).count("1") for w in F2) <= len(pats)
    assert sum(bin(w).count("1") for w in F1) <= bits
