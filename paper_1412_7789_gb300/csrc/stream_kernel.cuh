// The streaming form of the matching kernel for one long text, sm_103a, in two
// launches:
//   pfac_stream2 / pfac_stream8   read the text once, straight into registers,
//       test it against a root filter in shared memory, resolve the few
//       positions that pass with one or two table loads, write the -1 of every
//       other position, and list the walks that go further;
//   pfac_stream_walks             one thread per listed walk, and one lane per
//       position of the tiles left to it as a whole (list_tile).
//
// Text: a warp takes tiles of 2048 positions (lane l the 16 bytes at 16 l of
// each 512-byte chunk), with the next tile's loads issued as soon as a chunk's
// registers are free, so no shared-memory stage, barrier or work counter is
// needed: every tile costs about the same, because the walks are not done
// here, and the tiles are dealt out in a fixed order.
//
// What bounds it, and what it measured (GB300, 1 GiB of text): with 2-bit codes
// dense ids are bound by DRAM writes (0.875 ms, 0.90 of the copy peak; the
// filter kernel's own pass, 1,200 cycles of instructions a tile, took 1.065),
// counts by instruction issue (0.27 against 0.88 ms); with 8-bit codes both by
// the filter's lookups, 16 a lane and chunk, about 8 instructions each (count
// 0.85 against 2.15 ms, where every tenth position went through a global list).
//
// 2-bit codes (pfac_stream2).  Codes come from (byte >> 1) & 3, and bytes in no
// keyword get some code as well: the filter bit of a position with a result is
// set whatever codes follow the result's keyword (all completions of a keyword
// shorter than the window are set), so no position is lost, and only a
// survivor that would report something has its bytes checked.  With keywords
// long enough, only every S-th position is looked up (S = 2 or 4): the filter
// then holds the windows at offsets 0 .. S - 1 of every keyword, a set bit
// makes the S positions up to the sample candidates, and a second filter over
// longer windows drops most of the chance hits first.
//
// 8-bit codes (pfac_stream8).  Hashed windows of raw bytes: the shortest
// keyword's length (at most 8 bytes), and some bits of the next byte while the
// completions of the keywords that end before it are few.  With windows below
// 6 bytes the survivors are looked up again over 6 bytes, in a second filter
// that also knows the 4-byte windows of the keywords shorter than that.
#pragma once

#include <atomic>
#include <type_traits>

#include "filter_kernel.cuh"

namespace pfac {
namespace strm {

using filt::FilterParams;
using filt::kFull;

// Threads per CTA, one CTA per SM: what runs fastest without spills, which cost
// these loops more than the warps they buy.  GB300, 2-bit codes: 640 / 768
// threads, 256 MiB compacted 140 / 156 us, 1 GiB counted 286 / 325 (768 with no
// spill: 275); 8-bit codes, one text: 640 / 768, 1 GiB counted 930 / 919, dense
// 1074 / 1050, compacted 1164 / 1114; in a batch the kernel spills at 768.
constexpr int kBlock2 = 640;
constexpr int kBlock8 = 768, kBlock8Multi = 640;
constexpr int kMostWarps = (kBlock2 > kBlock8 ? kBlock2 : kBlock8) / 32;
__host__ __device__ constexpr int block_of(uint32_t form, bool batch) {
    return form == 2 ? kBlock2 : (batch ? kBlock8Multi : kBlock8);
}
constexpr uint32_t kTile = kStreamTile;  // positions a warp takes at a time
constexpr uint32_t kChunk = 512;         // positions per warp-wide 16-byte load
constexpr uint32_t kQueue = 256;         // survivors of a tile kept in shared memory at a time
constexpr uint32_t kNone = 1024;          // ids of -1 in shared memory, for bulk stores
// Whether the kernel writes its tiles of -1 by bulk stores (fill_none).
__host__ __device__ constexpr bool has_bulk(uint32_t form, int mode) { return form == 8 && mode == OUT_DENSE; }
constexpr uint32_t kRes2 = 160;          // 2-bit codes: candidates waiting to be resolved (31 + 4 * 32 at most)
constexpr uint32_t kRes8 = 64;           // 8-bit codes: survivors waiting (31 + 32 at most)
constexpr uint32_t kWarpBytes2 = kTile / 4 + 16 + 2 * kQueue + 16 + 8 * kRes2;  // (16: a step-1 tile's last marks)
constexpr uint32_t kWarpBytes8 = kTile + 16 + 2 * kQueue + 9 * kRes8;
static_assert(kWarpBytes2 % 16 == 0 && kWarpBytes8 % 16 == 0, "warp areas start on 16 bytes");


// 16 bytes of text, read once: around L1, first to leave L2.
__device__ __forceinline__ uint4 ldg_stream(const uint8_t *p, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}

// The 16 bytes at gbase + off with the bytes outside the text zero.
static __device__ __noinline__ uint4 load_fringe(const uint8_t *gbase, uint64_t off, uint64_t head, uint64_t end) {
    if (off >= head && off + 16u <= end) return __ldg(reinterpret_cast<const uint4 *>(gbase + off));
    uint32_t v[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (uint32_t j = 0; j < 16; ++j)
        if (off + j >= head && off + j < end) v[j >> 2] |= static_cast<uint32_t>(__ldg(gbase + off + j)) << (8u * (j & 3u));
    return make_uint4(v[0], v[1], v[2], v[3]);
}

// The text a warp's tiles belong to.  Positions are named by g, their index
// from the first position of tile t0: the text's position t0 * kTile + g - head.
// (One text: t0 = 0.  A batch: a few consecutive tiles of one text.)
struct Seg {
    const uint8_t *text;   // first byte
    const uint8_t *gbase;  // the same, rounded down to 16 bytes
    int32_t *out;          // dense ids
    uint64_t n;
    uint32_t head;         // text - gbase
    uint32_t t0;
    uint32_t in_lo, in_hi;  // the tiles wholly inside the text, with the 16 bytes after them
    uint32_t bit0;         // OUT_BITS: g + bit0 is the position's bit
    uint32_t unit0, item;  // a batch: work unit of tile t0, the text's entry in the planned list
};

__device__ __forceinline__ uint64_t text_pos(const Seg &sg, uint32_t g) {  // before the text wraps
    return static_cast<uint64_t>(sg.t0) * kTile + g - sg.head;
}

// The text's part of a segment.
__host__ __device__ __forceinline__ Seg make_seg(const uint8_t *text, int32_t *out, uint64_t n) {
    Seg sg;
    sg.text = text;
    sg.out = out;
    sg.n = n;
    sg.head = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(text) & 15u);
    sg.gbase = text - sg.head;
    const uint64_t a2 = (sg.head + n) & ~15ull;  // end of the text's 16-byte aligned part
    sg.in_lo = sg.head ? 1u : 0u;
    sg.in_hi = a2 >= 16u ? static_cast<uint32_t>((a2 - 16u) / kTile) : 0u;
    sg.t0 = sg.bit0 = sg.unit0 = sg.item = 0;
    return sg;
}

struct StreamParams {
    FilterParams f;        // tables, text, outputs, walk list (walks, walk_cap, list_count[1])
    const uint32_t *F1;    // root filter, f1bytes
    const uint32_t *F2;    // second filter (f2bytes; 0: none), with 8-bit codes then its short-keyword part
    uint32_t f1bytes, f2bytes;
    uint32_t ntiles;
    Seg sg;                // one text
    uint32_t four;         // 4
    uint32_t m1, m2;       // 8-bit codes: multipliers of the window's words
    uint32_t l2shift;      // 2-bit codes: left shift that drops the codes past the second filter's window
    uint32_t off_cta, off_warp;
};

// A tile's registers: lane l's 16 bytes of chunks 0-3, and (lane 0) the 16
// bytes after the tile.
struct TileRegs {
    uint4 c[4];
    uint4 look;
};

// Issue the loads of chunk C (4: the look-ahead) of the text's tile t.
template <int C>
__device__ __forceinline__ void load_chunk(const Seg &sg, uint32_t t, uint64_t pol, int lane, TileRegs &r) {
    const uint64_t lo = static_cast<uint64_t>(t) * kTile;
    if (t >= sg.in_lo && t < sg.in_hi) {
        if constexpr (C < 4)
            r.c[C] = ldg_stream(sg.gbase + lo + static_cast<uint32_t>(C) * kChunk + 16u * static_cast<uint32_t>(lane), pol);
        else if (lane == 0)
            r.look = ldg_stream(sg.gbase + lo + kTile, pol);
    } else {
        const uint64_t end = sg.head + sg.n;
        if constexpr (C < 4)
            r.c[C] = load_fringe(sg.gbase, lo + static_cast<uint32_t>(C) * kChunk + 16u * static_cast<uint32_t>(lane),
                                 sg.head, end);
        else if (lane == 0)
            r.look = load_fringe(sg.gbase, lo + kTile, sg.head, end);
    }
}

__device__ __forceinline__ void load_tile(const Seg &sg, uint32_t t, uint64_t pol, int lane, TileRegs &r) {
    load_chunk<0>(sg, t, pol, lane, r);
    load_chunk<1>(sg, t, pol, lane, r);
    load_chunk<2>(sg, t, pol, lane, r);
    load_chunk<3>(sg, t, pol, lane, r);
    load_chunk<4>(sg, t, pol, lane, r);
}

// The id of the longest keyword starting at text position gi, all from global
// memory: the window and stride tables, or the state hash, then the walk.
template <typename GT>
__device__ __forceinline__ int match_at(const FilterParams &p, const uint8_t *cls8, const TileText &tt, uint64_t gi,
                                        uint32_t B) {
    const int64_t gpb = static_cast<int64_t>(gi);
    if (B <= 4) {
        const uint32_t need = p.k + p.k2;
        if (gi + need <= tt.n) {
            uint32_t w = 0, bad = 0;
#pragma unroll
            for (uint32_t j = 0; j < 16; ++j)
                if (j < need) {
                    const uint32_t v = cls8[__ldg(tt.text + gi + j)];
                    bad |= v == 0xFFu ? 1u : 0u;
                    w |= (v & ((1u << B) - 1u)) << (B * j);
                }
            if (!bad) {
                const int e = __ldg(p.JK + (w & ((1u << (B * p.k)) - 1u)));
                if (e < 0) return decode_dead(e);
                uint32_t s = static_cast<uint32_t>(e), q = p.k;
                if (p.k2) {
                    const int e2 = __ldg(p.J2 + ((static_cast<uint64_t>(s - p.base_k) << (B * p.k2)) |
                                                 ((w >> (B * p.k)) & ((1u << (B * p.k2)) - 1u))));
                    if (e2 < 0) return decode_dead(e2);
                    s = static_cast<uint32_t>(e2);
                    q += p.k2;
                }
                return filt::walk_global<GT>(p, cls8, tt, gpb, s, q);
            }
        }
        return filt::walk_global<GT>(p, cls8, tt, gpb, 0u, 0u);
    }
    // 8-bit codes: no keyword is shorter than the state hash's window
    if (gi + p.k > tt.n) return -1;
    uint32_t w = 0, c = 0x100u;
#pragma unroll
    for (uint32_t j = 0; j <= kHashWindow; ++j) {
        if (j > p.k || gi + j >= tt.n) break;
        const uint32_t b = __ldg(tt.text + gi + j);
        const uint32_t v = p.identity ? b : cls8[b];
        const bool known = p.identity || v != 0xFFu;
        if (j < p.k) {
            if (!known) return -1;
            w |= v << (8u * j);
        } else if (known) {
            c = v;
        }
    }
    int r = -1;
    uint32_t s = 0, q = 0;
    if (filt::hk_outcome(p, filt::hk_find(p, w, __ldg(p.HK + filt::hk_slot(p, w))), 0u, c & 0xFFu, c < 0x100u, r, s, q))
        return r;
    return filt::walk_global<GT>(p, cls8, tt, gpb, s, q);
}

template <typename GT>
static __device__ __noinline__ int match_at_far(const FilterParams &p, const uint8_t *cls8, const TileText tt,
                                                uint64_t gi, uint32_t B) {
    return match_at<GT>(p, cls8, tt, gi, B);
}

// A warp's run of 32 * PER consecutive positions, lane l's g0, g0 + 32, ...  It
// reads their bytes and the 16 after them once, one byte a lane and load, and
// joins their codes into windows with log2(window) shuffles, so a position costs
// little more than a byte load and a load per table level; a lane's PER positions
// have theirs in flight together.  (g0 may lie before the text, and wraps then.)
template <int PER>
__device__ __forceinline__ void load_run(const uint8_t *text, uint64_t n, uint64_t g0, int lane, uint32_t (&c)[PER + 1],
                                         bool (&in)[PER + 1]) {
#pragma unroll
    for (int j = 0; j <= PER; ++j) {
        in[j] = g0 + 32u * j < n && (j < PER || lane < 16);
        c[j] = in[j] ? __ldg(text + g0 + 32u * j) : 0u;
    }
}

// A position after its first loads: its id, or the walk that is left (state s, the
// code at position + q next).
template <int PER>
struct RunState {
    int r[PER];
    uint32_t s[PER], q[PER];
    bool walk[PER];
};
template <int B, int PER, bool FIRST>
__device__ __forceinline__ void resolve_run(const FilterParams &p, const uint8_t *cls8, int lane, uint32_t (&c)[PER + 1],
                                            const bool (&in)[PER + 1], RunState<PER> &st) {
    // codes, and which positions hold none (a byte in no keyword, or the text's end)
    const bool id = B == 8 && p.identity;
    uint32_t bad[PER + 1];  // bit i: position i of the 32
#pragma unroll
    for (int j = 0; j <= PER; ++j) {
        if (!id) c[j] = cls8[c[j]];
        bad[j] = __ballot_sync(kFull, !in[j] || (!id && c[j] == 0xFFu));
        c[j] &= (1u << B) - 1u;
    }
    const uint32_t need = B == 8 ? p.k : p.k + p.k2;
    uint32_t after[PER];  // 8-bit codes: the code after the window
    if (B == 8) {
        const uint32_t x = static_cast<uint32_t>(lane) + p.k;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const uint32_t y = __shfl_sync(kFull, c[j], x & 31u), z = __shfl_sync(kFull, c[j + 1], x & 31u);
            after[j] = x < 32u ? y : z;
        }
    }
#pragma unroll
    for (uint32_t d = 1; d * B < 32u; d *= 2u) {  // windows of d codes -> 2 d
        const uint32_t x = static_cast<uint32_t>(lane) + d;
        uint32_t y = __shfl_sync(kFull, c[0], x & 31u);
#pragma unroll
        for (int j = 0; j <= PER; ++j) {  // (the last set's upper lanes are never read)
            const uint32_t z = j < PER ? __shfl_sync(kFull, c[j < PER ? j + 1 : j], x & 31u) : y;
            c[j] |= (x < 32u ? y : z) << (B * d);
            y = z;
        }
    }
    // first loads of all the lane's positions, then the second
    int e[PER];
    uint4 h[PER];
    bool keep[PER];
    uint32_t m[PER];
    auto &r = st.r;
    auto &s = st.s;
    auto &q = st.q;
    auto &walk = st.walk;
    // FIRST (longer texts, few of whose positions get past it): the root filter
    // first, whose 128 KiB stay in L1, not a sector of a table in L2 for each
    // position (2 MiB of ACGT 16.6 -> 14.7 us a call, of Zipf bytes 29.0 -> 25.8;
    // short texts would wait for one load more, and nearly all positions of the
    // tiles listed whole pass it)
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        keep[j] = true;
        if (!FIRST) continue;
        const uint32_t v = B == 8 ? ((c[j] & p.wmask) * kFilterHashMul) >> p.fshift
                                  : c[j] & ((1u << (B * p.k)) - 1u);
        keep[j] = (__ldg(p.Fg + (v >> 5)) << (v & 31u)) >> 31;
    }
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        m[j] = __funnelshift_r(bad[j], bad[j + 1], lane);  // bit i: position i after this one
        walk[j] = in[j];
        r[j] = -1;
        s[j] = q[j] = 0;
        e[j] = 0;
        h[j] = make_uint4(0u, 0u, 0u, 0u);
        if (m[j] & ((1u << need) - 1u)) {
            if (B == 8) walk[j] = false;  // no keyword is shorter than the state hash's window
            continue;
        }
        if (!keep[j]) {
            walk[j] = false;
            e[j] = -1;
            continue;
        }
        if (B == 8)
            h[j] = __ldg(p.HK + filt::hk_slot(p, c[j] & p.wmask));
        else
            e[j] = __ldg(p.JK + (c[j] & ((1u << (B * p.k)) - 1u)));
    }
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if ((m[j] & ((1u << need) - 1u)) || !keep[j]) continue;
        if (B == 8) {
            walk[j] = !filt::hk_outcome(p, filt::hk_find(p, c[j] & p.wmask, h[j]), 0u, after[j], !((m[j] >> p.k) & 1u),
                                        r[j], s[j], q[j]);
        } else if (e[j] >= 0 && p.k2) {
            q[j] = p.k + p.k2;
            e[j] = __ldg(p.J2 + ((static_cast<uint64_t>(static_cast<uint32_t>(e[j]) - p.base_k) << (B * p.k2)) |
                                 ((c[j] >> (B * p.k)) & ((1u << (B * p.k2)) - 1u))));
        } else {
            q[j] = p.k;
        }
    }
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if (B != 8 && !(m[j] & ((1u << need) - 1u))) {
            walk[j] = e[j] >= 0;
            s[j] = static_cast<uint32_t>(e[j]);
            if (e[j] < 0) r[j] = decode_dead(e[j]);
        }
    }
}

// put(j, id or -1) for each of the lane's positions (all lanes of the warp), each
// lane walking its own.
template <int B, typename GT, int PER, bool FIRST, typename Put>
__device__ __forceinline__ void match_run(const FilterParams &p, const uint8_t *cls8, const TileText &tt, uint64_t g0,
                                          int lane, uint32_t (&c)[PER + 1], const bool (&in)[PER + 1], Put put) {
    RunState<PER> st;
    resolve_run<B, PER, FIRST>(p, cls8, lane, c, in, st);
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if (st.walk[j])
            st.r[j] = filt::walk_global<GT>(p, cls8, tt, static_cast<int64_t>(g0 + 32u * j), st.s[j], st.q[j]);
        put(j, in[j] ? st.r[j] : -1);
    }
}

// An id found at position g.  OUT_BITS with tile (the warp's bits of the tile
// from position g0 on, in shared memory, every id of which passes here before
// the tile's bits and count are written): the bit goes there.
struct TileBits {
    uint32_t *bits;
    const uint16_t *marks;  // step 1: which of the tile's bytes are in no keyword, or outside the text
    uint32_t g0;
};
template <int MODE>
__device__ __forceinline__ void put_id(const FilterParams &p, const Seg &sg, uint32_t g, int r, uint32_t &cnt,
                                       const TileBits tile = TileBits{nullptr, nullptr, 0u}) {
    if (r < 0) return;
    if (MODE == OUT_DENSE) {
        sg.out[text_pos(sg, g)] = r;
    } else if (MODE == OUT_COUNT) {
        ++cnt;
    } else {
        const uint32_t b = g + sg.bit0;
        p.bo.ids[b] = r;
        if (tile.bits) {
            atomicOr(tile.bits + ((g - tile.g0) >> 5), 1u << (g & 31u));
        } else {
            atomicOr(p.bo.bits + (b >> 5), 1u << (b & 31u));
            atomicAdd(p.bo.counts + b / kTile, 1u);
        }
    }
}

// Walk-list entries.  One text: {g, state | d << 31}: the walk goes on from the
// state with the byte k + k2 + d after the position; state 0: not resolved at
// all.  A batch: {work unit, state | d << 31, automaton << 11 | position in the
// unit, planned-list entry}.  An empty entry's first word is 0xFFFFFFFF.
template <bool BATCH>
__device__ __forceinline__ void store_walk(const FilterParams &p, const Seg &sg, uint32_t slot, uint32_t g, uint32_t s) {
    if (BATCH)
        p.walks4[slot] = make_uint4(sg.unit0 + g / kTile, s, (p.aidx << 11) | (g & (kTile - 1u)), sg.item);
    else
        p.walks[slot] = make_uint2(g, s);
}
template <bool BATCH>
__device__ __forceinline__ void blank_walk(const FilterParams &p, uint32_t slot) {
    if (BATCH)
        p.walks4[slot] = make_uint4(0xFFFFFFFFu, 0u, 0u, 0u);
    else
        p.walks[slot] = make_uint2(0xFFFFFFFFu, 0u);
}

// Walks to the walk list (all lanes of the warp; want: this lane has one).
// Space is reserved in chunks; when one runs out its rest takes the first
// walks.  False for a lane whose walk found no room (the list is full).
struct WalkRoom {
    uint32_t next, end;  // the warp's chunk
    bool full;           // nothing more to reserve (the counter is left alone then)
    bool crowd;          // kSpread tiles were listed to spread them
};

// Tiles listed whole.  A tile with many candidates is not this launch's work: its
// 20 or 24 warps an SM wait for one dependent load after another.  The walks'
// launch takes such a tile with one lane a position (tile_run), over 48 warps an
// SM.  Texts of 64 MiB, dense ids, ms: walks listed one by one and, where there was
// no more room, done where they were found / these tiles listed whole / the filter
// kernel, which keeps eight walks a lane in flight: one DNA letter 3.13 / 1.61 /
// 2.10, one byte 3.45 / 1.75 / 2.11, a phrase of 78 bytes 3.30 / 2.50 / 2.64, a
// repeat of 1,009 letters 4.26 / 2.20 / 2.06.  Listed are
//   - tiles in which more than a quarter to a half of the positions looked up pass
//     the filter (kQueue in pfac_stream2, half a tile in pfac_stream8);
//   - once the walk list is full, tiles with more than kFew that pass (the walks of
//     the others are settled where they are found);
//   - in pfac_stream2 with S > 1, the first kSpread tiles with more candidates than
//     the warp resolves in 8 rounds: a few of them in a text would each keep one
//     warp busy long after the others have ended (5,000 keywords copied from the
//     first 4 KiB of 16 MiB).  Where there are many (a repeat of 4,096 letters, 5 %
//     of its positions walk) the warps resolve the rest: 64 MiB 429 us, all of them
//     listed 850.
constexpr uint32_t kSpread = 128;
constexpr uint32_t kFew = 128;
// True when tile t of sg is listed (all lanes).
template <bool BATCH>
__device__ __forceinline__ bool list_tile(const FilterParams &p, const Seg &sg, uint32_t t, int lane) {
    uint32_t i = 0;
    if (lane == 0) {
        i = atomicAdd(p.list_count + 2, 1u);
        if (i < p.tile_cap) {
            if (BATCH)
                p.walks4[p.walk_cap + i] = make_uint4(sg.unit0 + (t - sg.t0), 0u, p.aidx << 11, sg.item);
            else
                reinterpret_cast<uint32_t *>(p.walks + p.walk_cap)[i] = t;
        }
    }
    return __shfl_sync(kFull, i, 0) < p.tile_cap;
}

// Whether kSpread tiles were listed for their few but slow candidates (all lanes).
__device__ __forceinline__ bool crowded(const FilterParams &p, WalkRoom &room, int lane) {
    if (!room.crowd) {
        uint32_t i = 0;
        if (lane == 0) i = atomicAdd(p.list_count + 3, 1u);
        room.crowd = __shfl_sync(kFull, i, 0) >= kSpread;
    }
    return room.crowd;
}
template <bool BATCH>
__device__ __forceinline__ bool push_walk(const StreamParams &p, const Seg &sg, WalkRoom &room, bool want, uint32_t g,
                                          uint32_t s, int lane) {
    const unsigned m = __ballot_sync(kFull, want);
    if (!m) return true;
    const uint32_t need = __popc(m), rank = __popc(m & ((1u << lane) - 1u)), rest = room.end - room.next;
    uint32_t slot = room.next + rank;
    bool stored = want;
    if (rest < need) {
        uint32_t base = p.f.walk_cap, end = p.f.walk_cap;
        if (!room.full) {
            const uint32_t chunk = need - rest > p.f.walk_chunk ? need - rest : p.f.walk_chunk;
            if (lane == 0) base = atomicAdd(p.f.list_count + 1, chunk);
            base = __shfl_sync(kFull, base, 0);
            room.full = base >= p.f.walk_cap || p.f.walk_cap - base <= chunk;
            end = room.full ? p.f.walk_cap : base + chunk;
            if (base > end) base = end;
        }
        if (rank >= rest) {
            slot = base + (rank - rest);
            stored = want && slot < end;
        }
        room.next = end - base < need - rest ? end : base + (need - rest);
        room.end = end;
    } else {
        room.next += need;
    }
    if (stored) store_walk<BATCH>(p.f, sg, slot, g, s);
    return !want || stored;
}

// The warp's unused walk-list entries are empty.
template <bool BATCH>
__device__ __forceinline__ void close_room(const FilterParams &f, const WalkRoom &room, int lane) {
    for (uint32_t j = room.next + static_cast<uint32_t>(lane); j < room.end; j += 32u) blank_walk<BATCH>(f, j);
}

// -1 for every position of tile t inside the text.  BULK (8-bit codes): bulk
// stores of a constant buffer (none: kNone ids of -1 in shared memory) by lane
// 0, where the output shares the text's 16-byte boundaries: that kernel is
// bound by its shared-memory lookups, and plain stores wait in the same queue
// (1 GiB dense: 1.08 against 1.17 ms).  With 2-bit codes plain stores are the
// faster (0.90 against 0.97 ms): the kernel waits for memory, and the bulk
// stores' traffic comes with 9 % more DRAM reads.  Plain 16-byte stores follow
// the output's own alignment: a tile whose first id is m ids past a boundary
// writes its first 4 - m and last m ids one by one.
template <bool BULK>
__device__ __forceinline__ void fill_none(const Seg &sg, const int32_t *none, uint32_t t, int lane) {
    const int64_t lo = static_cast<int64_t>(static_cast<uint64_t>(t) * kTile) - sg.head;
    int32_t *o = sg.out + lo;
    if (t >= sg.in_lo && t < sg.in_hi) {
        if (BULK && (reinterpret_cast<uintptr_t>(o) & 15u) == 0u) {
            if (lane == 0) {
#pragma unroll
                for (uint32_t j = 0; j < kTile; j += kNone) bulk_store(o + j, none, kNone * 4u);
                bulk_commit();
                bulk_wait_read_keep8();  // bound the groups in flight
            }
            return;
        }
        const uint32_t m = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(o) >> 2) & 3u;
        const uint32_t f = (4u - m) & 3u;
        const int4 minus = make_int4(-1, -1, -1, -1);
        int4 *v = reinterpret_cast<int4 *>(o + f) + lane;
#pragma unroll
        for (uint32_t j = 0; j < 15; ++j) v[32u * j] = minus;
        if (m == 0u || lane < 31) v[32u * 15u] = minus;
        if (m != 0u && lane < 4) {
            const uint32_t i = static_cast<uint32_t>(lane);
            o[i < f ? i : kTile - 4u + i] = -1;
        }
    } else {
        for (uint32_t i = static_cast<uint32_t>(lane); i < kTile; i += 32u) {
            const int64_t g = lo + static_cast<int64_t>(i);
            if (g >= 0 && g < static_cast<int64_t>(sg.n)) o[i] = -1;
        }
    }
}

// OUT_BITS: no bits and no matches yet in tile t.
__device__ __forceinline__ void clear_bits(const FilterParams &f, const Seg &sg, uint32_t t, int lane) {
    const size_t u = sg.bit0 / kTile + (t - sg.t0);
    reinterpret_cast<uint2 *>(f.bo.bits + u * (kTile / 32u))[lane] = make_uint2(0u, 0u);
    if (lane == 0) f.bo.counts[u] = 0u;
}

// Before ids are written over the fill: the bulk stores have completed (found:
// some lane has an id), and every lane's plain stores come first.
template <int MODE, bool BULK>
__device__ __forceinline__ void fill_done(bool found, int lane) {
    if (MODE == OUT_COUNT) return;
    if (MODE == OUT_DENSE && BULK && __any_sync(kFull, found) && lane == 0) bulk_wait_all();
    __syncwarp();
}

// The id at position g, all here: the walk list is full.
template <int MODE>
__device__ __forceinline__ void settle_here(const StreamParams &p, const Seg &sg, uint32_t g, uint32_t B, uint32_t &cnt,
                                            const TileBits tile = TileBits{nullptr, nullptr, 0u}) {
    const TileText tt = make_text(sg.text, sg.out, sg.n, 0u);
    const int r = (p.f.kind & 0xFFu) == 16u ? match_at_far<int16_t>(p.f, p.f.cls8g, tt, text_pos(sg, g), B)
                                            : match_at_far<int32_t>(p.f, p.f.cls8g, tt, text_pos(sg, g), B);
    put_id<MODE>(p.f, sg, g, r, cnt, tile);
}

// Walks (want: this lane has one) to the list, or settled here when it is full.
template <int B, int MODE, bool BATCH>
__device__ __forceinline__ void list_walk(const StreamParams &p, const Seg &sg, WalkRoom &room, bool want, uint32_t g,
                                          uint32_t s, int lane, uint32_t &cnt,
                                          const TileBits tile = TileBits{nullptr, nullptr, 0u}) {
    const bool stored = push_walk<BATCH>(p, sg, room, want, g, s, lane);
    if (!room.full || __all_sync(kFull, stored)) return;
    fill_done<MODE, B == 8>(true, lane);
    if (!stored) settle_here<MODE>(p, sg, g, B, cnt, tile);
}

// The -1 buffer (all threads; a CTA barrier follows).
__device__ __forceinline__ void fill_constant(uint8_t *at) {
    for (uint32_t i = threadIdx.x; i < kNone / 4u; i += blockDim.x) reinterpret_cast<int4 *>(at)[i] = make_int4(-1, -1, -1, -1);
    fence_proxy_async_smem();  // read by bulk stores
}

// One CTA's filters into shared memory (all threads; a CTA barrier follows).
__device__ __forceinline__ void load_filters(const StreamParams &p, uint8_t *smem) {
    uint4 *d = reinterpret_cast<uint4 *>(smem);
    const uint4 *a = reinterpret_cast<const uint4 *>(p.F1), *b = reinterpret_cast<const uint4 *>(p.F2);
    const uint32_t na = p.f1bytes >> 4, nb = p.f2bytes >> 4;
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < na; i += blockDim.x) d[i] = __ldg(a + i);
    for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x) d[na + i] = __ldg(b + i);
}

// Exclusive sum over the lanes below; total: the warp's.
__device__ __forceinline__ uint32_t warp_excl(uint32_t v, uint32_t &total, int lane) {
    uint32_t inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, inc, d);
        if (lane >= d) inc += y;
    }
    total = __shfl_sync(kFull, inc, 31);
    return inc - v;
}

template <int MODE>
__device__ __forceinline__ void add_count(const FilterParams &p, uint32_t cnt, int lane) {
    if (MODE != OUT_COUNT) return;
    const uint32_t s = __reduce_add_sync(kFull, cnt);  // fewer than 2^32 positions a launch
    if (lane == 0 && s) atomicAdd(p.count, static_cast<unsigned long long>(s));
}

// ---- 2-bit codes -------------------------------------------------------------

// The codes of 16 bytes: masked in place, one multiply per word gathers its
// four codes into the top byte, byte permutes join the four.
__device__ __forceinline__ uint32_t codes16(const uint4 &v) {
    constexpr uint32_t dmask = 0x06060606u, dmul = 0x01041040u >> 1;
    return __byte_perm(__byte_perm((v.x & dmask) * dmul, (v.y & dmask) * dmul, 0x0073u),
                       __byte_perm((v.z & dmask) * dmul, (v.w & dmask) * dmul, 0x0073u), 0x5410u);
}

// Non-zero when one of 16 bytes is in no keyword: a byte is in one exactly when
// the keyword byte of its code equals it, and a byte permute selected by twice
// the codes (each word's next byte's moved to the high nibble) picks those.
__device__ __forceinline__ uint32_t unknown4(const FilterParams &f, uint32_t w) {
    const uint32_t x = w & 0x06060606u;
    return w ^ __byte_perm(f.dsel_lo, f.dsel_hi, __byte_perm(x | (x >> 4), 0u, 0x4420u));
}
__device__ __forceinline__ uint32_t unknown16(const FilterParams &f, const uint4 &v) {
    return unknown4(f, v.x) | unknown4(f, v.y) | unknown4(f, v.z) | unknown4(f, v.w);
}

// The same, a flag per byte.
__device__ __forceinline__ uint32_t unknown_marks(const FilterParams &f, const uint4 &v) {
    auto word = [&](uint32_t w) { return filt::nonzero_bytes(unknown4(f, w)); };
    return word(v.x) | (word(v.y) << 4) | (word(v.z) << 8) | (word(v.w) << 12);
}

// The 16 codes from tile position i on, from the tile's packed codes.
__device__ __forceinline__ uint32_t codes_at(const uint32_t *packed, uint32_t i) {
    return __funnelshift_r(packed[i >> 4], packed[(i >> 4) + 1u], 2u * (i & 15u));
}

// Whether the `need` (<= 16) bytes from text position gi on are inside the
// text and all in keywords: at most five aligned words, all in flight together
// (those that hold one of the bytes), and byte permutes as in unknown16.
__device__ __forceinline__ bool bytes_known(const FilterParams &f, const uint8_t *text, uint64_t n, uint64_t gi,
                                            uint32_t need) {
    if (gi + need > n) return false;
    const uint8_t *t = text + gi;
    const uint32_t a = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(t) & 3u), words = (a + need + 3u) >> 2;
    const uint32_t *w = reinterpret_cast<const uint32_t *>(t - a);
    uint32_t x[5], bad = 0;
#pragma unroll
    for (uint32_t j = 0; j < 5; ++j) x[j] = j < words ? __ldg(w + j) : 0u;
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
        const uint32_t v = __funnelshift_r(x[j], x[j + 1], 8u * a), left = need - 4u * j;
        if (need > 4u * j) bad |= unknown4(f, v) & (left >= 4u ? 0xFFFFFFFFu : (1u << (8u * left)) - 1u);
    }
    return bad == 0;
}

// ... those of a window: out of line for the matcher, which asks for the few
// results of sets with windows of several positions (inlined: 96 registers for 90).
static __device__ __noinline__ bool bytes_known_far(const FilterParams &f, const uint8_t *text, uint64_t n, uint64_t gi) {
    return bytes_known(f, text, n, gi, f.k + f.k2);
}

// A round of candidates (all lanes; on: this lane has one: position g and the
// 16 codes w from it): window table, stride table, then out or to the walk
// list.  The codes may be those of bytes in no keyword, or of bytes past the
// text: a keyword that ends before such a byte is on the walk of the codes too,
// so a position without a result has none; one with a result has its bytes
// looked at (known: no need to, they are keyword bytes of the text), and a
// walk's bytes are looked at when it goes on.
template <int MODE, bool BATCH, bool CHECK>
__device__ __forceinline__ void resolve2(const StreamParams &p, const Seg &sg, WalkRoom &room, uint32_t g, uint32_t w,
                                         bool on, bool known, int lane, uint32_t &cnt, const TileBits tile) {
    const FilterParams &f = p.f;
    const uint64_t gi = text_pos(sg, g);
    bool walk = false;
    uint32_t s = 0;
    int r = -1;
    if (on && gi < sg.n) {
        const int e = __ldg(f.JK + (w & ((1u << (2u * f.k)) - 1u)));
        if (e < 0) {
            r = decode_dead(e);
        } else {
            s = static_cast<uint32_t>(e);
            walk = true;
            if (f.k2) {
                const int e2 = __ldg(f.J2 + ((static_cast<uint64_t>(s - f.base_k) << (2u * f.k2)) |
                                             ((w >> (2u * f.k)) & ((1u << (2u * f.k2)) - 1u))));
                s = static_cast<uint32_t>(e2);
                if (e2 < 0) {
                    r = decode_dead(e2);
                    walk = false;
                }
            }
        }
        bool doubt = r >= 0 && !known;
        if (CHECK) {
            if (doubt) {
                const uint32_t i = g - tile.g0;
                const uint32_t m = tile.marks[i >> 4] | (static_cast<uint32_t>(tile.marks[(i >> 4) + 1u]) << 16);
                doubt = ((m >> (i & 15u)) & ((1u << (f.k + f.k2)) - 1u)) != 0u;
            }
        } else {
            doubt = doubt && !bytes_known_far(f, sg.text, sg.n, gi);
        }
        if (doubt) {
            walk = true;
            s = 0;
            r = -1;
        }
    }
    fill_done<MODE, false>(r >= 0, lane);
    put_id<MODE>(f, sg, g, r, cnt, tile);
    list_walk<2, MODE, BATCH>(p, sg, room, walk, g, s, lane, cnt, tile);
}

// One warp's state across its tiles: candidates or survivors waiting to be
// resolved, its walk-list chunk, its count.
struct WarpState {
    uint32_t nres, cnt;
    WalkRoom room;
};

// One warp: tiles t, t + step, ... below t_end of sg's text (tile t's loads are
// issued); what waits in shared memory belongs to sg (BATCH: flushed at the end).
template <int S, int MODE, bool BATCH>
__device__ __forceinline__ void tiles2(const StreamParams &p, uint8_t *smem, uint32_t off_warp, const int32_t *none,
                                       const Seg &sg, uint32_t t, uint32_t t_end, uint32_t step, uint64_t pol,
                                       TileRegs &r, WarpState &ws) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t *F1 = reinterpret_cast<const uint32_t *>(smem);
    const uint32_t *F2 = reinterpret_cast<const uint32_t *>(smem + p.f1bytes);
    uint32_t *packed = reinterpret_cast<uint32_t *>(smem + off_warp + static_cast<uint32_t>(warp) * kWarpBytes2);
    uint2 *res = reinterpret_cast<uint2 *>(packed + kTile / 16 + 4);
    uint16_t *queue = reinterpret_cast<uint16_t *>(res + kRes2);
    uint32_t nres = ws.nres, cnt = ws.cnt;  // candidates waiting in res: {g, codes}
    // every position looked up: the sets with many matches, so the tile's bytes
    // are looked at once for all of them, and only a tile with bytes in no
    // keyword (or of the text's ends) marks them; with fewer matches the check
    // costs more than it saves.  (64 MiB of uniform text, a fifth of it matches:
    // dense ids 330 -> 200 us; the filter kernel 240.)
    constexpr bool CHECK = S == 1;
    bool known = false;  // those waiting are from tiles without such bytes
    uint16_t *marks = queue + kTile / 16;  // 129 of them
    // ... and OUT_BITS collects the tile's bits in shared memory (the queue is
    // the second filter's, which these sets have not): its candidates are all
    // resolved before it ends, and no bit or count takes a global atomic
    constexpr bool LOCAL = CHECK && MODE == OUT_BITS;
    uint32_t *tbits = reinterpret_cast<uint32_t *>(queue);
    TileBits tile{LOCAL ? tbits : nullptr, marks, 0u};
    WalkRoom room = ws.room;
    auto flush = [&](uint32_t n) {  // resolve the last n (<= 32) of them
        __syncwarp();
        nres -= n;
        const bool on = static_cast<uint32_t>(lane) < n;
        const uint2 e = res[nres + (on ? static_cast<uint32_t>(lane) : 0u)];
        resolve2<MODE, BATCH, CHECK>(p, sg, room, e.x, e.y, on, known, lane, cnt, tile);
        __syncwarp();
    };
    for (; t < t_end; t += step) {
        // 1. codes; the registers are free for the next tile's loads
        uint32_t c[5];
#pragma unroll
        for (int j = 0; j < 4; ++j) c[j] = codes16(r.c[j]);
        c[4] = codes16(r.look);
        if (CHECK) {
            uint32_t bad = lane == 0 ? unknown16(p.f, r.look) : 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) bad |= unknown16(p.f, r.c[j]);
            const bool clean = t >= sg.in_lo && t < sg.in_hi && !__any_sync(kFull, bad != 0u);
            if (nres && !(clean && known)) flush(nres);  // before their tile's marks go
            known = clean;
            tile.g0 = (t - sg.t0) * kTile;
            if (!clean) {
                __syncwarp();
#pragma unroll
                for (uint32_t j = 0; j <= 4; ++j) {
                    const uint32_t i = j * kChunk + 16u * static_cast<uint32_t>(lane);
                    uint32_t m = unknown_marks(p.f, j < 4 ? r.c[j < 4 ? j : 0] : r.look);
                    m |= filt::outside_marks(static_cast<int64_t>(text_pos(sg, tile.g0 + i)), static_cast<int64_t>(sg.n));
                    if (j < 4 || lane == 0) marks[32u * j + static_cast<uint32_t>(lane)] = static_cast<uint16_t>(m);
                }
            }
        }
        if (t + step < t_end) load_tile(sg, t + step, pol, lane, r);
        __syncwarp();  // the previous tile's readers of packed and queue are done
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) packed[32u * j + static_cast<uint32_t>(lane)] = c[j];
        if (lane == 0) packed[128] = c[4];
        if (MODE == OUT_DENSE) fill_none<false>(sg, none, t, lane);
        if (MODE == OUT_BITS && !LOCAL) clear_bits(p.f, sg, t, lane);
        if (LOCAL) {
            reinterpret_cast<uint2 *>(tbits)[lane] = make_uint2(0u, 0u);
        }

        // 2. the root filter at every S-th position: one bit each, first
        //    position highest
        constexpr int kPer = 16 / S;         // samples per lane and chunk
        constexpr int kAcc = kPer == 16 ? 2 : 1;
        uint32_t acc[kAcc];
#pragma unroll
        for (int a = 0; a < kAcc; ++a) acc[a] = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t give = lane == 0 ? c[j + 1] : c[j];
            const uint32_t nb = __shfl_sync(kFull, give, (lane + 1) & 31);
#pragma unroll
            for (int x = 0; x < kPer; ++x) {
                const uint32_t w = __funnelshift_r(c[j], nb, 2 * (S * x + S - 1));
                const uint32_t word = F1[(w >> 5) & 0x7FFFu];
                uint32_t &a = acc[kAcc == 2 ? j >> 1 : 0];
                a = __funnelshift_l(__funnelshift_l(word, word, w), a, 1);
            }
        }
        __syncwarp();  // packed is written
        constexpr int kBits = 4 * kPer / kAcc;  // bits per accumulator
        if (S == 1 && room.full) {
            uint32_t found = 0;
#pragma unroll
            for (int a = 0; a < kAcc; ++a) found += static_cast<uint32_t>(__popc(acc[a]));
            if (__reduce_add_sync(kFull, found) > kFew && list_tile<BATCH>(p.f, sg, t, lane)) {
#pragma unroll
                for (int a = 0; a < kAcc; ++a) acc[a] = 0;
            }
        }
        const uint32_t g0 = (t - sg.t0) * kTile;
#pragma unroll
        for (int a = 0; a < kAcc; ++a) {
            uint32_t m = __brev(acc[a] << (32 - kBits));
            uint32_t left = __ballot_sync(kFull, m != 0u);
            if (!left) continue;
            auto sample = [&](uint32_t b) {  // tile position of bit b
                return static_cast<uint32_t>(a) * 2u * kChunk + kChunk * (b / kPer) +
                       16u * static_cast<uint32_t>(lane) + S * (b % kPer) + (S - 1u);
            };
            const uint32_t total = __reduce_add_sync(kFull, static_cast<uint32_t>(__popc(m)));
            if (S > 1 && total > kQueue / S && (total > kQueue || room.full || !crowded(p.f, room, lane)) &&
                list_tile<BATCH>(p.f, sg, t, lane))
                continue;
            if (S > 1 && p.f2bytes && total <= kQueue) {
                // 3. the second filter drops the chance hits among the samples
                uint32_t at = 0;
                for (; left; left = __ballot_sync(kFull, m != 0u)) {
                    if (m) queue[at + __popc(left & lt)] = static_cast<uint16_t>(sample(__ffs(m) - 1));
                    m &= m - 1u;
                    at += __popc(left);
                }
                __syncwarp();
                for (uint32_t b = 0; b < total; b += 32u) {
                    const uint32_t x = b + static_cast<uint32_t>(lane);
                    const uint32_t i = queue[x < total ? x : 0u];
                    const uint32_t h = (codes_at(packed, i) << p.l2shift) * kFilterHashMul;
                    const uint32_t word = F2[__umulhi(h, p.f2bytes >> 2)];
                    const bool pass = x < total && ((word >> ((h >> 12) & 31u)) & 1u);
                    const unsigned pm = __ballot_sync(kFull, pass);
                    if (!pm) continue;
                    if (pass) {
                        const uint32_t o = nres + S * __popc(pm & lt);
#pragma unroll
                        for (uint32_t y = 0; y < S; ++y) res[o + y] = make_uint2(g0 + i - y, codes_at(packed, i - y));
                    }
                    nres += S * __popc(pm);
                    while (nres >= 32u) flush(32u);
                }
                __syncwarp();
            } else {
                for (; left; left = __ballot_sync(kFull, m != 0u)) {
                    if (m) {
                        const uint32_t i = sample(__ffs(m) - 1), o = nres + S * __popc(left & lt);
#pragma unroll
                        for (uint32_t y = 0; y < S; ++y) res[o + y] = make_uint2(g0 + i - y, codes_at(packed, i - y));
                    }
                    m &= m - 1u;
                    nres += S * __popc(left);
                    while (nres >= 32u) flush(32u);
                }
            }
        }
        if (LOCAL) {
            if (nres) flush(nres);
            const uint2 b = reinterpret_cast<const uint2 *>(tbits)[lane];
            const uint32_t n = __reduce_add_sync(kFull, static_cast<uint32_t>(__popc(b.x) + __popc(b.y)));
            const size_t u = sg.bit0 / kTile + (t - sg.t0);
            reinterpret_cast<uint2 *>(p.f.bo.bits + u * (kTile / 32u))[lane] = b;
            if (lane == 0) p.f.bo.counts[u] = n;
        }
    }
    if (nres) flush(nres);
    ws.nres = nres;
    ws.cnt = cnt;
    ws.room = room;
}

// ---- 8-bit codes -------------------------------------------------------------

// A round of survivors (all lanes; on: this lane has one: position g, its
// window's four bytes w and the byte c after them): the state hash, for a
// branching state the first goto step, then out or to the walk list.
template <int MODE, bool BATCH>
__device__ __forceinline__ void resolve8(const StreamParams &p, const Seg &sg, WalkRoom &room, uint32_t g, uint32_t w,
                                         uint32_t c, bool on, int lane, uint32_t &cnt) {
    const FilterParams &f = p.f;
    const uint64_t gi = text_pos(sg, g);
    // windows past the text end (or before its start, which wraps) hold no keyword
    on = on && gi < sg.n && gi + f.k <= sg.n;
    bool c_ok = gi + f.k < sg.n;
    if (on && !f.identity) {
        uint32_t x = 0, bad = 0;
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) {
            const uint32_t v = __ldg(f.cls8g + ((w >> (8u * j)) & 0xFFu));
            bad |= v == 0xFFu ? 1u : 0u;
            x |= v << (8u * j);
        }
        w = x;
        on = bad == 0;
        c = __ldg(f.cls8g + c);
        c_ok = c_ok && c != 0xFFu;
    }
    int r = -1;
    uint32_t s = 0, q = 0;
    bool walk = false;
    if (on) {
        walk = !filt::hk_outcome(f, filt::hk_find(f, w, __ldg(f.HK + filt::hk_slot(f, w))), 0u, c, c_ok, r, s, q);
        if (walk && q == f.k) {  // a branching state
            const uint32_t col = c_ok ? c : f.C;
            const int e = (f.kind & 0xFFu) == 16u ? goto_ld(static_cast<const int16_t *>(f.G), s, f.W, col)
                                                  : goto_ld(static_cast<const int32_t *>(f.G), s, f.W, col);
            s = static_cast<uint32_t>(e);
            q = f.k + 1u;
            if (e < 0) {
                r = decode_dead(e);
                walk = false;
            }
        }
        if (walk) r = -1;
    }
    fill_done<MODE, true>(r >= 0, lane);
    put_id<MODE>(f, sg, g, r, cnt);
    list_walk<8, MODE, BATCH>(p, sg, room, walk, g, s | (1u << 31), lane, cnt);
}

// As tiles2, 8-bit codes.
template <int MODE, bool BATCH>
__device__ __forceinline__ void tiles8(const StreamParams &p, uint8_t *smem, uint32_t off_warp, const int32_t *none,
                                       const Seg &sg, uint32_t t, uint32_t t_end, uint32_t step, uint64_t pol,
                                       TileRegs &r, WarpState &ws) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t *F1 = reinterpret_cast<const uint32_t *>(smem);
    const uint32_t *F2 = reinterpret_cast<const uint32_t *>(smem + p.f1bytes);
    const uint32_t f2words = (p.f2bytes - kStreamShortBytes) >> 2;  // only used with a second filter
    const uint32_t *FS = F2 + f2words;
    uint32_t *stage = reinterpret_cast<uint32_t *>(smem + off_warp + static_cast<uint32_t>(warp) * kWarpBytes8);
    uint32_t *res_g = stage + kTile / 4 + 4, *res_w = res_g + kRes8;
    uint16_t *queue = reinterpret_cast<uint16_t *>(res_w + kRes8);
    uint8_t *res_c = reinterpret_cast<uint8_t *>(queue + kQueue);
    uint32_t nres = ws.nres, cnt = ws.cnt;  // survivors waiting in res_*
    // the address is one multiply-add (p.four, which the compiler does not know
    // to be 4), not a shift, a mask and an add on the pipe that bounds the loop:
    // 1 GiB counted 920 -> 899 us
    const uint32_t f1_at = smem_addr(F1);
    WalkRoom room = ws.room;
    auto flush = [&](uint32_t n) {  // resolve the last n (<= 32) of them
        __syncwarp();
        nres -= n;
        const bool on = static_cast<uint32_t>(lane) < n;
        const uint32_t x = nres + (on ? static_cast<uint32_t>(lane) : 0u);
        resolve8<MODE, BATCH>(p, sg, room, res_g[x], res_w[x], res_c[x], on, lane, cnt);
        __syncwarp();
    };
    for (; t < t_end; t += step) {
        const bool more = t + step < t_end;
        if (MODE == OUT_DENSE) fill_none<true>(sg, none, t, lane);
        if (MODE == OUT_BITS) clear_bits(p.f, sg, t, lane);
        __syncwarp();  // the previous tile's readers of stage and queue are done
        // 1. the first filter: one bit per position, first position highest;
        //    a chunk's registers take the next tile's bytes as soon as it is done
        uint32_t acc[2] = {0u, 0u};
        auto chunk = [&](auto cj) {
            constexpr int J = decltype(cj)::value;
            const uint4 cur = r.c[J];
            const uint4 nxt = J < 3 ? r.c[J < 3 ? J + 1 : 3] : r.look;
            uint32_t R[6] = {cur.x, cur.y, cur.z, cur.w, 0u, 0u};
            R[4] = __shfl_sync(kFull, lane == 0 ? nxt.x : cur.x, (lane + 1) & 31);
            R[5] = __shfl_sync(kFull, lane == 0 ? nxt.y : cur.y, (lane + 1) & 31);
            *reinterpret_cast<uint4 *>(stage + J * (kChunk / 4) + 4 * lane) = cur;
            if (J == 3 && lane == 0) *reinterpret_cast<uint4 *>(stage + kTile / 4) = nxt;
            if (more) {
                load_chunk<J>(sg, t + step, pol, lane, r);
                if (J == 3) load_chunk<4>(sg, t + step, pol, lane, r);
            }
            uint32_t win[20];
#pragma unroll
            for (int x = 0; x < 20; ++x)
                win[x] = (x & 3) ? __funnelshift_r(R[x >> 2], R[(x >> 2) + 1], 8 * (x & 3)) : R[x >> 2];
            uint32_t a = acc[J >> 1];
#pragma unroll
            for (int x = 0; x < 16; ++x) {
                // word: the top bits of the 32-bit hash; bit: the first word's
                // product past 32 bits (well mixed, and no shift to get it)
                const uint64_t h = static_cast<uint64_t>(win[x]) * p.m1;
                const uint32_t idx = (static_cast<uint32_t>(h) + win[x + 4] * p.m2) >> 17;
                uint32_t word;
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(word) : "r"(idx * p.four + f1_at));
                const uint32_t b = static_cast<uint32_t>(h >> 32);
                a = __funnelshift_l(__funnelshift_l(word, word, b), a, 1);
            }
            acc[J >> 1] = a;
        };
        chunk(std::integral_constant<int, 0>{});
        chunk(std::integral_constant<int, 1>{});
        chunk(std::integral_constant<int, 2>{});
        chunk(std::integral_constant<int, 3>{});
        __syncwarp();  // stage is written
        const uint32_t g0 = (t - sg.t0) * kTile;
        // 2. survivors, at most kQueue at a time: the second filter (if any),
        //    then the state hash, 32 a round
        uint32_t m[2] = {__brev(acc[0]), __brev(acc[1])};
        auto sample = [&](uint32_t half, uint32_t b) {
            return half * 2u * kChunk + kChunk * (b >> 4) + 16u * static_cast<uint32_t>(lane) + (b & 15u);
        };
        const uint32_t mine = static_cast<uint32_t>(__popc(m[0]) + __popc(m[1]));
        uint32_t at = 0;
        if (!__any_sync(kFull, mine != 0u)) continue;
        const uint32_t below = warp_excl(mine, at, lane);
        if ((at > kTile / 2 || (room.full && at > kFew)) && list_tile<BATCH>(p.f, sg, t, lane)) continue;
        for (uint32_t o = below, first = 0;;) {
            // the lane's survivors o, o + 1, ... of the warp's; the queue holds
            // those from `first` on
            const uint32_t end = first + kQueue;
#pragma unroll
            for (uint32_t half = 0; half < 2; ++half)
                while (m[half] && o < end) {
                    queue[o - first] = static_cast<uint16_t>(sample(half, __ffs(m[half]) - 1));
                    m[half] &= m[half] - 1u;
                    ++o;
                }
            const uint32_t held = at - first < kQueue ? at - first : kQueue;
            __syncwarp();
            for (uint32_t b = 0; b < held; b += 32u) {
                const uint32_t x = b + static_cast<uint32_t>(lane);
                const uint32_t i = queue[x < held ? x : 0u];
                const uint32_t w0 = stage[i >> 2], w1 = stage[(i >> 2) + 1], w2 = stage[(i >> 2) + 2];
                const uint32_t w = __funnelshift_r(w0, w1, 8u * (i & 3u)), c = __funnelshift_r(w1, w2, 8u * (i & 3u));
                bool pass = x < held;
                if (p.f2bytes) {
                    const uint32_t hs = w * kStateHashMul;
                    const uint32_t h6 = w * kFilterHashMul + (c << 16) * kStreamMul2;
                    const uint32_t bs = FS[hs >> 22] >> ((hs >> 17) & 31u);
                    const uint32_t b6 = F2[__umulhi(h6, f2words)] >> ((h6 >> 12) & 31u);
                    pass = pass && ((bs | b6) & 1u);
                }
                const unsigned pm = __ballot_sync(kFull, pass);
                if (!pm) continue;
                if (pass) {
                    const uint32_t o = nres + __popc(pm & lt);
                    res_g[o] = g0 + i;
                    res_w[o] = w;
                    res_c[o] = static_cast<uint8_t>(c);
                }
                nres += __popc(pm);
                if (nres >= 32u) flush(32u);
            }
            __syncwarp();
            first = end;
            if (first >= at) break;
        }
    }
    if (nres) flush(nres);
    ws.nres = nres;
    ws.cnt = cnt;
    ws.room = room;
}

// ---- the kernels -------------------------------------------------------------------

// One text: tiles dealt out warp by warp over the grid.
template <int FORM, int S, int MODE>
__device__ __forceinline__ void stream_text(const StreamParams &p) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    allow_next();  // the walks
    const uint32_t step = gridDim.x * (blockDim.x / 32);
    const uint32_t t = static_cast<uint32_t>(warp) * gridDim.x + blockIdx.x;
    const uint64_t pol = policy_evict_first();
    // 8-bit codes: from the parameters, whose values need no registers; with
    // 2-bit codes the copy spills less
    const Seg own = make_seg(p.f.text, p.f.out, p.f.n);
    using SegRef = typename std::conditional<FORM == 2, const Seg, const Seg &>::type;
    SegRef sg = FORM == 2 ? own : p.sg;
    const int32_t *none = reinterpret_cast<const int32_t *>(smem + p.off_cta + 128u);
    TileRegs r;
    r.look = make_uint4(0u, 0u, 0u, 0u);
    if (t < p.ntiles) load_tile(sg, t, pol, lane, r);
    if (has_bulk(FORM, MODE)) fill_constant(smem + p.off_cta + 128u);
    load_filters(p, smem);
    __syncthreads();  // the filters are in place
    WarpState ws{0u, 0u, {0u, 0u, false, false}};
    if constexpr (FORM == 2)
        tiles2<S, MODE, false>(p, smem, p.off_warp, none, sg, t, p.ntiles, step, pol, r, ws);
    else
        tiles8<MODE, false>(p, smem, p.off_warp, none, sg, t, p.ntiles, step, pol, r, ws);
    if (has_bulk(FORM, MODE) && lane == 0) bulk_wait_all();
    close_room<false>(p.f, ws.room, lane);
    add_count<MODE>(p.f, ws.cnt, lane);
}

template <int S, int MODE>
__global__ void __launch_bounds__(kBlock2, 1) pfac_stream2(const __grid_constant__ StreamParams p) {
    stream_text<2, S, MODE>(p);
}
template <int MODE>
__global__ void __launch_bounds__(kBlock8, 1) pfac_stream8(const __grid_constant__ StreamParams p) {
    stream_text<8, 1, MODE>(p);
}

// A batch: the units (tiles) of the launch's automata, all of one form.  A CTA
// starts with the automaton at its share of the units, so an automaton's
// filters are loaded by about as many CTAs as its share of the work, and goes
// on to the others in turn while they have units left; warps claim blocks of
// consecutive units from the automaton's counter, smaller ones towards its end.
// One launch per form: with every form in one kernel each would take the
// registers of the largest.
constexpr uint32_t kStreamMultiMax = 32;
struct StreamMulti {
    StreamParams a[kStreamMultiMax];
    uint32_t nh;
    uint32_t off_cta, off_warp;
};
static_assert(sizeof(StreamMulti) <= 32764, "kernel parameters are limited to 32764 bytes");

// The text of a batch that unit u belongs to, as a segment from u's tile on.
// The planned list is searched 32 ways: its first 32 samples stay in the lanes
// (sample_items), so up to 1,024 texts take one round of loads, which brings
// the entries themselves.
__device__ __forceinline__ uint32_t list_step(uint32_t n) { return n > 32u ? (n + 31u) / 32u : 1u; }
__device__ __forceinline__ uint32_t sample_items(const Work &wk, int lane) {
    const uint32_t i = static_cast<uint32_t>(lane) * list_step(wk.nlist);
    return i < wk.nlist ? __ldg(&wk.list[i].first_unit) : 0xFFFFFFFFu;
}
template <int MODE>
__device__ __forceinline__ Seg batch_seg(const FilterParams &f, const Work &wk, uint32_t sample, uint32_t u, int lane) {
    uint32_t step = list_step(wk.nlist);
    uint32_t lo = static_cast<uint32_t>(31 - __clz(__ballot_sync(kFull, sample <= u))) * step;  // list[0].first_unit == 0
    uint32_t hi = lo + step < wk.nlist ? lo + step : wk.nlist;
    while (hi - lo > 32u) {
        step = (hi - lo + 31u) / 32u;
        const uint32_t i = lo + static_cast<uint32_t>(lane) * step;
        const bool le = i < hi && __ldg(&wk.list[i].first_unit) <= u;
        lo += static_cast<uint32_t>(31 - __clz(__ballot_sync(kFull, le))) * step;
        hi = lo + step < hi ? lo + step : hi;
    }
    const uint32_t i = lo + static_cast<uint32_t>(lane);
    const uint4 *e = reinterpret_cast<const uint4 *>(wk.list + (i < hi ? i : lo));
    uint4 x = __ldg(e), y = __ldg(e + 1);  // {text_off, len}, {out_off, first_unit, item}
    const int at = 31 - __clz(__ballot_sync(kFull, i < hi && y.z <= u));
    x.x = __shfl_sync(kFull, x.x, at);
    x.y = __shfl_sync(kFull, x.y, at);
    x.z = __shfl_sync(kFull, x.z, at);
    x.w = __shfl_sync(kFull, x.w, at);
    y.z = __shfl_sync(kFull, y.z, at);
    uint64_t ooff = 0;
    if (MODE == OUT_DENSE) ooff = __shfl_sync(kFull, y.x, at) | (static_cast<uint64_t>(__shfl_sync(kFull, y.y, at)) << 32);
    Seg sg = make_seg(f.text + (x.x | (static_cast<uint64_t>(x.y) << 32)), MODE == OUT_DENSE ? f.out + ooff : nullptr,
                      x.z | (static_cast<uint64_t>(x.w) << 32));
    sg.t0 = u - y.z;
    sg.unit0 = u;
    sg.item = lo + static_cast<uint32_t>(at);
    sg.bit0 = MODE == OUT_BITS ? (f.sl.ubase + u) * kTile : 0u;
    return sg;
}

template <int FORM, int S, int MODE>
__device__ __forceinline__ void stream_batch(const StreamMulti &mp) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31;
    const uint64_t pol = policy_evict_first();
    const int32_t *none = reinterpret_cast<const int32_t *>(smem + mp.off_cta + 128u);
    // (dynamic too: a kernel with static shared memory cannot take the most dynamic)
    volatile uint32_t &start = reinterpret_cast<uint32_t *>(smem + mp.off_cta)[0];
    volatile uint32_t &open = reinterpret_cast<uint32_t *>(smem + mp.off_cta)[1];
    // the next form's launch, or the walks: neither reads what this one writes
    // before it has ended
    allow_next();
    if (has_bulk(FORM, MODE)) fill_constant(smem + mp.off_cta + 128u);
    uint64_t total = 0;
    for (uint32_t a = 0; a < mp.nh; ++a) total += __ldg(&mp.a[a].f.batch->units);
    if (threadIdx.x == 0) {
        const uint64_t mine = total * (2u * blockIdx.x + 1u) / (2u * gridDim.x);
        uint64_t sum = 0;
        uint32_t a = 0;
        for (; a + 1u < mp.nh; ++a) {
            sum += __ldg(&mp.a[a].f.batch->units);
            if (mine < sum) break;
        }
        start = a;
    }
    __syncthreads();
    TileRegs r;
    r.look = make_uint4(0u, 0u, 0u, 0u);
    WarpState ws{0u, 0u, {0u, 0u, false, false}};
    const uint32_t first = start;
    for (uint32_t k = 0; k < mp.nh; ++k) {
        const uint32_t a = (first + k) % mp.nh;
        const StreamParams &p = mp.a[a];
        const Work wk = load_work(p.f.batch, p.f.lists, 0u);
        // another automaton than its own: only with units left for a good part
        // of its warps (the filters cost some 5 us), or when too small a share
        // of the units gave it no CTA of its own
        if (threadIdx.x == 0) {
            const uint32_t taken = *reinterpret_cast<volatile unsigned int *>(p.f.counter);
            const uint32_t left = taken < wk.units ? wk.units - taken : 0u;
            const bool owned = static_cast<uint64_t>(wk.units) * gridDim.x >= total;
            open = left > (k > 0u && owned ? gridDim.x * (blockDim.x / 32u) / 4u : 0u) ? 1u : 0u;
        }
        __syncthreads();
        const bool go = open != 0u;  // the same for every thread
        if (go) load_filters(p, smem);
        __syncthreads();
        if (!go) continue;
        // warps on this automaton, about
        const uint32_t share = static_cast<uint32_t>(static_cast<uint64_t>(gridDim.x) * (blockDim.x / 32u) * wk.units / total) + 1u;
        // blocks of four units, one towards the end (1 / 2 / 4 / 6 units: 1,024
        // texts of the benchmark batch in 625 / 578 / 573 / 575 us; shares of what
        // is left, up to 64, scatter the traffic over the whole buffer); the next
        // block is claimed while this one is matched
        auto block = [&](uint32_t seen) { return seen < wk.units && wk.units - seen > 8u * share ? 4u : 1u; };
        const uint32_t sample = sample_items(wk, lane);
        uint32_t blk = block(0u), ahead = 0;
        if (lane == 0) ahead = atomicAdd(p.f.counter, blk);
        for (;;) {
            uint32_t u = __shfl_sync(kFull, ahead, 0);
            if (u >= wk.units) break;
            const uint32_t end = wk.units - u < blk ? wk.units : u + blk;
            blk = block(end);
            if (lane == 0) ahead = atomicAdd(p.f.counter, blk);
            while (u < end) {  // the block's tiles, text by text
                const Seg sg = batch_seg<MODE>(p.f, wk, sample, u, lane);
                const uint64_t tiles = (sg.n + sg.head + kTile - 1u) / kTile;
                const uint32_t n = tiles - sg.t0 < end - u ? static_cast<uint32_t>(tiles - sg.t0) : end - u;
                load_tile(sg, sg.t0, pol, lane, r);
                if constexpr (FORM == 2)
                    tiles2<S, MODE, true>(p, smem, mp.off_warp, none, sg, sg.t0, sg.t0 + n, 1u, pol, r, ws);
                else
                    tiles8<MODE, true>(p, smem, mp.off_warp, none, sg, sg.t0, sg.t0 + n, 1u, pol, r, ws);
                u += n;
            }
        }
        __syncthreads();  // every warp is done with the automaton's filters
    }
    if (has_bulk(FORM, MODE) && lane == 0) bulk_wait_all();
    close_room<true>(mp.a[0].f, ws.room, lane);
    wait_previous();
}

template <int S, int MODE>
__global__ void __launch_bounds__(kBlock2, 1) pfac_stream2_multi(const __grid_constant__ StreamMulti mp) {
    stream_batch<2, S, MODE>(mp);
}
template <int MODE>
__global__ void __launch_bounds__(kBlock8Multi, 1) pfac_stream8_multi(const __grid_constant__ StreamMulti mp) {
    stream_batch<8, 1, MODE>(mp);
}

// ---- the listed walks ----------------------------------------------------------

// Walks wait for dependent loads, so threads count: 12 CTAs of 128 fill the SM
// at 40 registers a thread.
constexpr int kWalkBlock = 128;
constexpr int kWalkCtas = 12;

// One listed walk of text sg: its id at position g.
template <typename GT>
__device__ __forceinline__ int finish_walk(const FilterParams &p, const uint8_t *cls8, const Seg &sg, uint32_t g,
                                           uint32_t e, uint32_t B) {
    const TileText tt = make_text(sg.text, sg.out, sg.n, 0u);
    const uint64_t gi = text_pos(sg, g);
    const uint32_t s = e & 0x7FFFFFFFu;
    // 2-bit codes: the walk so far took the codes for keyword bytes'
    if (s && (B == 8 || bytes_known(p, sg.text, sg.n, gi, p.k + p.k2)))
        return filt::walk_global<GT>(p, cls8, tt, static_cast<int64_t>(gi), s, p.k + p.k2 + (e >> 31));
    return match_at<GT>(p, cls8, tt, gi, B);
}

// How much the launch has to do: walks, and runs of kRun positions (a warp's at a
// time) of the tiles listed whole.
constexpr int kRunPer = 1;
constexpr uint32_t kRun = 32u * kRunPer, kTileRuns = kTile / kRun;
struct Listed {
    uint32_t m, runs;
};
__device__ __forceinline__ Listed listed(const FilterParams &p) {
    const uint4 c = __ldcg(reinterpret_cast<const uint4 *>(p.list_count));  // (read once: what is compared is what is used)
    Listed l;
    l.m = c.y < p.walk_cap ? c.y : p.walk_cap;
    l.runs = (c.z < p.tile_cap ? c.z : p.tile_cap) * kTileRuns;
    return l;
}

// The first run a warp takes: a warp of each CTA first, from the CTA after those
// that take the walks on, so that a few runs go to as many SMs, and to CTAs that
// started early.  (16 MiB of ACGT, two tiles listed: 4 runs a CTA from the first
// CTA on 67 us a call, one from the first / the last / this one 46.5 / 44.9 / 43.3.)
__device__ __forceinline__ uint32_t first_run(const Listed &l) {
    const uint32_t after = (l.m + blockDim.x - 1u) / blockDim.x % gridDim.x;
    return (threadIdx.x / 32u) * gridDim.x + (blockIdx.x >= after ? blockIdx.x - after : blockIdx.x + gridDim.x - after);
}

// One warp: the kRun positions of a listed tile from g on (a multiple of kRun).
template <int B, typename GT, int MODE>
__device__ __forceinline__ void tile_run(const FilterParams &p, const uint8_t *cls8, const Seg &sg, uint32_t g,
                                         uint32_t &cnt, int lane) {
    const uint64_t g0 = text_pos(sg, g + static_cast<uint32_t>(lane));
    uint32_t c[kRunPer + 1];
    bool in[kRunPer + 1];
    load_run<kRunPer>(sg.text, sg.n, g0, lane, c, in);
    match_run<B, GT, kRunPer, false>(p, cls8, make_text(sg.text, sg.out, sg.n, 0u), g0, lane, c, in, [&](int j, int r) {
        if (MODE != OUT_BITS) {
            put_id<MODE>(p, sg, g + 32u * j + static_cast<uint32_t>(lane), r, cnt);
            return;
        }
        const uint32_t b = g + 32u * j + sg.bit0, bits = __ballot_sync(kFull, r >= 0);
        if (r >= 0) p.bo.ids[b + static_cast<uint32_t>(lane)] = r;
        if (lane == 0 && bits) {
            p.bo.bits[b >> 5] = bits;
            atomicAdd(p.bo.counts + b / kTile, static_cast<uint32_t>(__popc(bits)));
        }
    });
}

template <int B, typename GT, int MODE>
__global__ void __launch_bounds__(kWalkBlock, kWalkCtas) pfac_stream_walks(const __grid_constant__ FilterParams p) {
    __shared__ uint8_t cls8[256];
    const int lane = threadIdx.x & 31;
    allow_next();  // the lists' scan
    wait_previous();
    const Listed l = listed(p);
    const bool idle = blockIdx.x * blockDim.x >= l.m;
    if (idle && l.runs == 0u) return;
    const uint32_t first = l.runs ? first_run(l) : 0u, *tiles = reinterpret_cast<const uint32_t *>(p.walks + p.walk_cap);
    if (idle && first % gridDim.x >= l.runs) return;
    // (2-bit codes: the first tile's number is on its way meanwhile; with 8-bit
    // codes it would cost the walks' loop spills)
    uint32_t t = B == 2 && first < l.runs ? tiles[first / kTileRuns] : 0u;
    for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x) cls8[i] = __ldg(p.cls8g + i);
    __syncthreads();
    const Seg sg = make_seg(p.text, p.out, p.n);
    uint32_t cnt = 0;
    // (not by the read-only path: written by the launch before)
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < l.m; j += gridDim.x * blockDim.x) {
        const uint2 e = p.walks[j];
        if (e.x != 0xFFFFFFFFu) put_id<MODE>(p, sg, e.x, finish_walk<GT>(p, cls8, sg, e.x, e.y, B), cnt);
    }
    for (uint32_t j = first; j < l.runs;) {
        if (B != 2) t = tiles[j / kTileRuns];
        tile_run<B, GT, MODE>(p, cls8, sg, t * kTile + kRun * (j % kTileRuns), cnt, lane);
        j += gridDim.x * (blockDim.x / 32u);
        if (B == 2 && j < l.runs) t = tiles[j / kTileRuns];
    }
    add_count<MODE>(p, cnt, lane);
}

// A batch's walks: the automata's parameters (a[0 .. nh), in the order of the
// entries' automaton numbers) and byte tables in shared memory.
struct WalkMulti {
    FilterParams a[kStreamMultiMax];
    uint32_t nh;
};
static_assert(sizeof(WalkMulti) <= 32764, "kernel parameters are limited to 32764 bytes");

// The segment of an entry's unit.
template <int MODE>
__device__ __forceinline__ Seg entry_seg(const FilterParams &p, const uint4 &e) {
    const Work wk = load_work(p.batch, p.lists, 0u);
    const uint4 *q = reinterpret_cast<const uint4 *>(wk.list + e.w);
    const uint4 x = __ldg(q), y = __ldg(q + 1);
    Seg sg = make_seg(p.text + (x.x | (static_cast<uint64_t>(x.y) << 32)),
                      MODE == OUT_DENSE ? p.out + (y.x | (static_cast<uint64_t>(y.y) << 32)) : nullptr,
                      x.z | (static_cast<uint64_t>(x.w) << 32));
    sg.t0 = e.x - y.z;
    sg.bit0 = MODE == OUT_BITS ? (p.sl.ubase + e.x) * kTile : 0u;
    return sg;
}

// An entry's walk, and tile_run of an entry's tile: out of line, as the copies
// for every kind of automaton would spill.
template <typename GT, int MODE>
static __device__ __noinline__ void entry_walk(const FilterParams &p, const uint8_t *cls8, const uint4 e, uint32_t g) {
    uint32_t cnt = 0;
    const Seg sg = entry_seg<MODE>(p, e);
    put_id<MODE>(p, sg, g, finish_walk<GT>(p, cls8, sg, g, e.y, p.kind >> 8), cnt);
}
template <int B, typename GT, int MODE>
static __device__ __noinline__ void entry_run(const FilterParams &p, const uint8_t *cls8, const uint4 e, uint32_t g,
                                              int lane) {
    uint32_t cnt = 0;
    tile_run<B, GT, MODE>(p, cls8, entry_seg<MODE>(p, e), g, cnt, lane);
}

template <int MODE>
__global__ void __launch_bounds__(kWalkBlock, 8) pfac_stream_walks_multi(const __grid_constant__ WalkMulti mp) {
    extern __shared__ __align__(16) uint8_t msm[];
    const int lane = threadIdx.x & 31;
    allow_next();
    wait_previous();
    const Listed l = listed(mp.a[0]);
    const bool idle = blockIdx.x * blockDim.x >= l.m;
    if (idle && (l.runs == 0u || first_run(l) % gridDim.x >= l.runs)) return;
    FilterParams *ps = reinterpret_cast<FilterParams *>(msm);
    uint8_t *cls = msm + mp.nh * sizeof(FilterParams);
    for (uint32_t i = threadIdx.x; i < mp.nh * static_cast<uint32_t>(sizeof(FilterParams) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t *>(ps)[i] = reinterpret_cast<const uint32_t *>(mp.a)[i];
    for (uint32_t i = threadIdx.x; i < mp.nh * 256u; i += blockDim.x) cls[i] = __ldg(mp.a[i >> 8].cls8g + (i & 255u));
    __syncthreads();
    uint32_t cnt = 0;
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < l.m; j += gridDim.x * blockDim.x) {
        const uint4 e = mp.a[0].walks4[j];
        if (e.x == 0xFFFFFFFFu) continue;
        const uint32_t a = e.z >> 11, g = e.z & (kTile - 1u);
        const FilterParams &p = ps[a];
        if ((p.kind & 0xFFu) == 16u)
            entry_walk<int16_t, MODE>(p, cls + 256u * a, e, g);
        else
            entry_walk<int32_t, MODE>(p, cls + 256u * a, e, g);
    }
    for (uint32_t j = first_run(l); j < l.runs; j += gridDim.x * (blockDim.x / 32u)) {
        const uint4 e = mp.a[0].walks4[mp.a[0].walk_cap + j / kTileRuns];
        const uint32_t a = e.z >> 11, g = kRun * (j % kTileRuns);
        const FilterParams &p = ps[a];
        const uint8_t *cls8 = cls + 256u * a;
        if ((p.kind >> 8) == 2u) {
            if ((p.kind & 0xFFu) == 16u)
                entry_run<2, int16_t, MODE>(p, cls8, e, g, lane);
            else
                entry_run<2, int32_t, MODE>(p, cls8, e, g, lane);
        } else if ((p.kind & 0xFFu) == 16u) {
            entry_run<8, int16_t, MODE>(p, cls8, e, g, lane);
        } else {
            entry_run<8, int32_t, MODE>(p, cls8, e, g, lane);
        }
    }
}

// ---- launches --------------------------------------------------------------------

template <auto Kernel, typename P>
cudaError_t launch_form(const P &p, uint32_t grid, uint32_t block, uint32_t smem, int max_smem, cudaStream_t stream,
                        bool next = false) {
    static std::atomic<uint64_t> configured{0};  // bit d: device d (as many as filter_device_shape knows)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!((configured.load() >> dev) & 1u)) {
        e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
        if (e != cudaSuccess) return e;
        configured.fetch_or(1ull << dev);
    }
    if (next) return launch_next(Kernel, grid, block, smem, stream, p);
    Kernel<<<grid, block, smem, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_stream2(OutMode mode, const StreamParams &p, uint32_t step, uint32_t grid, uint32_t smem,
                           int max_smem, cudaStream_t stream);
cudaError_t launch_stream8(OutMode mode, const StreamParams &p, uint32_t grid, uint32_t smem, int max_smem,
                           cudaStream_t stream);
cudaError_t launch_stream2_multi(OutMode mode, const StreamMulti &mp, uint32_t step, uint32_t grid, uint32_t smem,
                                 int max_smem, cudaStream_t stream, bool next);
cudaError_t launch_stream8_multi(OutMode mode, const StreamMulti &mp, uint32_t grid, uint32_t smem, int max_smem,
                                 cudaStream_t stream, bool next);

}  // namespace strm
}  // namespace pfac
