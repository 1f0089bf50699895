// The streaming form of the matching kernel for one long text, sm_103a, in two
// launches:
//   pfac_stream2 / pfac_stream8   read the text once, straight into registers,
//       test it against a root filter in shared memory, resolve the few
//       positions that pass with one or two table loads, write the -1 of every
//       other position, and list the walks that go further;
//   pfac_stream_walks             one thread per listed walk.
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
// counts by instruction issue (0.29 against 0.88 ms); with 8-bit codes both by
// the filter's lookups, 16 a lane and chunk, about 8 instructions each (count
// 0.88 against 2.15 ms, where every tenth position went through a global list).
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

constexpr int kBlock = 768;
constexpr int kWarps = kBlock / 32;
constexpr uint32_t kTile = kStreamTile;  // positions a warp takes at a time
constexpr uint32_t kUnit = kStreamUnit;  // positions per unit of a walk entry
constexpr uint32_t kChunk = 512;         // positions per warp-wide 16-byte load
constexpr uint32_t kQueue = 256;         // survivors of a tile kept in shared memory at a time
constexpr uint32_t kNone = 1024;          // ids of -1 in shared memory
constexpr uint32_t kRes2 = 160;          // 2-bit codes: candidates waiting to be resolved (31 + 4 * 32 at most)
constexpr uint32_t kRes8 = 64;           // 8-bit codes: survivors waiting (31 + 32 at most)
constexpr uint32_t kWarpBytes2 = kTile / 4 + 16 + 2 * kQueue + 8 * kRes2;
constexpr uint32_t kWarpBytes8 = kTile + 16 + 2 * kQueue + 9 * kRes8;
static_assert(kWarpBytes2 % 16 == 0 && kWarpBytes8 % 16 == 0, "warp areas start on 16 bytes");

struct StreamParams {
    FilterParams f;        // tables, text, outputs, walk list (walks, walk_cap, list_count[1])
    const uint32_t *F1;    // root filter, f1bytes
    const uint32_t *F2;    // second filter (f2bytes; 0: none), with 8-bit codes then its short-keyword part
    uint32_t f1bytes, f2bytes;
    uint32_t ntiles;
    uint32_t in_lo, in_hi;  // the tiles wholly inside the text, with the 16 bytes after them
    uint32_t head;         // text - f.gbase
    uint32_t m1, m2;       // 8-bit codes: multipliers of the window's words
    uint32_t l2shift;      // 2-bit codes: left shift that drops the codes past the second filter's window
    uint32_t off_none, off_warp;
};

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
    uint32_t v[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (uint32_t j = 0; j < 16; ++j)
        if (off + j >= head && off + j < end) v[j >> 2] |= static_cast<uint32_t>(__ldg(gbase + off + j)) << (8u * (j & 3u));
    return make_uint4(v[0], v[1], v[2], v[3]);
}

// A tile's registers: lane l's 16 bytes of chunks 0-3, and (lane 0) the 16
// bytes after the tile.
struct TileRegs {
    uint4 c[4];
    uint4 look;
};

// The loads of a warp's tiles: lane l's address in tile 0.
struct Loader {
    const uint8_t *base;
    uint64_t pol;
    // chunk C (4: the look-ahead) of tile t (< ntiles)
    template <int C>
    __device__ __forceinline__ void load(const StreamParams &p, uint32_t t, int lane, TileRegs &r) const {
        const uint64_t lo = static_cast<uint64_t>(t) * kTile;
        if (t >= p.in_lo && t < p.in_hi) {
            if constexpr (C < 4)
                r.c[C] = ldg_stream(base + lo + static_cast<uint32_t>(C) * kChunk, pol);
            else if (lane == 0)
                r.look = ldg_stream(base + lo + kTile, pol);
        } else {
            const uint64_t end = p.head + p.f.n;
            if constexpr (C < 4)
                r.c[C] = load_fringe(p.f.gbase, lo + static_cast<uint32_t>(C) * kChunk + 16u * static_cast<uint32_t>(lane),
                                     p.head, end);
            else if (lane == 0)
                r.look = load_fringe(p.f.gbase, lo + kTile, p.head, end);
        }
    }
};

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

// An id found at text position gi.
template <int MODE>
__device__ __forceinline__ void put_id(const FilterParams &p, uint64_t gi, int r, uint32_t &cnt) {
    if (r < 0) return;
    if (MODE == OUT_DENSE) {
        p.out[gi] = r;
    } else if (MODE == OUT_COUNT) {
        ++cnt;
    } else {
        const uint32_t g = static_cast<uint32_t>(gi) + p.bits_head;
        p.bo.ids[g] = r;
        atomicOr(p.bo.bits + (g >> 5), 1u << (g & 31u));
        atomicAdd(p.bo.counts + g / kTile, 1u);
    }
}

// Positions are named by g, their index from gbase (text position + head).
// Walk-list entry: {g, state | d << 31}: the walk goes on from the state with
// the byte k + k2 + d after the position; state 0: not resolved at all.  An
// empty entry's g is 0xFFFFFFFF.

// Walks to the walk list (all lanes of the warp; want: this lane has one).
// Space is reserved in chunks; when one runs out its rest takes the first
// walks.  False for a lane whose walk found no room (the list is full).
struct WalkRoom {
    uint32_t next, end;  // the warp's chunk
    bool full;           // nothing more to reserve (the counter is left alone then)
};
__device__ __forceinline__ bool push_walk(const StreamParams &p, WalkRoom &room, bool want, uint2 e, int lane) {
    const unsigned m = __ballot_sync(kFull, want);
    if (!m) return true;
    const uint32_t need = __popc(m), rank = __popc(m & ((1u << lane) - 1u)), rest = room.end - room.next;
    uint32_t slot = room.next + rank;
    bool stored = want;
    if (rest < need) {
        uint32_t base = p.f.walk_cap, end = p.f.walk_cap;
        if (!room.full) {
            if (lane == 0) base = atomicAdd(p.f.list_count + 1, kWalkChunkEntries);
            base = __shfl_sync(kFull, base, 0);
            room.full = base >= p.f.walk_cap || p.f.walk_cap - base <= kWalkChunkEntries;
            end = room.full ? p.f.walk_cap : base + kWalkChunkEntries;
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
    if (stored) p.f.walks[slot] = e;
    return !want || stored;
}

// The warp's unused walk-list entries are empty.
__device__ __forceinline__ void close_room(const StreamParams &p, const WalkRoom &room, int lane) {
    for (uint32_t j = room.next + static_cast<uint32_t>(lane); j < room.end; j += 32u)
        p.f.walks[j] = make_uint2(0xFFFFFFFFu, 0u);
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
__device__ __forceinline__ void fill_none(const StreamParams &p, const int32_t *none, uint32_t t, int lane) {
    const int64_t lo = static_cast<int64_t>(static_cast<uint64_t>(t) * kTile) - p.head;
    int32_t *o = p.f.out + lo;
    if (t >= p.in_lo && t < p.in_hi) {
        if (BULK && p.f.vec_ok) {
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
            if (g >= 0 && g < static_cast<int64_t>(p.f.n)) o[i] = -1;
        }
    }
}

// OUT_BITS: no bits and no matches yet in tile t.
__device__ __forceinline__ void clear_bits(const StreamParams &p, uint32_t t, int lane) {
    reinterpret_cast<uint2 *>(p.f.bo.bits + static_cast<size_t>(t) * (kTile / 32u))[lane] = make_uint2(0u, 0u);
    if (lane == 0) p.f.bo.counts[t] = 0u;
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
__device__ __forceinline__ void settle_here(const StreamParams &p, uint32_t g, uint32_t B, uint32_t &cnt) {
    const TileText tt = make_text(p.f.text, p.f.out, p.f.n, 0u);
    const uint64_t gi = static_cast<uint64_t>(g) - p.head;
    const int r = (p.f.kind & 0xFFu) == 16u ? match_at_far<int16_t>(p.f, p.f.cls8g, tt, gi, B)
                                            : match_at_far<int32_t>(p.f, p.f.cls8g, tt, gi, B);
    put_id<MODE>(p.f, gi, r, cnt);
}

// Walks (want: this lane has one) to the list, or settled here when it is full.
template <int B, int MODE>
__device__ __forceinline__ void list_walk(const StreamParams &p, WalkRoom &room, bool want, uint2 e, int lane,
                                          uint32_t &cnt) {
    const bool stored = push_walk(p, room, want, e, lane);
    if (!room.full || __all_sync(kFull, stored)) return;
    fill_done<MODE, B == 8>(true, lane);
    if (!stored) settle_here<MODE>(p, e.x, B, cnt);
}

// One CTA's filters into shared memory (all threads; a CTA barrier follows).
__device__ __forceinline__ void load_filters(const StreamParams &p, uint8_t *smem) {
    uint4 *d = reinterpret_cast<uint4 *>(smem);
    const uint4 *a = reinterpret_cast<const uint4 *>(p.F1), *b = reinterpret_cast<const uint4 *>(p.F2);
    const uint32_t na = p.f1bytes >> 4, nb = p.f2bytes >> 4;
    int4 *none = reinterpret_cast<int4 *>(smem + p.off_none);
    for (uint32_t i = threadIdx.x; i < kNone / 4u; i += kBlock) none[i] = make_int4(-1, -1, -1, -1);
    fence_proxy_async_smem();  // read by bulk stores
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < na; i += kBlock) d[i] = __ldg(a + i);
    for (uint32_t i = threadIdx.x; i < nb; i += kBlock) d[na + i] = __ldg(b + i);
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

// The 16 codes from tile position i on, from the tile's packed codes.
__device__ __forceinline__ uint32_t codes_at(const uint32_t *packed, uint32_t i) {
    return __funnelshift_r(packed[i >> 4], packed[(i >> 4) + 1u], 2u * (i & 15u));
}

// Whether the `need` (<= 16) bytes from text position gi on are inside the
// text and all in keywords (cls8: the byte table).
__device__ __forceinline__ bool bytes_known(const FilterParams &p, const uint8_t *cls8, uint64_t gi, uint32_t need) {
    if (gi + need > p.n) return false;
    uint32_t b[16], bad = 0;
#pragma unroll
    for (uint32_t j = 0; j < 16; ++j) b[j] = j < need ? __ldg(p.text + gi + j) : 0u;  // all in flight together
#pragma unroll
    for (uint32_t j = 0; j < 16; ++j) bad |= j < need && cls8[b[j]] == 0xFFu ? 1u : 0u;
    return bad == 0;
}

// A round of candidates (all lanes; on: this lane has one: position g and the
// 16 codes w from it): window table, stride table, then out or to the walk
// list.  The codes may be those of bytes in no keyword, or of bytes past the
// text: a keyword that ends before such a byte is on the walk of the codes too,
// so a position without a result has none; one with a result has its bytes
// looked at, and a walk's bytes are looked at when it goes on.
template <int MODE>
__device__ __forceinline__ void resolve2(const StreamParams &p, WalkRoom &room, uint32_t g, uint32_t w, bool on,
                                         int lane, uint32_t &cnt) {
    const FilterParams &f = p.f;
    const uint64_t gi = static_cast<uint64_t>(g) - p.head;  // before the text wraps
    bool walk = false;
    uint32_t s = 0;
    int r = -1;
    if (on && gi < f.n) {
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
        if (r >= 0 && !bytes_known(f, f.cls8g, gi, f.k + f.k2)) {
            walk = true;
            s = 0;
            r = -1;
        }
    }
    fill_done<MODE, false>(r >= 0, lane);
    put_id<MODE>(f, gi, r, cnt);
    list_walk<2, MODE>(p, room, walk, make_uint2(g, s), lane, cnt);
}

template <int S, int MODE>
__global__ void __launch_bounds__(kBlock, 1) pfac_stream2(const __grid_constant__ StreamParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t step = gridDim.x * kWarps, lt = (1u << lane) - 1u;
    uint32_t t = static_cast<uint32_t>(warp) * gridDim.x + blockIdx.x;
    const Loader ld{p.f.gbase + 16u * static_cast<uint32_t>(lane), policy_evict_first()};
    TileRegs r;
    r.look = make_uint4(0u, 0u, 0u, 0u);
    auto load = [&](uint32_t u) {
        ld.load<0>(p, u, lane, r);
        ld.load<1>(p, u, lane, r);
        ld.load<2>(p, u, lane, r);
        ld.load<3>(p, u, lane, r);
        ld.load<4>(p, u, lane, r);
    };
    if (t < p.ntiles) load(t);
    load_filters(p, smem);
    const uint32_t *F1 = reinterpret_cast<const uint32_t *>(smem);
    const uint32_t *F2 = reinterpret_cast<const uint32_t *>(smem + p.f1bytes);
    uint32_t *packed = reinterpret_cast<uint32_t *>(smem + p.off_warp + static_cast<uint32_t>(warp) * kWarpBytes2);
    uint2 *res = reinterpret_cast<uint2 *>(packed + kTile / 16 + 4);
    uint16_t *queue = reinterpret_cast<uint16_t *>(res + kRes2);
    const int32_t *none = reinterpret_cast<const int32_t *>(smem + p.off_none);
    WalkRoom room{0u, 0u, false};
    uint32_t cnt = 0, nres = 0;  // candidates waiting in res: {g, codes}
    auto flush = [&](uint32_t n) {  // resolve the last n (<= 32) of them
        __syncwarp();
        nres -= n;
        const bool on = static_cast<uint32_t>(lane) < n;
        const uint2 e = res[nres + (on ? static_cast<uint32_t>(lane) : 0u)];
        resolve2<MODE>(p, room, e.x, e.y, on, lane, cnt);
        __syncwarp();
    };
    __syncthreads();  // the filters are in place
    for (; t < p.ntiles; t += step) {
        // 1. codes; the registers are free for the next tile's loads
        uint32_t c[5];
#pragma unroll
        for (int j = 0; j < 4; ++j) c[j] = codes16(r.c[j]);
        c[4] = codes16(r.look);
        if (t + step < p.ntiles) load(t + step);
        __syncwarp();  // the previous tile's readers of packed and queue are done
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) packed[32u * j + static_cast<uint32_t>(lane)] = c[j];
        if (lane == 0) packed[128] = c[4];
        if (MODE == OUT_DENSE) fill_none<false>(p, none, t, lane);
        if (MODE == OUT_BITS) clear_bits(p, t, lane);

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
        const uint32_t g0 = t * kTile;
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
            if (total > kQueue / S) {
                // a tile dense in survivors: all of them to the walk list,
                // unresolved, in one reservation (the positions before or
                // past the text as empty entries)
                uint32_t base = p.f.walk_cap;
                const uint32_t need = total * S;
                if (!room.full) {
                    if (lane == 0) base = atomicAdd(p.f.list_count + 1, need);
                    base = __shfl_sync(kFull, base, 0);
                    room.full = base >= p.f.walk_cap || p.f.walk_cap - base < need;
                    if (base > p.f.walk_cap) base = p.f.walk_cap;
                }
                uint32_t all = 0, o = base + S * warp_excl(static_cast<uint32_t>(__popc(m)), all, lane);
                fill_done<MODE, false>(true, lane);
                for (; m; m &= m - 1u) {
                    const uint32_t g = g0 + sample(__ffs(m) - 1);
#pragma unroll 1
                    for (uint32_t x = 0; x < S; ++x, ++o) {
                        const bool in = static_cast<uint64_t>(g - x) - p.head < p.f.n;
                        if (o < p.f.walk_cap)
                            p.f.walks[o] = make_uint2(in ? g - x : 0xFFFFFFFFu, 0u);
                        else if (in)
                            settle_here<MODE>(p, g - x, 2u, cnt);
                    }
                }
                __syncwarp();
                continue;
            }
            if (S > 1 && p.f2bytes) {
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
    }
    if (nres) flush(nres);
    if (MODE == OUT_DENSE && lane == 0) bulk_wait_all();
    close_room(p, room, lane);
    add_count<MODE>(p.f, cnt, lane);
}

// ---- 8-bit codes -------------------------------------------------------------

// A round of survivors (all lanes; on: this lane has one: position g, its
// window's four bytes w and the byte c after them): the state hash, for a
// branching state the first goto step, then out or to the walk list.
template <int MODE>
__device__ __forceinline__ void resolve8(const StreamParams &p, WalkRoom &room, uint32_t g, uint32_t w, uint32_t c,
                                         bool on, int lane, uint32_t &cnt) {
    const FilterParams &f = p.f;
    const uint64_t gi = static_cast<uint64_t>(g) - p.head;
    // windows past the text end (or before its start, which wraps) hold no keyword
    on = on && gi < f.n && gi + f.k <= f.n;
    bool c_ok = gi + f.k < f.n;
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
    put_id<MODE>(f, gi, r, cnt);
    list_walk<8, MODE>(p, room, walk, make_uint2(g, s | (1u << 31)), lane, cnt);
}

// One warp's 8-bit-code tile: its bytes, survivors and their resolution.
template <int MODE>
__global__ void __launch_bounds__(kBlock, 1) pfac_stream8(const __grid_constant__ StreamParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t step = gridDim.x * kWarps, lt = (1u << lane) - 1u;
    uint32_t t = static_cast<uint32_t>(warp) * gridDim.x + blockIdx.x;
    const Loader ld{p.f.gbase + 16u * static_cast<uint32_t>(lane), policy_evict_first()};
    TileRegs r;
    r.look = make_uint4(0u, 0u, 0u, 0u);
    if (t < p.ntiles) {
        ld.load<0>(p, t, lane, r);
        ld.load<1>(p, t, lane, r);
        ld.load<2>(p, t, lane, r);
        ld.load<3>(p, t, lane, r);
        ld.load<4>(p, t, lane, r);
    }
    load_filters(p, smem);
    const uint32_t *F1 = reinterpret_cast<const uint32_t *>(smem);
    const uint32_t *F2 = reinterpret_cast<const uint32_t *>(smem + p.f1bytes);
    const uint32_t f2words = (p.f2bytes - kStreamShortBytes) >> 2;  // only used with a second filter
    const uint32_t *FS = F2 + f2words;
    uint32_t *stage = reinterpret_cast<uint32_t *>(smem + p.off_warp + static_cast<uint32_t>(warp) * kWarpBytes8);
    uint32_t *res_g = stage + kTile / 4 + 4, *res_w = res_g + kRes8;
    uint16_t *queue = reinterpret_cast<uint16_t *>(res_w + kRes8);
    uint8_t *res_c = reinterpret_cast<uint8_t *>(queue + kQueue);
    const int32_t *none = reinterpret_cast<const int32_t *>(smem + p.off_none);
    WalkRoom room{0u, 0u, false};
    uint32_t cnt = 0, nres = 0;  // survivors waiting in res_*
    auto flush = [&](uint32_t n) {  // resolve the last n (<= 32) of them
        __syncwarp();
        nres -= n;
        const bool on = static_cast<uint32_t>(lane) < n;
        const uint32_t x = nres + (on ? static_cast<uint32_t>(lane) : 0u);
        resolve8<MODE>(p, room, res_g[x], res_w[x], res_c[x], on, lane, cnt);
        __syncwarp();
    };
    __syncthreads();  // the filters are in place
    for (; t < p.ntiles; t += step) {
        const bool more = t + step < p.ntiles;
        if (MODE == OUT_DENSE) fill_none<true>(p, none, t, lane);
        if (MODE == OUT_BITS) clear_bits(p, t, lane);
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
                ld.load<J>(p, t + step, lane, r);
                if (J == 3) ld.load<4>(p, t + step, lane, r);
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
                const uint32_t word = F1[(static_cast<uint32_t>(h) + win[x + 4] * p.m2) >> 17];
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
        const uint32_t g0 = t * kTile;
        // 2. survivors, at most kQueue at a time: the second filter (if any),
        //    then the state hash, 32 a round
        uint32_t m[2] = {__brev(acc[0]), __brev(acc[1])};
        auto sample = [&](uint32_t half, uint32_t b) {
            return half * 2u * kChunk + kChunk * (b >> 4) + 16u * static_cast<uint32_t>(lane) + (b & 15u);
        };
        const uint32_t mine = static_cast<uint32_t>(__popc(m[0]) + __popc(m[1]));
        uint32_t at = 0;
        if (!__any_sync(kFull, mine != 0u)) continue;
        for (uint32_t o = warp_excl(mine, at, lane), first = 0;;) {
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
    if (MODE == OUT_DENSE && lane == 0) bulk_wait_all();
    close_room(p, room, lane);
    add_count<MODE>(p.f, cnt, lane);
}

// ---- the listed walks ----------------------------------------------------------

// Walks wait for dependent loads, so threads count: 12 CTAs of 128 fill the SM
// at 40 registers a thread.
constexpr int kWalkBlock = 128;
constexpr int kWalkCtas = 12;

template <int B, typename GT, int MODE>
__global__ void __launch_bounds__(kWalkBlock, kWalkCtas) pfac_stream_walks(const __grid_constant__ FilterParams p) {
    __shared__ uint8_t cls8[256];
    const int lane = threadIdx.x & 31;
    const uint32_t listed = *reinterpret_cast<volatile const unsigned int *>(p.list_count + 1);
    const uint32_t m = listed < p.walk_cap ? listed : p.walk_cap;
    if (blockIdx.x * blockDim.x >= m) return;
    for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x) cls8[i] = __ldg(p.cls8g + i);
    __syncthreads();
    const uint64_t head = reinterpret_cast<uintptr_t>(p.text) & 15u;
    const TileText tt = make_text(p.text, p.out, p.n, 0u);
    uint32_t cnt = 0;
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < m; j += gridDim.x * blockDim.x) {
        const uint2 e = __ldg(p.walks + j);
        if (e.x == 0xFFFFFFFFu) continue;
        const uint64_t gi = static_cast<uint64_t>(e.x) - head;
        const uint32_t s = e.y & 0x7FFFFFFFu;
        int r;
        // 2-bit codes: the walk so far took the codes for keyword bytes'
        if (s && (B == 8 || bytes_known(p, cls8, gi, p.k + p.k2)))
            r = filt::walk_global<GT>(p, cls8, tt, static_cast<int64_t>(gi), s, p.k + p.k2 + (e.y >> 31));
        else
            r = match_at<GT>(p, cls8, tt, gi, B);
        put_id<MODE>(p, gi, r, cnt);
    }
    add_count<MODE>(p, cnt, lane);
}

// ---- launches --------------------------------------------------------------------

template <void (*Kernel)(const StreamParams)>
cudaError_t launch_form(const StreamParams &p, uint32_t grid, uint32_t smem, int max_smem, cudaStream_t stream) {
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
    Kernel<<<grid, kBlock, smem, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_stream2(OutMode mode, const StreamParams &p, uint32_t step, uint32_t grid, uint32_t smem,
                           int max_smem, cudaStream_t stream);
cudaError_t launch_stream8(OutMode mode, const StreamParams &p, uint32_t grid, uint32_t smem, int max_smem,
                           cudaStream_t stream);

}  // namespace strm
}  // namespace pfac
