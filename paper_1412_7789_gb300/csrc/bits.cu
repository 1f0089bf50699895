// Compacted and full output of one text from a bit per position: after the
// short-text or the streaming form has left, for every position with a match,
// its bit and its id (OUT_BITS), the lists are made here:
//   streaming form, compacted:  the scan of the tiles' match counts
//                               (compact.cu), then bits_gather;
//   streaming form, full:       full_bits_count (per tile, the occurrences its
//                               results stand for), their scan, bits_gather;
//   short texts:                bits_gather alone (full: full_bits_count
//                               first), each CTA adding up what lies before
//                               its own tiles.
// bits_gather takes a tile with one warp: the tile's positions with a match go
// to shared memory in ascending order, then one lane takes each, so a tile
// dense in matches costs no more per match than a sparse one (the per-tile
// slots and dense fallback of compact.cu rank 32 matches at most, and a fuller
// tile's positions are all read back).
#include <cuda_runtime.h>

#include <cstdint>

#include "pfac_device.cuh"

namespace pfac {

namespace {

// (What an earlier launch wrote is read with plain loads: these kernels may
// have started before it ended.)
constexpr unsigned kFull = 0xffffffffu;
constexpr int kThreads = 256;
constexpr uint32_t kWarps = kThreads / 32;
constexpr uint32_t kTile = kStreamTile;
constexpr uint32_t kWords = kTile / 32;  // bit words of a tile: two a lane

struct BitsParams {
    const uint32_t *bits;
    const int32_t *ids;
    uint32_t words, ntiles;  // bit words written, tiles
    uint32_t head;           // bit position of the text's first byte
    const uint32_t *counts;             // per tile: what it adds to the list (small, compacted: null)
    const unsigned long long *prefix;   // its exclusive sum (small: null)
    uint32_t *fcounts;                  // full_bits_count's output
    // full output
    const uint4 *rec;
    const uint32_t *dups;
    uint32_t max_clen, nkw;
    unsigned int *err;
    CompactOut out;
};

// A lane's two bit words of tile t (words past the last are 0).
__device__ __forceinline__ uint2 tile_bits(const BitsParams &p, uint32_t t, int lane) {
    const uint32_t w = t * kWords + 2u * static_cast<uint32_t>(lane);
    uint2 b = make_uint2(0u, 0u);
    if (w < p.words) b.x = p.bits[w];
    if (w + 1u < p.words) b.y = p.bits[w + 1u];
    return b;
}

// The tile positions of the set bits, in ascending order, to list; returns
// how many there are.
__device__ __forceinline__ uint32_t list_bits(uint2 b, uint16_t *list, int lane) {
    const uint32_t c = static_cast<uint32_t>(__popc(b.x) + __popc(b.y));
    uint32_t inc = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, inc, d);
        if (lane >= d) inc += y;
    }
    const uint32_t total = __shfl_sync(kFull, inc, 31);
    uint32_t o = inc - c;
    __syncwarp();  // the previous tile's readers are done
    for (uint32_t m = b.x; m; m &= m - 1u) list[o++] = static_cast<uint16_t>(64u * lane + (__ffs(m) - 1));
    for (uint32_t m = b.y; m; m &= m - 1u) list[o++] = static_cast<uint16_t>(64u * lane + 32u + (__ffs(m) - 1));
    __syncwarp();
    return total;
}

// One warp: the `total` matches listed of the tile whose bits start at g0, from
// index at of the list on; p0: the text position of its first bit (before the
// text wraps).  R rounds of 32 matches at a time, their ids in flight together.
template <uint32_t R>
__device__ __forceinline__ void put_compact(const BitsParams &p, size_t g0, uint32_t p0, uint32_t total,
                                            unsigned long long at, const uint16_t *list, int lane) {
    for (uint32_t k0 = 0; k0 < total; k0 += 32u * R) {
        uint32_t i[R], id[R];
#pragma unroll
        for (uint32_t j = 0; j < R; ++j) {
            const uint32_t k = k0 + 32u * j + static_cast<uint32_t>(lane);
            i[j] = k < total ? list[k] : 0u;
            id[j] = k < total ? static_cast<uint32_t>(p.ids[g0 + i[j]]) : 0u;
        }
#pragma unroll
        for (uint32_t j = 0; j < R; ++j) {
            const uint32_t k = k0 + 32u * j + static_cast<uint32_t>(lane);
            if (k < total && at + k < p.out.cap) {
                p.out.pos[at + k] = p0 + i[j];
                p.out.ids[at + k] = id[j];
            }
        }
    }
}

__device__ __forceinline__ void put_full(const BitsParams &p, size_t g0, uint32_t p0, uint32_t total,
                                         unsigned long long at, const uint16_t *list, int lane) {
    for (uint32_t k0 = 0; k0 < total; k0 += 32u) {
        const uint32_t k = k0 + static_cast<uint32_t>(lane);
        uint32_t i = 0, id = 0, cl = 0;
        if (k < total) {
            i = list[k];
            id = static_cast<uint32_t>(p.ids[g0 + i]);
            cl = chain_len(p, id);
        }
        uint32_t inc = cl;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, inc, d);
            if (lane >= d) inc += y;
        }
        if (k < total) put_chain(p, at + (inc - cl), p0 + i, id);
        at += __shfl_sync(kFull, inc, 31);
    }
}

// One warp: the occurrences of the `total` results listed of the tile whose bits
// start at g0, four rounds of 32 in flight.
__device__ __forceinline__ uint32_t sum_chains(const BitsParams &p, size_t g0, uint32_t total, const uint16_t *list,
                                               int lane) {
    uint32_t sum = 0;
    for (uint32_t k0 = static_cast<uint32_t>(lane); k0 < total; k0 += 128u) {
        uint32_t id[4];
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j) id[j] = k0 + 32u * j < total ? static_cast<uint32_t>(p.ids[g0 + list[k0 + 32u * j]]) : 0u;
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j)
            if (k0 + 32u * j < total) sum += chain_len(p, id[j]);
    }
    return __reduce_add_sync(kFull, sum);
}

// Full output: a tile with more than kDense matches is left to the whole CTA,
// each warp an eighth of its positions: one warp waits 64 rounds for the chains
// of a tile where every position matches (16 MiB of ACGT, two such tiles: 200 ->
// 115 us a call; 1 GiB 579 -> 412 with the empty tiles not read).  A CTA notes up to kNoted of them;
// its warps do the others themselves.
constexpr uint32_t kDense = 256, kNoted = 64;
constexpr uint32_t kSlice = kTile / kWarps;
static_assert(kSlice == 256, "eight positions a lane");
struct DenseTiles {
    uint32_t n;
    uint32_t tile[kNoted];
    unsigned long long at[kNoted];
    uint32_t sum[kWarps];
};
__device__ __forceinline__ bool note_tile(DenseTiles &d, uint32_t t, unsigned long long at, uint32_t total, int lane) {
    if (total <= kDense) return false;
    uint32_t i = 0;
    if (lane == 0) {
        i = atomicAdd(&d.n, 1u);
        if (i < kNoted) {
            d.tile[i] = t;
            d.at[i] = at;
        }
    }
    return __shfl_sync(kFull, i, 0) < kNoted;
}
__device__ __forceinline__ uint32_t list_slice(const BitsParams &p, uint32_t t, uint32_t warp, uint16_t *list, int lane) {
    const uint32_t w = t * kWords + warp * (kSlice / 32u) + static_cast<uint32_t>(lane) / 4u;
    const uint32_t b = w < p.words ? (p.bits[w] >> (8u * (lane & 3))) & 0xFFu : 0u;
    const uint32_t c = static_cast<uint32_t>(__popc(b));
    uint32_t inc = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, inc, d);
        if (lane >= d) inc += y;
    }
    uint32_t o = inc - c;
    __syncwarp();
    for (uint32_t m = b; m; m &= m - 1u)
        list[o++] = static_cast<uint16_t>(warp * kSlice + 8u * lane + static_cast<uint32_t>(__ffs(m) - 1));
    __syncwarp();
    return __shfl_sync(kFull, inc, 31);
}
// The whole CTA: the occurrences of the tiles noted (WRITE: their lists).
template <bool WRITE>
__device__ __forceinline__ void noted_tiles(const BitsParams &p, DenseTiles &d, uint16_t *list, int lane, int warp) {
    __syncthreads();
    const uint32_t n = d.n < kNoted ? d.n : kNoted;
    for (uint32_t i = 0; i < n; ++i) {
        const uint32_t t = d.tile[i];
        const size_t g0 = static_cast<size_t>(t) * kTile;
        const uint32_t total = list_slice(p, t, static_cast<uint32_t>(warp), list, lane);
        const uint32_t sum = sum_chains(p, g0, total, list, lane);
        if (lane == 0) d.sum[warp] = sum;
        __syncthreads();
        unsigned long long before = 0;
        for (uint32_t w = 0; w < (WRITE ? static_cast<uint32_t>(warp) : kWarps); ++w) before += d.sum[w];
        if (WRITE)
            put_full(p, g0, t * kTile - p.head, total, d.at[i] + before, list, lane);
        else if (threadIdx.x == 0)
            p.fcounts[t] = static_cast<uint32_t>(before);
        __syncthreads();
    }
}

// One warp: tile t's part of the list.  Compacted: a tile dense in matches is
// one warp's work, so it goes four rounds at a time (256 MiB of ACGT, its 4,096
// matches in the first tiles: 10 against 20 us).
template <bool FULL>
__device__ __forceinline__ void put_tile(const BitsParams &p, uint32_t t, uint32_t p0, uint2 b, unsigned long long at,
                                         uint16_t *list, int lane, DenseTiles *noted = nullptr) {
    const uint32_t total = list_bits(b, list, lane);
    const size_t g0 = static_cast<size_t>(t) * kTile;
    if (FULL) {
        if (!note_tile(*noted, t, at, total, lane)) put_full(p, g0, p0, total, at, list, lane);
    } else if (total <= 32u)
        put_compact<1>(p, g0, p0, total, at, list, lane);
    else
        put_compact<4>(p, g0, p0, total, at, list, lane);
}

// The occurrences of each tile's results, one warp per tile; tiles that hold no
// match by their counts (short texts have none) are not read.
__global__ void __launch_bounds__(kThreads) full_bits_count(const BitsParams p) {
    allow_next();
    wait_previous();
    __shared__ uint16_t lists[kWarps][kTile];
    __shared__ DenseTiles noted;
    if (threadIdx.x == 0) noted.n = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t gw = blockIdx.x * kWarps + static_cast<uint32_t>(warp), nw = gridDim.x * kWarps;
    for (uint64_t u0 = gw; u0 < p.ntiles; u0 += 32ull * nw) {
        const uint64_t u = u0 + static_cast<uint64_t>(lane) * nw;
        const bool some = u < p.ntiles && (!p.counts || p.counts[u] != 0u);
        if (u < p.ntiles && !some) p.fcounts[u] = 0u;
        for (uint32_t todo = __ballot_sync(kFull, some); todo; todo &= todo - 1u) {
            const uint32_t t = static_cast<uint32_t>(u0 + static_cast<uint64_t>(__ffs(todo) - 1) * nw);
            const uint32_t total = list_bits(tile_bits(p, t, lane), lists[warp], lane);
            if (note_tile(noted, t, 0u, total, lane)) continue;
            const uint32_t sum = sum_chains(p, static_cast<size_t>(t) * kTile, total, lists[warp], lane);
            if (lane == 0) p.fcounts[t] = sum;
        }
    }
    noted_tiles<false>(p, noted, lists[warp], lane, warp);
}

// The lists.  SMALL: a CTA has kWarps consecutive tiles, one a warp, and adds
// up what lies before them; else warps take tiles in grid stride, at their
// prefix, and skip the empty ones by their counts.
template <bool FULL, bool SMALL>
__global__ void __launch_bounds__(kThreads) bits_gather(const BitsParams p) {
    wait_previous();
    __shared__ uint16_t lists[kWarps][kTile];
    __shared__ DenseTiles noted;
    if (FULL) {
        if (threadIdx.x == 0) noted.n = 0;
        __syncthreads();
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (SMALL) {
        __shared__ unsigned long long before[kWarps];
        __shared__ uint32_t own[kWarps];
        const uint32_t t0 = blockIdx.x * kWarps, t = t0 + static_cast<uint32_t>(warp);
        unsigned long long sum = 0;
        if (FULL) {
            for (uint32_t i = threadIdx.x; i < t0; i += kThreads) sum += p.counts[i];
        } else {  // the words before the CTA's tiles, 16 bytes a thread
            const uint4 *b = reinterpret_cast<const uint4 *>(p.bits);
            for (uint32_t i = threadIdx.x; i < t0 * (kWords / 4u); i += kThreads) {
                const uint4 v = b[i];
                sum += static_cast<uint32_t>(__popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w));
            }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(kFull, sum, d);
        uint2 b = make_uint2(0u, 0u);
        if (t < p.ntiles) b = tile_bits(p, t, lane);
        uint32_t mine = 0;
        if (FULL)
            mine = t < p.ntiles ? p.counts[t] : 0u;
        else
            mine = __reduce_add_sync(kFull, static_cast<uint32_t>(__popc(b.x) + __popc(b.y)));
        if (lane == 0) {
            before[warp] = sum;
            own[warp] = mine;
        }
        __syncthreads();
        unsigned long long at = 0, all = 0;
        for (uint32_t w = 0; w < kWarps; ++w) all += before[w];
        at = all;
        for (uint32_t w = 0; w < kWarps; ++w) {
            if (w < static_cast<uint32_t>(warp)) at += own[w];
            all += own[w];
        }
        if (t < p.ntiles) put_tile<FULL>(p, t, t * kTile - p.head, b, at, lists[warp], lane, &noted);
        if (t0 + kWarps >= p.ntiles && threadIdx.x == 0) *p.out.count = all;
    } else {
        const uint32_t gw = blockIdx.x * kWarps + static_cast<uint32_t>(warp), nw = gridDim.x * kWarps;
        for (uint64_t u0 = gw; u0 < p.ntiles; u0 += 32ull * nw) {
            const uint64_t u = u0 + static_cast<uint64_t>(lane) * nw;
            const uint32_t c = u < p.ntiles ? p.counts[u] : 0u;
            for (uint32_t todo = __ballot_sync(kFull, c != 0u); todo; todo &= todo - 1u) {
                const uint32_t t = static_cast<uint32_t>(u0 + static_cast<uint64_t>(__ffs(todo) - 1) * nw);
                put_tile<FULL>(p, t, t * kTile - p.head, tile_bits(p, t, lane), p.prefix[t], lists[warp], lane,
                               &noted);
            }
        }
        if (gw == 0 && lane == 0)
            *p.out.count = p.prefix[p.ntiles - 1u] + p.counts[p.ntiles - 1u];
    }
    if constexpr (FULL) noted_tiles<true>(p, noted, lists[warp], lane, warp);
}

// The lists of several texts (streaming form): as bits_gather, each unit's text
// found by a 32-way search.
__global__ void __launch_bounds__(kThreads) bits_gather_texts(BitsParams p, const BitsText *texts, uint32_t nt) {
    wait_previous();
    __shared__ uint16_t lists[kWarps][kTile];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t gw = blockIdx.x * kWarps + static_cast<uint32_t>(warp), nw = gridDim.x * kWarps;
    for (uint64_t u0 = gw; u0 < p.ntiles; u0 += 32ull * nw) {
        const uint64_t u = u0 + static_cast<uint64_t>(lane) * nw;
        const uint32_t c = u < p.ntiles ? p.counts[u] : 0u;
        for (uint32_t todo = __ballot_sync(kFull, c != 0u); todo; todo &= todo - 1u) {
            const uint32_t t = static_cast<uint32_t>(u0 + static_cast<uint64_t>(__ffs(todo) - 1) * nw);
            uint32_t lo = 0, hi = nt;  // the last text whose first unit is <= t
            while (hi - lo > 1u) {
                const uint32_t step = hi - lo > 32u ? (hi - lo + 31u) / 32u : 1u;
                const uint32_t i = lo + static_cast<uint32_t>(lane) * step;
                const unsigned le = __ballot_sync(kFull, i < hi && __ldg(&texts[i].first) <= t);
                lo += static_cast<uint32_t>(31 - __clz(le)) * step;
                hi = lo + step < hi ? lo + step : hi;
            }
            const BitsText x = texts[lo];
            p.out = x.out;
            put_tile<false>(p, t, (t - x.first) * kTile - x.head, tile_bits(p, t, lane),
                            p.prefix[t] - p.prefix[x.first], lists[warp], lane);
        }
    }
    for (uint32_t i = gw * 32u + static_cast<uint32_t>(lane); i < nt; i += nw * 32u) {
        const BitsText x = texts[i];
        const uint32_t last = x.first + x.units - 1u;
        *x.out.count = p.prefix[last] + p.counts[last] - p.prefix[x.first];
    }
}

inline size_t round256(size_t v) { return (v + 255u) & ~static_cast<size_t>(255u); }

// Scratch: list counters (32) | per tile: matches, occurrences (4 each),
// prefix (8) | partial sums | bits | walk and tile list | ids.
struct Layout {
    size_t counts, fcounts, prefix, partials, bits, walks, ids, bytes;
    uint32_t ntiles;
    StreamLists lists;
    bool small;
};

Layout layout_of(const DevTables &t, const Tuning &tu, const uint8_t *text, uint64_t n, bool full, bool captured) {
    Layout l{};
    l.small = at_serves(t, tu, n);
    const uint64_t head = l.small ? 0u : reinterpret_cast<uintptr_t>(text) & 15u;
    l.ntiles = static_cast<uint32_t>((n + head + kTile - 1) / kTile);
    if (!l.small) l.lists = stream_lists(t.stream.form, n, captured);
    size_t at = 256;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += round256(bytes);
        return o;
    };
    l.counts = take(l.small ? 0 : 4ull * l.ntiles);
    l.fcounts = take(full ? 4ull * l.ntiles : 0);
    l.prefix = take(l.small ? 0 : 8ull * l.ntiles);
    l.partials = take(l.small ? 0 : 8ull * kScanCtas);
    l.bits = take(4ull * kWords * l.ntiles);
    l.walks = take(l.lists.bytes());
    l.ids = take(4ull * kTile * l.ntiles);
    l.bytes = at;
    return l;
}

}  // namespace

bool bits_serve(const DevTables &t, const Tuning &tu, uint64_t n) {
    return at_serves(t, tu, n) || stream_serves(t, tu, n);
}

cudaError_t launch_bits_texts(const BitsText *texts, uint32_t nt, uint32_t units, const BitsOut &b,
                              const unsigned long long *prefix, cudaStream_t stream) {
    if (!texts || nt == 0 || units == 0 || !b.bits || !b.ids || !b.counts || !prefix) return cudaErrorInvalidValue;
    BitsParams p{};
    p.bits = b.bits;
    p.ids = b.ids;
    p.words = units * kWords;
    p.ntiles = units;
    p.counts = b.counts;
    p.prefix = prefix;
    const uint32_t need = (units + kWarps - 1) / kWarps, sms = device_sm_count();
    if (sms == 0) return cudaErrorInvalidDevice;
    return launch_next(bits_gather_texts, need < sms * 6u ? need : sms * 6u, kThreads, 0u, stream, p, texts, nt);
}

size_t bits_scratch_bytes(const DevTables &t, const Tuning &tu, const uint8_t *text, uint64_t n, bool full,
                          bool captured) {
    return layout_of(t, tu, text, n, full, captured).bytes;
}

cudaError_t enqueue_bits(const DevTables &t, const Tuning &tu, const uint8_t *text, uint64_t n, const CompactOut &out,
                         bool full, bool captured, void *scratch, size_t scratch_bytes, cudaStream_t stream) {
    if (!bits_serve(t, tu, n) || n == 0 || n > 0xFFFFFFFFull || !scratch || (full && (!t.full_rec || !t.full_dups)))
        return cudaErrorInvalidValue;
    const Layout l = layout_of(t, tu, text, n, full, captured);
    if (scratch_bytes < l.bytes) return cudaErrorInvalidValue;
    uint8_t *b = static_cast<uint8_t *>(scratch);
    MatchRequest r;
    r.text = text;
    r.n = n;
    r.bits.bits = reinterpret_cast<uint32_t *>(b + l.bits);
    r.bits.ids = reinterpret_cast<int32_t *>(b + l.ids);
    cudaError_t e = cudaSuccess;
    if (l.small) {
        e = launch_at(t, r, OUT_BITS, stream);
    } else {
        r.bits.counts = reinterpret_cast<uint32_t *>(b + l.counts);
        r.list_count = reinterpret_cast<unsigned int *>(b);
        r.walks = reinterpret_cast<uint2 *>(b + l.walks);
        r.walk_cap = l.lists.walk_cap;
        r.tile_cap = l.lists.tile_cap;
        e = cudaMemsetAsync(b, 0, 32, stream);
        if (e == cudaSuccess) e = launch_stream(t, r, OUT_BITS, tu, stream);
    }
    if (e != cudaSuccess) return e;

    BitsParams p{};
    p.bits = r.bits.bits;
    p.ids = r.bits.ids;
    p.head = l.small ? 0u : static_cast<uint32_t>(reinterpret_cast<uintptr_t>(text) & 15u);
    p.words = l.small ? static_cast<uint32_t>((n + 31u) / 32u) : l.ntiles * kWords;
    p.ntiles = l.ntiles;
    p.counts = r.bits.counts;
    p.fcounts = reinterpret_cast<uint32_t *>(b + l.fcounts);
    unsigned long long *prefix = reinterpret_cast<unsigned long long *>(b + l.prefix);
    p.prefix = l.small ? nullptr : prefix;
    p.rec = t.full_rec;
    p.dups = t.full_dups;
    p.max_clen = t.full_max_clen;
    p.nkw = t.nkw;
    p.out = out;
    e = device_error_word(&p.err);
    if (e != cudaSuccess) return e;
    const uint32_t need = (l.ntiles + kWarps - 1) / kWarps, sms = device_sm_count();
    if (sms == 0) return cudaErrorInvalidDevice;
    const uint32_t grid = need < sms * 6u ? need : sms * 6u;
    if (full) {
        e = launch_next(full_bits_count, grid, kThreads, 0u, stream, p);
        if (e != cudaSuccess) return e;
        p.counts = p.fcounts;
    }
    if (l.small)
        return full ? launch_next(bits_gather<true, true>, need, kThreads, 0u, stream, p)
                    : launch_next(bits_gather<false, true>, need, kThreads, 0u, stream, p);
    e = launch_compact_scan(p.counts, l.ntiles, nullptr, prefix, reinterpret_cast<unsigned long long *>(b + l.partials),
                            stream);
    if (e != cudaSuccess) return e;
    return full ? launch_next(bits_gather<true, false>, grid, kThreads, 0u, stream, p)
                : launch_next(bits_gather<false, false>, grid, kThreads, 0u, stream, p);
}

}  // namespace pfac
