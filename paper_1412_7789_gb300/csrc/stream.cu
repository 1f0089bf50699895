// One text in two launches, or one: the streaming form (stream_kernel.cuh) and
// its walk step, and the form for short texts (one thread per position).

#include <mutex>

#include "stream_kernel.cuh"

namespace pfac {

using namespace strm;

namespace {

// Texts up to this length take a lane for every position or few: no filter to load
// into every SM, no list, one launch.  4 KiB of the sweep set, where every position
// walks to a match: 10 us a call against 70 in the filter kernel, whose few tiles
// kept a handful of warps busy.  The line against the streaming form, us a call,
// short-text / streaming form at 2 MiB: dense ids of ACGT 14.7 / 21.5 (100 keywords)
// and 16.6 / 17.3 (3,000), Zipf bytes 22.8 / 25.6, the alphabet repeated 18.1 /
// 21.3; lists, which both make in a second pass, 29.0 / 31.3, 30.8 / 25.1, 38.5 /
// 33.0 and 32.0 / 35.8.  At 3 MiB dense ids 18.8 / 22.1, 20.8 / 17.9, 29.5 / 25.9
// and 24.8 / 22.5, lists 38.6 / 31.3, 40.9 / 25.9, 51.6 / 35.6 and 44.0 / 41.0.
constexpr uint64_t kAtMax = 2u << 20;
// Threads per CTA: a lane's worth a position, 64 / 128 / 256 take the same within a
// microsecond; with more a lane, 128 / 256 / 512: ACGT, 3,000 keywords, 1 MiB 11.5 /
// 10.7 / 12.4 us a call, Zipf bytes 2 MiB 22.9 / 22.9 / 24.9.
__host__ __device__ constexpr int at_block(int per) { return per == 1 ? 128 : 256; }

// One lane per position (a text this short and the tables it touches stay in L2):
// runs of 32 * PER positions a warp, whose walks are dealt out again over its
// lanes: a warp with several positions a lane else issues as many walks one after
// the other, for a lane or two each.  (Dense ids of 1 MiB, two positions a lane, us
// a call: the alphabet repeated, a walk in 26 positions, 16.7 -> 12.8; words 16.0 ->
// 14.1; where no walk is left to deal out as before.  Over the whole CTA: 12.4 and
// 14.5, but 1 to 2 us more for every text.)
template <int B, typename GT, int MODE, int PER>
__global__ void __launch_bounds__(at_block(PER)) pfac_at(const __grid_constant__ FilterParams p) {
    __shared__ uint8_t cls8[256];
    allow_next();  // the lists' gather
    const int lane = threadIdx.x & 31;
    const uint64_t g0 = (static_cast<uint64_t>(blockIdx.x) * (at_block(PER) / 32) + (threadIdx.x >> 5)) * (32u * PER) + lane;
    uint32_t c[PER + 1];
    bool in[PER + 1];
    load_run<PER>(p.text, p.n, g0, lane, c, in);
    for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x) cls8[i] = __ldg(p.cls8g + i);
    const TileText tt = make_text(p.text, p.out, p.n, 0u);
    uint32_t cnt = 0;
    if constexpr (PER == 1) {
        __syncthreads();
        match_run<B, GT, PER, false>(p, cls8, tt, g0, lane, c, in, [&](int, int r) {
            if (MODE == OUT_DENSE) {
                if (in[0]) p.out[g0] = r;
            } else if (MODE == OUT_COUNT) {
                cnt += r >= 0 ? 1u : 0u;
            } else {
                if (r >= 0) p.bo.ids[g0] = r;
                const uint32_t bits = __ballot_sync(kFull, r >= 0);
                if (lane == 0 && in[0]) p.bo.bits[g0 >> 5] = bits;
            }
        });
    } else {
        __shared__ uint2 walks[at_block(PER) / 32][32 * PER];  // {position in the warp's | q << 16, state}
        __shared__ uint32_t words[at_block(PER) / 32][PER];
        uint2 *mine = walks[threadIdx.x >> 5];
        uint32_t *bits = words[threadIdx.x >> 5];
        __syncthreads();
        RunState<PER> st;
        resolve_run<B, PER, true>(p, cls8, lane, c, in, st);
        uint32_t n = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const bool walk = st.walk[j] && in[j], hit = in[j] && !st.walk[j] && st.r[j] >= 0;
            const unsigned m = __ballot_sync(kFull, walk);
            if (walk)
                mine[n + static_cast<uint32_t>(__popc(m & ((1u << lane) - 1u)))] =
                    make_uint2(32u * j + static_cast<uint32_t>(lane) | (st.q[j] << 16), st.s[j]);
            n += static_cast<uint32_t>(__popc(m));
            if (MODE == OUT_DENSE) {
                if (in[j] && !walk) p.out[g0 + 32u * j] = st.r[j];
            } else if (MODE == OUT_COUNT) {
                cnt += hit ? 1u : 0u;
            } else {
                if (hit) p.bo.ids[g0 + 32u * j] = st.r[j];
                const uint32_t w = __ballot_sync(kFull, hit);
                if (lane == 0) bits[j] = w;
            }
        }
        __syncwarp();
        const uint64_t w0 = g0 - static_cast<uint32_t>(lane);
        for (uint32_t i = static_cast<uint32_t>(lane); i < n; i += 32u) {
            const uint2 e = mine[i];
            const uint32_t l = e.x & 0xFFFFu;
            const int r = filt::walk_global<GT>(p, cls8, tt, static_cast<int64_t>(w0 + l), e.y, e.x >> 16);
            if (MODE == OUT_DENSE) {
                p.out[w0 + l] = r;
            } else if (MODE == OUT_COUNT) {
                cnt += r >= 0 ? 1u : 0u;
            } else if (r >= 0) {
                p.bo.ids[w0 + l] = r;
                atomicOr(bits + (l >> 5), 1u << (l & 31u));
            }
        }
        if (MODE == OUT_BITS) {
            __syncwarp();
            if (lane < PER && w0 + 32u * lane < p.n) p.bo.bits[(w0 >> 5) + lane] = bits[lane];
        }
    }
    add_count<MODE>(p, cnt, lane);
}

// Positions a lane: 1, where the walks of a text dense in matches need every warp;
// from kAtWide on 2 (fewer CTAs, and two chains of loads in flight); with 8-bit
// codes from kAtWider on 4.  A lane's walks run one after another, which is what
// counts against more with 2-bit codes.  us a call, 2 / 4 positions: 1 MiB of ACGT
// 10.5 / 10.4, of the alphabet repeated 12.8 / 10.6, words 14.1 / 12.5, Zipf bytes
// 14.9 / 16.5; 2 MiB 14.7 / 14.5, 22.8 / 18.1, 20.8 / 18.7, 23.0 / 22.8; where the
// first 4 KiB of ACGT all match 18.8 / 27.
constexpr uint64_t kAtWide = 768u << 10, kAtWider = 1u << 20;

template <int B, typename GT, int MODE, int PER>
void launch_at_per(const FilterParams &p, cudaStream_t stream) {
    const uint64_t block = at_block(PER);
    pfac_at<B, GT, MODE, PER><<<static_cast<uint32_t>((p.n + block * PER - 1) / (block * PER)), block, 0, stream>>>(p);
}
template <int B, typename GT, int MODE>
void launch_at_one(const FilterParams &p, cudaStream_t stream) {
    if (p.n < kAtWide)
        launch_at_per<B, GT, MODE, 1>(p, stream);
    else if (B != 8 || p.n < kAtWider)
        launch_at_per<B, GT, MODE, 2>(p, stream);
    else
        launch_at_per<B, GT, MODE, B == 8 ? 4 : 2>(p, stream);
}

template <int B, typename GT>
cudaError_t launch_at_modes(OutMode mode, const FilterParams &p, cudaStream_t stream) {
    switch (mode) {
        case OUT_DENSE: launch_at_one<B, GT, OUT_DENSE>(p, stream); break;
        case OUT_COUNT: launch_at_one<B, GT, OUT_COUNT>(p, stream); break;
        case OUT_BITS: launch_at_one<B, GT, OUT_BITS>(p, stream); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

constexpr uint64_t kWalkEarly = 16u << 20;
template <int B, typename GT>
cudaError_t launch_walk_modes(OutMode mode, const FilterParams &p, uint32_t sms, cudaStream_t stream) {
    const uint32_t grid = sms * kWalkCtas;
    auto kernel = mode == OUT_DENSE ? pfac_stream_walks<B, GT, OUT_DENSE>
                  : mode == OUT_COUNT ? pfac_stream_walks<B, GT, OUT_COUNT>
                                      : pfac_stream_walks<B, GT, OUT_BITS>;
    // (started early, but with bytes for short texts only: on long ones the walks'
    // CTAs cost the form before them more than the gap they save.  us a call, plain /
    // early: ACGT 4 MiB 17.9 / 15.9, 64 MiB 73.6 / 70.6; 20,000 keywords in Zipf
    // bytes, counted 4 MiB 29.2 / 28.8, 16 MiB 41.5 / 39.8, 24 MiB 48.3 / 47.5, 32
    // MiB 54.9 / 57.0, 64 MiB 81.0 / 86.9; dense 16 MiB 45.2 / 44.4, 24 MiB 54.9 /
    // 56.4; compacted 16 MiB 52.3 / 50.2, 24 MiB 58.2 / 58.5, 64 MiB 97.8 / 105.2)
    if (B == 2 || p.n <= kWalkEarly) return launch_next(kernel, grid, kWalkBlock, 0u, stream, p);
    kernel<<<grid, kWalkBlock, 0, stream>>>(p);
    return cudaGetLastError();
}

// Every knob as built: the caller asks for no particular form.
bool untuned(const Tuning &tu) {
    return tu.block == 0 && tu.stages == 0 && tu.grid == 0 && tu.variant == 0 && tu.per_thread != 4 &&
           tu.halo <= 16 && tu.survivor_list == 0 && !tu.stall_help;
}

}  // namespace

bool at_serves(const DevTables &t, const Tuning &tu, uint64_t n) {
    return untuned(tu) && n <= kAtMax && (t.filter || (t.hashed && t.HK));
}

cudaError_t launch_at(const DevTables &t, const MatchRequest &r, OutMode mode, cudaStream_t stream) {
    if (r.batch || r.n == 0) return cudaErrorInvalidValue;
    FilterParams p;
    const cudaError_t e = filter_params(t, r, mode, Tuning{}, p);
    if (e != cudaSuccess) return e;
    const bool g16 = t.gbits == 16;
    if (t.B == 2) return g16 ? launch_at_modes<2, int16_t>(mode, p, stream) : launch_at_modes<2, int32_t>(mode, p, stream);
    if (t.B == 4) return g16 ? launch_at_modes<4, int16_t>(mode, p, stream) : launch_at_modes<4, int32_t>(mode, p, stream);
    return g16 ? launch_at_modes<8, int16_t>(mode, p, stream) : launch_at_modes<8, int32_t>(mode, p, stream);
}

bool stream_serves(const DevTables &t, const Tuning &tu, uint64_t n) {
    // (positions, and what rounds a text up to whole tiles, are numbered in 32 bits)
    if (!t.stream.form || !untuned(tu) || n >= (1ull << 32) - kTile) return false;
    return t.stream.root == (t.stream.form == 2 ? t.k : t.fbits);
}

StreamLists stream_lists(uint32_t form, uint64_t n, bool captured) {
    // Every tile; each warp's last reservation; and a walk for every eighth
    // position, with 2-bit codes for every sixteenth: few of their windows of 14 or
    // 16 letters go on, and the filter kernel takes no list for most of these sets.
    // A text with more has its other tiles listed whole, which costs time only:
    // 64 MiB, a tenth of it runs of one letter, dense ids with 8 / 4 / 2 bits of
    // list a position 297 / 399 / 421 us (filter kernel 653), 5 % of a repeat
    // 424 / 423 / 661 (360); bytes, prose, 285 / 461 / 700 (371).
    // In a captured graph the memory is the graph's and no other form can step in
    // when it is not to be had: 2-bit codes make do with the warps' reservations.
    StreamLists l;
    const uint64_t walks = form == 2 ? (captured ? 0u : n / 16) : n / 8;
    l.walk_cap = static_cast<uint32_t>(walks) + device_sm_count() * static_cast<uint32_t>(kMostWarps) * kWalkChunkEntries;
    l.tile_cap = static_cast<uint32_t>(n / kTile) + 2u;
    return l;
}

namespace {

// Entries a warp reserves of a walk list at a time: no more than half the list
// over all warps, so that a short list (a wave's, which stays within what its
// requests were charged) is not used up by empty entries.
uint32_t walk_chunk(uint32_t walk_cap) {
    const uint32_t c = walk_cap / (2u * device_sm_count() * static_cast<uint32_t>(kMostWarps) + 1u);
    return c < 1u ? 1u : (c < kWalkChunkEntries ? c : kWalkChunkEntries);
}

// The streaming form's parameters of one automaton, all but the places in
// shared memory.
cudaError_t stream_params(const DevTables &t, const MatchRequest &r, OutMode mode, const Tuning &tu, StreamParams &p) {
    const cudaError_t e = filter_params(t, r, mode, tu, p.f);
    if (e != cudaSuccess) return e;
    if (mode == OUT_BITS && !r.bits.counts) return cudaErrorInvalidValue;
    p.f.walks = r.walks;
    p.f.walk_cap = r.walk_cap;
    p.f.tile_cap = r.tile_cap;
    p.f.list_count = r.list_count;
    p.f.walk_chunk = walk_chunk(r.walk_cap);
    p.F1 = t.stream_F1 ? t.stream_F1 : t.F;
    p.f1bytes = (1u << kFilterBits) / 8u;
    p.F2 = t.stream_F2;
    p.f2bytes = t.stream_F2 ? t.stream_f2bytes : 0u;
    p.four = 4u;
    p.m1 = t.stream.m1;
    p.m2 = t.stream.m2;
    p.l2shift = t.stream.form == 2 ? 32u - 2u * t.stream.win2 : 0u;
    return cudaSuccess;
}

// Shared memory of a launch: the filters, 128 bytes for the CTA, the -1 buffer
// (where it has bulk stores), the warps' areas.
uint32_t stream_smem(uint32_t form, OutMode mode, bool batch, uint32_t filters, uint32_t *off_cta, uint32_t *off_warp) {
    *off_cta = (filters + 127u) & ~127u;
    *off_warp = *off_cta + 128u + (has_bulk(form, mode) ? 4u * kNone : 0u);
    return *off_warp + static_cast<uint32_t>(block_of(form, batch) / 32) * (form == 2 ? kWarpBytes2 : kWarpBytes8);
}

}  // namespace

cudaError_t launch_stream(const DevTables &t, const MatchRequest &r, OutMode mode, const Tuning &tu,
                          cudaStream_t stream) {
    if (!stream_serves(t, tu, r.n) || r.batch || r.n == 0 || !r.walks || !r.list_count || r.walk_cap == 0)
        return cudaErrorInvalidValue;
    int sms = 0, max_smem = 0;
    cudaError_t e = filter_device_shape(&sms, &max_smem);
    if (e != cudaSuccess) return e;
    StreamParams p{};
    e = stream_params(t, r, mode, tu, p);
    if (e != cudaSuccess) return e;
    p.sg = make_seg(r.text, r.out, r.n);
    p.ntiles = static_cast<uint32_t>((r.n + p.sg.head + kTile - 1) / kTile);
    const uint32_t smem = stream_smem(t.stream.form, mode, false, p.f1bytes + p.f2bytes, &p.off_cta, &p.off_warp);
    if (static_cast<int>(smem) > max_smem) return cudaErrorInvalidConfiguration;
    // short texts spread over the SMs, a tile to each of eight warps (3 MiB of
    // ACGT 17.5 -> 15.7 us a call, of Zipf bytes 23.7 -> 21.7)
    const uint32_t need = (p.ntiles + 7) / 8;
    const uint32_t grid = need < static_cast<uint32_t>(sms) ? need : static_cast<uint32_t>(sms);
    e = t.stream.form == 2 ? launch_stream2(mode, p, t.stream.step, grid, smem, max_smem, stream)
                           : launch_stream8(mode, p, grid, smem, max_smem, stream);
    if (e != cudaSuccess) return e;
    const uint32_t n_sm = static_cast<uint32_t>(sms);
    const bool g16 = t.gbits == 16;
    if (t.B == 2)
        return g16 ? launch_walk_modes<2, int16_t>(mode, p.f, n_sm, stream)
                   : launch_walk_modes<2, int32_t>(mode, p.f, n_sm, stream);
    return g16 ? launch_walk_modes<8, int16_t>(mode, p.f, n_sm, stream)
               : launch_walk_modes<8, int32_t>(mode, p.f, n_sm, stream);
}

bool stream_batch_serves(const DevTables &t, const Tuning &tu) { return stream_serves(t, tu, 0); }

StreamLists stream_batch_lists(uint64_t text_bytes, uint32_t texts) {
    // a text's two ragged tiles too, as far as they are long enough to be listed
    StreamLists l = stream_lists(8, text_bytes, false);
    const uint64_t ragged = 2ull * texts, most = text_bytes / kFew;
    l.tile_cap += static_cast<uint32_t>(ragged < most ? ragged : most);
    return l;
}

cudaError_t launch_stream_batch(const DevTables *const *ts, const MatchRequest *rs, uint32_t nh, OutMode mode,
                                unsigned long long wait_ns, void *lists, const StreamLists &l, cudaStream_t stream) {
    if (nh == 0 || nh > kStreamMultiMax || !lists || l.walk_cap == 0 || (mode != OUT_DENSE && mode != OUT_BITS))
        return cudaErrorInvalidValue;
    int sms = 0, max_smem = 0;
    cudaError_t e = filter_device_shape(&sms, &max_smem);
    if (e != cudaSuccess) return e;
    // some 20 KiB of parameters a launch: kept off the stack, filled and
    // launched under a lock
    static StreamMulti mp;
    static WalkMulti wm;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    Tuning tu;
    tu.wait_ns = wait_ns;
    uint8_t *b = static_cast<uint8_t *>(lists);
    wm.nh = nh;
    // one launch per form and step, then the walks of all
    bool next = false;  // after another of these launches
    for (uint32_t group = 0; group < 4; ++group) {
        const uint32_t form = group < 3 ? 2u : 8u, step = group < 3 ? 1u << group : 1u;
        uint32_t filters = 0;
        mp.nh = 0;
        for (uint32_t a = 0; a < nh; ++a) {
            const DevTables &t = *ts[a];
            if (t.stream.form != form || t.stream.step != step) continue;
            const MatchRequest &r = rs[a];
            if (!stream_batch_serves(t, tu) || !r.batch || !r.lists || !r.scratch || r.scratch_bytes < 16)
                return cudaErrorInvalidValue;
            StreamParams &p = mp.a[mp.nh++];
            p = StreamParams{};
            e = stream_params(t, r, mode, tu, p);
            if (e != cudaSuccess) return e;
            p.f.sl.ubase = r.slots.ubase;
            p.f.aidx = a;
            p.f.list_count = reinterpret_cast<unsigned int *>(b);
            p.f.walks4 = reinterpret_cast<uint4 *>(b + 32);
            p.f.walk_cap = l.walk_cap;
            p.f.tile_cap = l.tile_cap;
            p.f.walk_chunk = walk_chunk(l.walk_cap);
            wm.a[a] = p.f;
            filters = filters > p.f1bytes + p.f2bytes ? filters : p.f1bytes + p.f2bytes;
        }
        if (mp.nh == 0) continue;
        const uint32_t smem = stream_smem(form, mode, true, filters, &mp.off_cta, &mp.off_warp);
        if (static_cast<int>(smem) > max_smem) return cudaErrorInvalidConfiguration;
        const uint32_t grid = static_cast<uint32_t>(sms);
        e = form == 2 ? launch_stream2_multi(mode, mp, step, grid, smem, max_smem, stream, next)
                      : launch_stream8_multi(mode, mp, grid, smem, max_smem, stream, next);
        if (e != cudaSuccess) return e;
        next = true;
    }
    const uint32_t grid = static_cast<uint32_t>(sms) * 8u;
    const uint32_t smem = nh * (static_cast<uint32_t>(sizeof(FilterParams)) + 256u);
    return mode == OUT_DENSE ? launch_next(pfac_stream_walks_multi<OUT_DENSE>, grid, kWalkBlock, smem, stream, wm)
                             : launch_next(pfac_stream_walks_multi<OUT_BITS>, grid, kWalkBlock, smem, stream, wm);
}

}  // namespace pfac
