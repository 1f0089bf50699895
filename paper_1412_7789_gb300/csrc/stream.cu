// One text in two launches, or one: the streaming form (stream_kernel.cuh) and
// its walk step, and the form for short texts (one thread per position).

#include <mutex>

#include "stream_kernel.cuh"

namespace pfac {

using namespace strm;

namespace {

// Texts up to this length take one lane per position: no filter to load into
// every SM, no list, one launch.  4 KiB of the sweep set, where every position
// walks to a match: 10 us a call against 70 in the filter kernel, whose few
// tiles kept a handful of warps busy.  The line against the streaming form (us
// a call): ACGT 2 MiB 14.5 / 15.5, 3 MiB 18.7 / 15.7; where the first 4 KiB all
// match 18.8 / 24.0 at 2 MiB; Zipf bytes 2 MiB 25.7 / 25.5, 3 MiB 24.9 / 21.7.
constexpr uint64_t kAtMax = 2u << 20;
// Threads per CTA: short texts want their positions on many SMs, longer ones
// fewer CTAs (1 MiB of ACGT, 128 / 256 / 512: 11.8 / 10.7 / 12.4 us a call).
__host__ __device__ constexpr int at_block(int per) { return per == 1 ? 128 : 256; }

// One lane per position (a text this short and the tables it touches stay in
// L2).  A warp reads its PER x 32 bytes and the 16 after them once, one byte a
// lane and load, and joins their codes into windows with log2(window) shuffles,
// so a position costs little more than a byte load and a load per table level;
// a lane's PER positions have theirs in flight together.
template <int B, typename GT, int MODE, int PER>
__global__ void __launch_bounds__(at_block(PER)) pfac_at(const __grid_constant__ FilterParams p) {
    __shared__ uint8_t cls8[256];
    allow_next();  // the lists' gather
    const int lane = threadIdx.x & 31;
    const uint64_t g0 = (static_cast<uint64_t>(blockIdx.x) * (at_block(PER) / 32) + (threadIdx.x >> 5)) * (32u * PER) + lane;
    uint32_t c[PER + 1];
    bool in[PER + 1];
#pragma unroll
    for (int j = 0; j <= PER; ++j) {
        in[j] = g0 + 32u * j < p.n && (j < PER || lane < 16);
        c[j] = in[j] ? __ldg(p.text + g0 + 32u * j) : 0u;
    }
    for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x) cls8[i] = __ldg(p.cls8g + i);
    __syncthreads();
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
    int e[PER], r[PER];
    uint4 h[PER];
    bool walk[PER], keep[PER];
    uint32_t s[PER], q[PER], m[PER];
    // several positions a lane (longer texts, few of whose positions get past it):
    // the root filter first, whose 128 KiB stay in L1, not a sector of a table
    // in L2 for each position (2 MiB of ACGT 16.6 -> 14.7 us a call, of Zipf
    // bytes 29.0 -> 25.8; short texts would wait for one load more)
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        keep[j] = true;
        if (PER == 1) continue;
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
    const TileText tt = make_text(p.text, p.out, p.n, 0u);
    uint32_t cnt = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if (B != 8 && !(m[j] & ((1u << need) - 1u))) {
            walk[j] = e[j] >= 0;
            s[j] = static_cast<uint32_t>(e[j]);
            if (e[j] < 0) r[j] = decode_dead(e[j]);
        }
        const uint64_t gi = g0 + 32u * j;
        if (walk[j]) r[j] = filt::walk_global<GT>(p, cls8, tt, static_cast<int64_t>(gi), s[j], q[j]);
        if (MODE == OUT_DENSE) {
            if (in[j]) p.out[gi] = r[j];
        } else if (MODE == OUT_COUNT) {
            cnt += in[j] && r[j] >= 0 ? 1u : 0u;
        } else {
            if (in[j] && r[j] >= 0) p.bo.ids[gi] = r[j];
            const uint32_t bits = __ballot_sync(kFull, in[j] && r[j] >= 0);
            if (lane == 0 && in[j]) p.bo.bits[gi >> 5] = bits;
        }
    }
    add_count<MODE>(p, cnt, lane);
}

// Positions a lane from this length on: 2 (fewer CTAs, and two chains of loads
// in flight); below, 1, where the walks of a text dense in matches need every
// warp.  A lane's walks run one after another, which is what counts against 4:
// us a call, 2 / 4 positions, 1 MiB of ACGT 11.9 / 10.6, 2 MiB 14.7 / 14.0;
// where the first 4 KiB all match 18.7 / 31.0 and 19.2 / 33.
constexpr uint64_t kAtWide = 768u << 10;

template <int B, typename GT, int MODE>
void launch_at_one(const FilterParams &p, cudaStream_t stream) {
    const uint32_t per = p.n >= kAtWide ? 2u : 1u;
    const uint32_t block = at_block(static_cast<int>(per));
    const uint32_t grid = static_cast<uint32_t>((p.n + block * per - 1) / (block * per));
    if (per == 2u)
        pfac_at<B, GT, MODE, 2><<<grid, block, 0, stream>>>(p);
    else
        pfac_at<B, GT, MODE, 1><<<grid, block, 0, stream>>>(p);
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
    // (started early, but with bytes for short texts only: on long ones the
    // walks' CTAs cost the form before them more than the gap they save.  us a
    // call, plain / early: ACGT 4 MiB 17.9 / 15.9, 64 MiB 73.6 / 70.6; Zipf bytes
    // 4 MiB counted 28.8 / 27.0, 24 MiB 46.4 / 45.8, 64 MiB full 112 / 120, 1 GiB
    // compacted 1155 / 1360)
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
    if (!t.stream.form || !untuned(tu) || n / kStreamUnit >= (1ull << 22) - 2) return false;
    return t.stream.root == (t.stream.form == 2 ? t.k : t.fbits);
}

uint32_t stream_walk_cap(uint64_t n) {
    // a walk for every eighth position, and each warp's last reservation
    // (positions past that are settled where they are found)
    return static_cast<uint32_t>(n / 8) + device_sm_count() * static_cast<uint32_t>(kMostWarps) * kWalkChunkEntries;
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

// Shared memory of a launch: the filters, the -1 buffer (and 128 bytes for the
// CTA), the warps' areas.
uint32_t stream_smem(uint32_t form, bool batch, uint32_t filters, uint32_t *off_none, uint32_t *off_warp) {
    *off_none = (filters + 127u) & ~127u;
    *off_warp = *off_none + 4u * kNone + 128u;
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
    const uint32_t smem = stream_smem(t.stream.form, false, p.f1bytes + p.f2bytes, &p.off_none, &p.off_warp);
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

uint32_t stream_batch_cap(uint64_t text_bytes) { return stream_walk_cap(text_bytes); }

cudaError_t launch_stream_batch(const DevTables *const *ts, const MatchRequest *rs, uint32_t nh, OutMode mode,
                                unsigned long long wait_ns, void *walks, uint32_t walk_cap, cudaStream_t stream) {
    if (nh == 0 || nh > kStreamMultiMax || !walks || walk_cap == 0 || (mode != OUT_DENSE && mode != OUT_BITS))
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
    uint8_t *b = static_cast<uint8_t *>(walks);
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
            p.f.walk_cap = walk_cap;
            p.f.walk_chunk = walk_chunk(walk_cap);
            wm.a[a] = p.f;
            filters = filters > p.f1bytes + p.f2bytes ? filters : p.f1bytes + p.f2bytes;
        }
        if (mp.nh == 0) continue;
        const uint32_t smem = stream_smem(form, true, filters, &mp.off_none, &mp.off_warp);
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
