// hd_encode.cu -- the encoders of the full-length codes (the transmitter side
// of Sec. II: checksum bits are added to the message) and of their SECDED
// extensions.
//
// Bound: HBM from n = 31 up (k/8 bytes read, n/8, with SECDED (n + 1)/8, written
// per codeword), the integer ALU below (n = 15: 13 operations a codeword).  The
// checksum bits come from superset_xor (hd_lane.cuh), not from popcounts.
// Measured on GB300 at 1 Gbit of codewords, of the measured copy bandwidth:
// n = 3 / 7 / 15 / 31 / 63 / 127 / 255: 0.82 / 0.58 / 0.72 / 0.86 / 0.85 / 0.84 /
// 0.88, SECDED 0.80 / 0.60 / 0.62 / 0.78 / 0.79 / 0.83 / 0.82.  The kernels these
// replaced (a lane's bits moved one run at a time through shared memory;
// SECDED bit by bit with atomics into a cleared stream) took 397 us for n = 63
// at 2^24 codewords, this one 43.
#include <algorithm>
#include <cstdint>

#include "hd_device.cuh"
#include "hd_internal.h"
#include "hd_lane.cuh"
#include "hd_stream.cuh"
#include "hd_tile.cuh"

namespace hd {
namespace {

// ---------------------------------------------------------------------------
// Plain codes: the streaming decoder's scheme turned round.  A warp chunk is
// 32*G codewords (G per thread); every warp owns S stages filled by 1-D bulk
// copies; each thread re-aligns its message words in registers, and the
// codewords overwrite the chunk's own stage, which a bulk store drains while
// the next chunk is encoded.  32 codewords of odd n keep the lanes' writes at
// an odd word stride (no bank conflicts).  The warps that hold the fewest
// chunks (the last ones of the grid) encode a ragged tail's tiles, one codeword
// per lane, before their first chunk, so a tail costs no launch of its own.
// ---------------------------------------------------------------------------
// CH: chunks a stage holds.  The short codes' chunks are a few hundred bytes;
// several per stage share the iteration's fixed cost (the wait, the refill, the
// bulk store: about 80 instructions): 1 Gbit of n = 3 in 32 us with 8 against 50
// with one, n = 7 in 54 with 4 against 60; n = 15 gains nothing (50 against 48).  Every lane reads its parts of all of
// them before the first is overwritten.
template <int N_, int T, int S, int G, int CH>
struct EncCfg {
    using C = Code<N_>;
    static constexpr int WARPS = T / 32, H = 32 / G, TEAMS = 32 / H;
    static constexpr int GI = G * C::k, GO = G * N_;  // message and codeword bits per thread
    static constexpr bool IN_ALIGNED = H == 1 || GI % 32 == 0, OUT_ALIGNED = H == 1 || GO % 32 == 0;
    static constexpr int R = (GI + 31) / 32;
    static constexpr uint32_t chunk_cw = 32u * G * CH;  // codewords per stage
    static constexpr uint32_t in_words = CH * TEAMS * C::k, out_words = CH * TEAMS * N_;
    static constexpr uint32_t in_bytes = in_words * 4, out_bytes = out_words * 4;
    static constexpr int SLOT = lane_slot_words(C::Wy);
    static constexpr uint32_t slot_bytes = 32u * SLOT * 4u;
    static constexpr uint32_t stage_bytes = out_bytes + 16;  // a spill word past the end
    static constexpr uint32_t ring_bytes = S * stage_bytes > slot_bytes ? S * stage_bytes : slot_bytes;
    static constexpr uint32_t warp_bytes = (64 + ring_bytes + 127) / 128 * 128;
    static constexpr uint32_t smem = WARPS * warp_bytes;
    static_assert(in_bytes % 16 == 0 && out_bytes % 16 == 0, "bulk copies need 16B sizes");
    static_assert(smem <= 232448 && S >= 2 && S <= 8, "shared memory per CTA");
};

// (The buffers are kernel parameters of their own, so that the compiler knows
// them for global memory.)
struct EncArgs {
    uint64_t data_words, stream_words, num_cw;
    uint64_t nchunks;              // whole chunks encoded as such
    uint64_t tile_begin, tile_end;  // 32-codeword tiles for the per-lane path
    uint32_t *status;
};

template <int N_, int T, int S, int G, int CH>
__global__ void __launch_bounds__(T) k_encode_stream(const uint32_t *__restrict__ data, uint32_t *__restrict__ stream, const EncArgs a)
{
    using Cfg = EncCfg<N_, T, S, G, CH>;
    using C = Code<N_>;
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    grid_dep_launch_dependents();
    uint8_t *wbase = smem + warp * Cfg::warp_bytes;
    uint64_t *bar = reinterpret_cast<uint64_t *>(wbase);
    uint8_t *ring = wbase + 64;
    const uint64_t gw = (uint64_t)blockIdx.x * Cfg::WARPS + warp, tw = (uint64_t)gridDim.x * Cfg::WARPS;
    grid_dep_wait();  // the kernels ahead have finished: what produced the messages, what still reads the stream

    // the tail's tiles, from the grid's last warp on
    for (uint64_t t = a.tile_begin + (tw - 1 - gw); t < a.tile_end; t += tw)
        encode_lane_tile<N_>(data, a.data_words, a.num_cw, t, stream, a.stream_words,
                             reinterpret_cast<uint32_t *>(ring), lane);
    if (gw >= a.nchunks) return;

    auto load = [&](uint64_t c, int s) {
        mbar_arrive_expect_tx(&bar[s], Cfg::in_bytes);
        bulk_g2s(ring + s * Cfg::stage_bytes, data + c * (uint64_t)Cfg::in_words, Cfg::in_bytes, &bar[s]);
    };
    fence_proxy_async_smem();  // the tiles above used the ring
    __syncwarp();
    if (lane == 0) {
#pragma unroll
        for (int s = 0; s < S; ++s) mbar_init(&bar[s], 1);
        fence_mbar_init();
#pragma unroll
        for (int s = 0; s < S; ++s)
            if (gw + (uint64_t)s * tw < a.nchunks) load(gw + (uint64_t)s * tw, s);
    }
    __syncwarp();

    const int team = lane / Cfg::H, h = lane % Cfg::H;
    const uint32_t in_bit = (uint32_t)h * (uint32_t)Cfg::GI, in_sh = in_bit & 31u;
    const uint32_t in_w = team * C::k + (in_bit >> 5);
    const uint32_t out_bit = (uint32_t)h * (uint32_t)Cfg::GO, out_sh = out_bit & 31u;
    const uint32_t out_w = team * N_ + (out_bit >> 5);
    uint32_t it = 0;
    bool aborted = false;
    for (uint64_t c = gw; c < a.nchunks; c += tw, ++it) {
        const int s = (int)(it % S);
        const bool ok = mbar_wait_bounded(&bar[s], (it / S) & 1u);
        if (__any_sync(0xFFFFFFFFu, !ok)) {
            aborted = true;
            break;
        }
        uint32_t *stage = reinterpret_cast<uint32_t *>(ring + s * Cfg::stage_bytes);
        uint32_t r[CH][Cfg::R];
#pragma unroll
        for (int ch = 0; ch < CH; ++ch) {
            const uint32_t *src = stage + ch * Cfg::TEAMS * C::k + in_w;
            if constexpr (Cfg::IN_ALIGNED) {
#pragma unroll
                for (int w = 0; w < Cfg::R; ++w) r[ch][w] = src[w];
            } else {
                uint32_t lo = src[0];
#pragma unroll
                for (int w = 0; w < Cfg::R; ++w) {
                    const uint32_t hi = src[w + 1];
                    r[ch][w] = __funnelshift_r(lo, hi, in_sh);
                    lo = hi;
                }
            }
        }
        __syncwarp();  // the whole stage is in registers
#pragma unroll
        for (int ch = 0; ch < CH; ++ch) {
            OutPacker<Cfg::GO, Cfg::OUT_ALIGNED, 1> op(stage + ch * Cfg::TEAMS * N_ + out_w, out_sh);
            encode_part<N_, G, Cfg::R>(r[ch], op);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
            // the store issued last iteration has read its stage: refill it (lookahead S - 1)
            bulk_wait_read<0>();
            const uint64_t cn = c - tw + (uint64_t)S * tw;
            if (it > 0 && cn < a.nchunks) load(cn, (int)((it - 1) % S));
            bulk_s2g(stream + c * (uint64_t)Cfg::out_words, stage, Cfg::out_bytes);
            bulk_commit();
        }
        __syncwarp();
    }
    if (lane == 0) {
        if (aborted) {
            atomicOr(a.status, (uint32_t)HD_ERR_TIMEOUT);
            const uint32_t pending = it > 0 ? S - 1 : S;  // loads still in flight into this warp's ring
            for (uint32_t j = it; j < it + pending; ++j)
                if (gw + (uint64_t)j * tw < a.nchunks) (void)mbar_wait_bounded(&bar[j % S], (j / S) & 1u);
        }
        bulk_wait_all<0>();
    }
}

// Short streams: one codeword per lane throughout (a chunk is G codewords a
// lane, one after the other, so few chunks leave the GPU idle for as long as
// one takes), and no ring, so that an SM holds up to 64 warps.
constexpr int kLaneWarps = 8;

template <int N_>
__global__ void __launch_bounds__(kLaneWarps * 32) k_encode_lanes(const uint32_t *__restrict__ data, uint32_t *__restrict__ stream, const EncArgs a)
{
    __shared__ uint32_t slots[kLaneWarps][32 * lane_slot_words(Code<N_>::Wy)];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    grid_dep_launch_dependents();
    grid_dep_wait();
    for (uint64_t t = (uint64_t)blockIdx.x * kLaneWarps + warp; t < a.tile_end; t += (uint64_t)gridDim.x * kLaneWarps)
        encode_lane_tile<N_>(data, a.data_words, a.num_cw, t, stream, a.stream_words, slots[warp], lane);
}

template <int N_, int T, int S, int G, int CH = 1>
cudaError_t launch_encode_stream(const uint32_t *data, uint32_t *stream, EncArgs a, cudaStream_t st)
{
    using Cfg = EncCfg<N_, T, S, G, CH>;
    a.tile_end = (a.num_cw + 31) / 32;
    static BlocksPerSm lane_blocks, blocks;
    const int lane_bps = lane_blocks.get(reinterpret_cast<const void *>(k_encode_lanes<N_>), kLaneWarps * 32, 0);
    const uint64_t lane_cap = (uint64_t)num_sms() * (uint64_t)std::max(lane_bps, 1);
    // At most one round of tiles on the CTAs the device holds at once (152 SMs:
    // 311,296 codewords, fewer for the long codes' wider kernels): the two paths cross
    // about there on GB300.  n = 31, lanes against chunks: 1.4 against 2.9 us at
    // 20,000 codewords, 2.6 against 3.1 at 300,000, 3.9 against 3.3 at 600,000;
    // n = 255: 2.8 against 3.6 at 100,000, 4.8 against 4.4 at 200,000.
    if (a.tile_end <= (uint64_t)decode_grid(lane_cap, lane_cap) * kLaneWarps) {
        const int grid = decode_grid((a.tile_end + kLaneWarps - 1) / kLaneWarps, lane_cap);
        return launch_kernel(k_encode_lanes<N_>, dim3((unsigned)grid), dim3(kLaneWarps * 32), 0, st, true,
                             data, stream, a);
    }
    auto kern = k_encode_stream<N_, T, S, G, CH>;
    const int bps = blocks.get(reinterpret_cast<const void *>(kern), T, Cfg::smem);
    if (bps <= 0) return cudaErrorInvalidConfiguration;
    a.nchunks = a.num_cw / Cfg::chunk_cw;
    a.tile_begin = a.nchunks * (Cfg::chunk_cw / 32);
    const int grid = decode_grid((a.nchunks + Cfg::WARPS - 1) / Cfg::WARPS, (uint64_t)num_sms() * (uint64_t)bps);
    return launch_kernel(kern, dim3((unsigned)grid), dim3(T), Cfg::smem, st, true, data, stream, a);
}

// ---------------------------------------------------------------------------
// SECDED: a codeword of n + 1 = 2^m bits is one or more whole words (or a
// word holds 32 / (n + 1) of them), so a lane makes whole words and
// neighbouring lanes write neighbouring words: coalesced stores without a trip
// through shared memory, at every size.  An item is four words up to n = 31
// (one 16-byte store), else one codeword.  Its message bits start at any bit
// of the input (at a word for n = 3 and 7); the lane reads the words that
// cover them (its neighbours' reads overlap in L1), U items ahead of their use.
// ---------------------------------------------------------------------------
constexpr int kXhThreads = 256;

template <int N_>
struct XhItem {
    static constexpr int W = N_ <= 31 ? 4 : Code<N_>::Wy;                     // words
    static constexpr int CW = N_ < 31 ? 4 * kFieldCodewords<N_> : N_ == 31 ? 4 : 1;  // codewords
    static constexpr int BITS = CW * Code<N_>::k;                             // message bits
    static constexpr int LW = BITS % 32 == 0 ? BITS / 32 : (BITS + 62) / 32;  // words that cover them
};

template <int N_, int U>
__global__ void __launch_bounds__(kXhThreads)
    k_encode_secded(const uint32_t *__restrict__ data, uint64_t data_words, uint64_t num_cw,
                    uint32_t *__restrict__ stream)
{
    using C = Code<N_>;
    using I = XhItem<N_>;
    constexpr int W = I::W, CW = I::CW, BITS = I::BITS, LW = I::LW, RW = (BITS + 31) / 32;
    const int lane = threadIdx.x & 31;
    grid_dep_launch_dependents();
    const uint64_t gw = (uint64_t)blockIdx.x * (kXhThreads / 32) + (threadIdx.x >> 5);
    const uint64_t tw = (uint64_t)gridDim.x * (kXhThreads / 32);
    constexpr uint64_t kGroupCw = (uint64_t)32 * U * CW;  // codewords a warp takes per step
    const uint64_t groups = (num_cw + kGroupCw - 1) / kGroupCw;
    const uint32_t bit = (uint32_t)lane * BITS, sh = bit & 31u, first = bit >> 5;
    grid_dep_wait();
    for (uint64_t g = gw; g < groups; g += tw) {
        // 32 items fill BITS input words and 32 * W output words
        const uint32_t *src = data + g * (uint64_t)(U * BITS) + first;
        uint32_t *dst = stream + g * (uint64_t)(U * 32 * W) + (uint32_t)lane * W;
        // whole groups (all but the last) read and write without a test
        const bool whole = (g + 1) * kGroupCw <= num_cw && (g + 1) * (uint64_t)(U * BITS) + LW <= data_words;
        uint32_t raw[U][LW];
        if (whole) {
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int w = 0; w < LW; ++w) raw[u][w] = __ldg(src + u * BITS + w);
        } else {
            const uint64_t at = g * (uint64_t)(U * BITS) + first;
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int w = 0; w < LW; ++w)
                    raw[u][w] = at + u * BITS + w < data_words ? __ldg(src + u * BITS + w) : 0u;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            uint32_t d[RW], y[W];
#pragma unroll
            for (int w = 0; w < RW; ++w)
                d[w] = LW == RW ? raw[u][w] : __funnelshift_r(raw[u][w], w + 1 < LW ? raw[u][w + 1] : 0u, sh);
            // codewords of this item; messages past the last one are pad bits
            const uint64_t cw0 = ((g * U + u) * 32 + lane) * CW;
            const uint32_t left = whole ? (uint32_t)CW : cw0 < num_cw ? (uint32_t)min((uint64_t)CW, num_cw - cw0) : 0u;
            if (!whole) {
#pragma unroll
                for (int w = 0; w < RW; ++w) {
                    const int have = (int)left * C::k - 32 * w;
                    d[w] = have >= 32 ? d[w] : have > 0 ? d[w] & ((1u << have) - 1u) : 0u;
                }
            }
            if constexpr (N_ <= 31) {
                constexpr int F = N_ < 31 ? kFieldCodewords<N_> : 1;  // codewords per word
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    uint32_t x = bits_at(d, w * F * C::k);
                    if constexpr (N_ < 31) {
                        if constexpr (F * C::k < 32) x &= (1u << (F * C::k)) - 1u;
                        y[w] = encode_fields<N_, true>(x);
                    } else {
                        const uint32_t one[1] = {x};
                        uint32_t v[1];
                        encode_words<N_, true>(one, 0, v);
                        y[w] = v[0];
                    }
                }
            } else {
                encode_words<N_, true>(d, 0, y);
            }
            uint32_t *o = dst + u * 32 * W;
            if (whole || left == (uint32_t)CW) {
                if constexpr (W == 2) {
                    *reinterpret_cast<uint2 *>(o) = make_uint2(y[0], y[1]);
                } else {
#pragma unroll
                    for (int w = 0; w < W; w += 4)
                        *reinterpret_cast<uint4 *>(o + w) = make_uint4(y[w], y[w + 1], y[w + 2], y[w + 3]);
                }
            } else if (left != 0) {
#pragma unroll
                for (int w = 0; w < W; ++w)
                    if (w * 32 < (int)left * (N_ + 1)) o[w] = y[w];
            }
        }
    }
}

template <int N_, int U>
cudaError_t launch_encode_xh(const uint32_t *data, uint64_t data_words, uint64_t num_cw, uint32_t *stream,
                             cudaStream_t st)
{
    constexpr uint64_t per_warp = (uint64_t)U * 32 * XhItem<N_>::CW;
    const uint64_t warps = (num_cw + per_warp - 1) / per_warp, per_cta = kXhThreads / 32;
    const int grid = decode_grid((warps + per_cta - 1) / per_cta, (uint64_t)num_sms() * 8);
    return launch_kernel(k_encode_secded<N_, U>, dim3((unsigned)grid), dim3(kXhThreads), 0, st, true, data,
                         data_words, num_cw, stream);
}

}  // namespace

cudaError_t launch_encode(const uint32_t *data, uint64_t data_words, uint32_t n, uint64_t num_cw, uint32_t *stream,
                          uint64_t stream_words, cudaStream_t st)
{
    EncArgs a{};
    a.data_words = data_words;
    a.stream_words = stream_words;
    a.num_cw = num_cw;
    a.status = status_ptr();
    if (a.status == nullptr) return cudaErrorInvalidSymbol;
    switch (n) {
        case 3: return launch_encode_stream<3, 128, 2, 32, 8>(data, stream, a, st);
        case 7: return launch_encode_stream<7, 128, 2, 32, 4>(data, stream, a, st);
        case 15: return launch_encode_stream<15, 256, 4, 32>(data, stream, a, st);
        case 31: return launch_encode_stream<31, 128, 3, 32>(data, stream, a, st);
        case 63: return launch_encode_stream<63, 128, 3, 32>(data, stream, a, st);
        case 127: return launch_encode_stream<127, 256, 3, 8>(data, stream, a, st);
        case 255: return launch_encode_stream<255, 128, 2, 8>(data, stream, a, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_encode_secded(const uint32_t *data, uint64_t data_words, uint32_t n, uint64_t num_cw,
                                 uint32_t *stream, cudaStream_t st)
{
    switch (n) {
        case 3: return launch_encode_xh<3, 2>(data, data_words, num_cw, stream, st);
        case 7: return launch_encode_xh<7, 2>(data, data_words, num_cw, stream, st);
        case 15: return launch_encode_xh<15, 2>(data, data_words, num_cw, stream, st);
        case 31: return launch_encode_xh<31, 2>(data, data_words, num_cw, stream, st);
        case 63: return launch_encode_xh<63, 4>(data, data_words, num_cw, stream, st);
        case 127: return launch_encode_xh<127, 2>(data, data_words, num_cw, stream, st);
        case 255: return launch_encode_xh<255, 2>(data, data_words, num_cw, stream, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace hd
