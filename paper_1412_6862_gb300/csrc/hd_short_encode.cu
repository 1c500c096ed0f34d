// hd_short_encode.cu -- the encoder of the shortened codes (segments of any
// length n = 3..32767; the transmitter's side of the paper's packet splitter,
// Sec. II).
//
// A warp takes tiles of g consecutive segments.  Pass 1: teams of T lanes per
// segment build its position-domain words (bit p is position p) straight from
// the message bits in global memory -- word j >= 1 is one 32-bit window of the
// message, moved down by the checksum positions before it, word 0 an expansion
// of the first 26 bits -- keep them in shared memory and fold them into the
// checksum bits.  Pass 2: the tile's stream words, lane by lane, each one funnel
// shift of two position-domain words (plus the heads of the segments that begin
// inside it).  Words shared with a neighbouring tile are written with atomic
// AND/OR of the tile's own bits, so nothing needs clearing first.
//
// Bound: the issue slots and the shared-memory pipe.  A tile's message arrives by
// one bulk copy into the warp's stage (plain loads spread over several segments
// kept the L1 busy at 75 % of its wavefronts and took 1.4 to 2 times as long); the
// stage is free once pass 1 has read it, so the next tile's copy runs behind pass
// 2 and one stage a warp suffices.  Measured on GB300, 512 Mbit of segments, of the measured
// copy bandwidth: n = 100 / 544 / 1078 / 3212 / 16000 / 32767: 0.36 / 0.48 / 0.43 / 0.66 / 0.70 / 0.82
// (bit by bit before: 0.01); below n = 64, where a stream word holds parts of several
// segments, 0.08 to 0.23.
#include <algorithm>
#include <cstdint>

#include "hd_device.cuh"
#include "hd_internal.h"
#include "hd_lane.cuh"

namespace hd {
namespace {

constexpr uint32_t kWarps = 24;       // most warps of a CTA, one CTA per SM
constexpr uint32_t kSmemPerCta = 227u << 10;
constexpr uint32_t kMaxTile = 256;     // segments per tile

struct EncShortArgs {
    uint64_t data_words, num_cw, ntiles;
    uint32_t *status;
    uint32_t n, k, g;          // segment length, message bits, segments per tile
    uint32_t Y, ylast;         // position-domain words per segment, valid bits of the last one
    uint32_t ystride;          // words between two segments' position domains (odd, at least Y + 1)
    uint32_t off_area, warp_bytes;
};

__device__ __forceinline__ uint32_t low_bits(uint32_t b) { return b >= 32 ? 0xFFFFFFFFu : (1u << b) - 1u; }

// A warp's shared memory: the barrier, the message stage (a tile's bits behind up to 127
// others, in whole 16-byte pieces, and slack for the last window) and the
// position-domain words of g segments.
constexpr uint32_t kOffStage = 16;

inline uint32_t area_offset(uint32_t k, uint32_t g) { return kOffStage + (g * k + 254u) / 128u * 16u + 16u; }

inline uint32_t warp_smem(uint32_t k, uint32_t ystride, uint32_t g)
{
    return (area_offset(k, g) + g * ystride * 4u + 15u) / 16u * 16u;
}

// Pass 1 for one segment per team: the lane's position-domain words tl + T*i
// into `y` and their fold.  x is the XOR of the words; h the XOR of the
// indices i of the odd-parity words.  Four words at a time: the two low index
// bits come from XORs of the words that have them, so one popcount serves four
// words.  J0: floor(log2(32 tl)) (tl > 0), mask0: ~1 where word tl begins with a
// checksum position.
template <int TLOG>
__device__ __forceinline__ void fold_segment(const uint32_t *st, int32_t bit0, uint32_t Y, uint32_t ylast,
                                             uint32_t tl, uint32_t J0, uint32_t mask0, uint32_t *y, uint32_t &x_out,
                                             uint32_t &h_out)
{
    constexpr uint32_t T = 1u << TLOG;
    const uint32_t last = Y - 1u;
    uint32_t x = 0, A = 0, B = 0, hq = 0;
    // words past the segment are 0, the last one holds positions up to n only
    auto trim = [&](uint32_t j, uint32_t v) { return j < last ? v : j == last ? v & ylast : 0u; };
    auto take = [&](const uint32_t (&v)[4], uint32_t q) {
        A ^= v[1] ^ v[3];
        B ^= v[2] ^ v[3];
        const uint32_t b = v[0] ^ v[1] ^ v[2] ^ v[3];
        x ^= b;
        hq ^= q & (0u - parity32(b));
    };
    // word j (>= 1, floor(log2(32 j)) = J) is the window at message bit 32 j - J - 2
    {  // i = 0..3
        uint32_t v[4];
        const int32_t b = tl == 0 ? bit0 : bit0 - (int32_t)J0 - 2;
        const uint32_t *p = st + (b >> 5) + (int32_t)tl;
        v[0] = tl < Y ? __funnelshift_r(p[0], p[1], (uint32_t)b & 31u) : 0u;
        if (tl == 0) v[0] = expand_runs<5>(v[0]);
        v[0] = trim(tl, v[0] & mask0);
#pragma unroll
        for (uint32_t u = 1; u < 4; ++u) {
            v[u] = 0u;
            if (u * T >= Y) continue;  // the whole warp: short segments have no such words
            const int32_t bu = bit0 - (int32_t)(7u + TLOG + (u >> 1));
            const uint32_t j = tl + u * T;
            const uint32_t *pu = st + (bu >> 5) + (int32_t)tl;
            v[u] = j < Y ? __funnelshift_r(pu[u * T], pu[u * T + 1], (uint32_t)bu & 31u) : 0u;
            v[u] = trim(j, u < 3 && tl == 0 ? v[u] & ~1u : v[u]);
        }
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
            if (tl + u * T < Y) y[tl + u * T] = v[u];
        take(v, 0);
    }
    uint32_t J = 7u + TLOG;
    for (uint32_t q = 1; (q << (TLOG + 2)) < Y; ++q) {
        const bool octave = (q & (q - 1u)) == 0;  // i = 4q is a power of two: J goes up (q = 1 starts at its own)
        if (octave && q > 1) ++J;
        const int32_t b = bit0 - (int32_t)J - 2;
        const uint32_t j0 = tl + (q << (TLOG + 2)), sh = (uint32_t)b & 31u;
        const uint32_t *p = st + (b >> 5) + (int32_t)j0;
        uint32_t *yp = y + j0;
        uint32_t v[4];
        if (j0 + 3u * T < last) {
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) v[u] = __funnelshift_r(p[u * T], p[u * T + 1], sh);
            if (octave && tl == 0) v[0] &= ~1u;
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) yp[u * T] = v[u];
        } else {
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                const uint32_t j = j0 + u * T;
                v[u] = j < Y ? trim(j, __funnelshift_r(p[u * T], p[u * T + 1], sh)) : 0u;
                if (u == 0 && octave && tl == 0) v[0] &= ~1u;
                if (j < Y) yp[u * T] = v[u];
            }
        }
        take(v, q);
    }
    x_out = x;
    h_out = hq << 2 | parity32(B) << 1 | parity32(A);
}

// TLOG: log2 of the team size, so that a lane's word strides are constants.
template <int TLOG>
__global__ void __launch_bounds__(kWarps * 32, 1) k_encode_short(const uint32_t *__restrict__ data, uint32_t *__restrict__ stream, const EncShortArgs a)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t *wbase = smem + warp * a.warp_bytes;
    uint64_t *bar = reinterpret_cast<uint64_t *>(wbase);
    uint32_t *stage = reinterpret_cast<uint32_t *>(wbase + kOffStage);
    uint32_t *area = reinterpret_cast<uint32_t *>(wbase + a.off_area);
    constexpr uint32_t T = 1u << TLOG, G = 32u >> TLOG;
    const uint32_t tl = lane & (T - 1u), team = lane >> TLOG;
    const uint32_t n = a.n, k = a.k, Y = a.Y, ys = a.ystride;
    const uint32_t J0 = 36u - __clz(tl | 1u), mask0 = tl != 0 && (tl & (tl - 1u)) == 0 ? ~1u : ~0u;
    const uint64_t bulk_end = a.data_words * 4 / 16 * 16;  // bytes that 16-byte copies may read
    grid_dep_launch_dependents();
    grid_dep_wait();

    // the 16-byte groups that hold tile t's messages: first byte and length
    auto span = [&](uint64_t t, uint64_t &byte0, uint32_t &bytes) {
        const uint64_t c0 = t * a.g, c1 = min(c0 + a.g, a.num_cw);
        byte0 = c0 * k / 128 * 16;
        const uint64_t byte1 = min((c1 * k + 127) / 128 * 16, bulk_end);
        bytes = byte1 > byte0 ? (uint32_t)(byte1 - byte0) : 0u;
    };
    auto load = [&](uint64_t t) {
        uint64_t byte0;
        uint32_t bytes;
        span(t, byte0, bytes);
        mbar_arrive_expect_tx(bar, bytes);
        if (bytes) bulk_g2s(stage, reinterpret_cast<const uint8_t *>(data) + byte0, bytes, bar);
    };
    const uint32_t W = blockDim.x >> 5;
    const uint64_t tw = (uint64_t)gridDim.x * W;
    uint64_t t = (uint64_t)blockIdx.x * W + warp;
    if (lane == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
        if (t < a.ntiles) load(t);
    }
    __syncwarp();
    for (uint32_t phase = 0; t < a.ntiles; t += tw, phase ^= 1u) {
        const bool ok = mbar_wait_bounded(bar, phase);
        if (__any_sync(0xFFFFFFFFu, !ok)) {
            // nothing else of this warp is in flight; a late copy may still land, so wait once more
            if (lane == 0) {
                atomicOr(a.status, (uint32_t)HD_ERR_TIMEOUT);
                (void)mbar_wait_bounded(bar, phase);
            }
            break;
        }
        const uint64_t c0 = t * a.g;
        const uint32_t gcnt = (uint32_t)min((uint64_t)a.g, a.num_cw - c0);
        const uint64_t bit_out = c0 * n;
        const uint32_t off = (uint32_t)(c0 * k) & 127u;
        {  // words past the last 16-byte boundary of the messages arrive by plain loads
            uint64_t byte0;
            uint32_t bytes;
            span(t, byte0, bytes);
            const uint64_t w0 = byte0 >> 2, wb = (byte0 + bytes) >> 2, we = ((c0 + gcnt) * k + 31) >> 5;
            if (wb < we) {
                for (uint64_t w = wb + lane; w < we; w += 32) stage[w - w0] = data[w];
                __syncwarp();
            }
        }

        for (uint32_t cb = 0; cb < gcnt; cb += G) {
            const uint32_t c = cb + team;
            uint32_t *y = area + c * ys;
            uint32_t x = 0, h = 0;
            if (c < gcnt) {
                fold_segment<TLOG>(stage, (int32_t)(off + c * k), Y, a.ylast, tl, J0, mask0, y, x, h);
                if (tl == 0) y[Y] = 0u;
            }
            // the lane's share of the checksum bits in one word: the five low ones on bits
            // 1, 2, 4, 8, 16 of word 0's transform, the high ones (the XOR of the indices
            // j = tl + T*i of odd-parity words) from bit 17 up; XOR over the team
            h = (h << TLOG) ^ (parity32(x) ? tl : 0u);
            uint32_t chk = (superset_xor<5>(x) & 0x00010116u) | h << 17;
            if constexpr (T == 32)
                chk = __reduce_xor_sync(0xFFFFFFFFu, chk);
            else
                for (uint32_t o = T >> 1; o > 0; o >>= 1)  // stays inside aligned groups of T lanes
                    chk ^= __shfl_xor_sync(0xFFFFFFFFu, chk, o);
            __syncwarp();  // the team's words are in place
            if (c < gcnt) {
                // checksum positions 1, 2, 4, 8, 16 lie in word 0 (those past n do not exist and
                // their parities are 0: no position has such a bit), 32 * 2^b in word 2^b
                if (tl == 0) y[0] |= chk & 0x00010116u;
                for (uint32_t b = tl; b < 10u && (1u << b) < Y; b += T) y[1u << b] |= (chk >> (17u + b)) & 1u;
            }
        }
        // the stage has been read: the next tile's messages arrive behind pass 2
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0 && t + tw < a.ntiles) load(t + tw);

        // pass 2: stream words, counted from the word holding the tile's first bit.  Segment c
        // covers the tile's bits [s, s + n), s = ob + c * n.
        const uint32_t ob = (uint32_t)bit_out & 31u;
        uint32_t *out = stream + (bit_out >> 5);
        const bool last_tile = c0 + gcnt == a.num_cw;
        // words inside one segment: the shift is the segment's own
        for (uint32_t c = team; c < gcnt; c += G) {
            const uint32_t s = ob + c * n, w1 = (s + 31u) >> 5, w2 = (s + n) >> 5;
            const uint32_t sh = (1u - s) & 31u;
            const uint32_t *y = area + c * ys + ((32u * w1 - s + 1u) >> 5) + tl;
            uint32_t *o = out + w1 + tl;
            int32_t left = (int32_t)(w2 - w1) - (int32_t)tl;  // words from this lane's first one on
            for (; left > (int32_t)(3 * T); left -= (int32_t)(4 * T), y += 4 * T, o += 4 * T) {
                uint32_t v[4];
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) v[u] = __funnelshift_r(y[u * T], y[u * T + 1], sh);
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) o[u * T] = v[u];
            }
            for (; left > 0; left -= (int32_t)T, y += T, o += T) *o = __funnelshift_r(y[0], y[1], sh);
        }
        // the other words, one lane each: the first one when it begins in the tile before, and
        // the ones a segment ends in, by the segment that reaches back to the word's first bit
        if (ob != 0 && lane == 0) {
            uint32_t v = area[0] >> 1, avail = n;
            for (uint32_t c = 1; avail < 32u && c < gcnt; ++c, avail += n) v |= (area[c * ys] >> 1) << avail;
            v <<= ob;
            uint32_t own = ~low_bits(ob);
            if (ob + gcnt * n < 32u && !last_tile) own &= low_bits(ob + gcnt * n);
            atomicAnd(out, v | ~own);
            atomicOr(out, v & own);
        }
        for (uint32_t c = lane; c < gcnt; c += 32) {
            const uint32_t s = ob + c * n, w = (s + n) >> 5;
            uint32_t avail = (s + n) & 31u;
            if (avail == 0 || s > 32u * w) continue;
            const uint32_t *y = area + c * ys;
            const uint32_t q = 32u * w - s + 1u;  // position of the word's first bit
            uint32_t v = __funnelshift_r(y[q >> 5], y[(q >> 5) + 1], q & 31u);
            for (uint32_t e = c + 1; avail < 32u && e < gcnt; ++e, avail += n) v |= (area[e * ys] >> 1) << avail;
            if (avail < 32u && !last_tile) {
                atomicAnd(&out[w], v | ~low_bits(avail));
                atomicOr(&out[w], v);
            } else {
                out[w] = v;
            }
        }
        __syncwarp();  // the next tile overwrites the area
    }
}

// How a stream is cut: segments per tile, log2 of the team size and the warps per CTA.
// The warps work through their tiles in step, so every one of the R rounds should be
// full, g = ceil(num_cw / (R * warps)), and g should fill the lanes of the teams: a round of
// 32 / T segments costs a lane its ceil(Y / 4T) blocks of four words (dearer the more segments
// a warp's accesses are spread over, and where they share few banks) and a fixed chain
// (the transform, the team's XOR, the inserts, the heads), and more the more warps share the SM.
// Weights fitted on GB300 to every T, seven warp counts and three R at 20 lengths and streams
// of 128 .. 512 Mbit: the pick is 3.5 % off the fastest on average.  Against g of the
// fewest rounds on three CTAs of 8 warps with areas of 1056 words: 22 lengths of 16 .. 32,767 at
// eight sizes 1.09x on average (512 Mbit of n = 200 65 -> 48 us, 3212 41 -> 30, 4095 59 -> 39;
// at worst 1.15x slower, 128 Mbit of n = 2500).
struct EncShape {
    uint32_t g, tlog, warps;
};

EncShape encode_shape(uint32_t n, uint32_t k, uint32_t ystride, uint64_t num_cw, uint64_t ctas)
{
    const uint32_t Y = (n + 32) / 32;
    const BankWays &ways = bank_ways(k);
    EncShape pick{1, 0, kWarps};
    uint64_t best = ~0ull;
    auto consider = [&](uint64_t R, uint32_t g, uint32_t w) {
        for (uint32_t lg = 0; lg <= 5; ++lg) {
            const uint32_t G = 32u >> lg, blocks = (Y + (4u << lg) - 1) >> (lg + 2);
            const uint64_t round = (uint64_t)blocks * std::max(40 + 6 * std::min(G, g), 32u * ways[lg]) + 200;
            const uint64_t cost = R * ((g + G - 1) >> (5 - lg)) * round * (w + 12);
            if (cost < best) {
                best = cost;
                pick = EncShape{g, lg, w};
            }
        }
    };
    // the most segments that fit one of w warps' share of the shared memory (warp_smem)
    auto most = [&](uint32_t w) { return std::min((kSmemPerCta / w - 96u) * 8u / (k + 32u * ystride), kMaxTile); };
    // up to half of that in one round of all warps; more take two rounds at least, so that
    // the second one's loads run behind the first one's stores
    if (num_cw <= ctas * kWarps * std::max(1u, most(kWarps) / 2)) {
        consider(1, (uint32_t)((num_cw + ctas * kWarps - 1) / (ctas * kWarps)), kWarps);
        return pick;
    }
    for (uint32_t w = kWarps; w >= 12; w -= 2) {
        const uint64_t warps = ctas * w, gmax = most(w);
        const uint64_t r0 = std::max<uint64_t>(2, (num_cw + gmax * warps - 1) / (gmax * warps));
        for (uint64_t R = r0; R < r0 + 3; ++R) consider(R, (uint32_t)((num_cw + R * warps - 1) / (R * warps)), w);
    }
    return pick;
}

}  // namespace

cudaError_t launch_encode_short(const uint32_t *data, uint32_t n, uint32_t k, uint64_t num_cw, uint32_t *stream,
                                cudaStream_t st)
{
    EncShortArgs a{};
    a.data_words = words_for_bits(num_cw * k);
    a.num_cw = num_cw;
    a.status = status_ptr();
    if (a.status == nullptr) return cudaErrorInvalidSymbol;
    a.n = n;
    a.k = k;
    a.Y = (n + 32) / 32;
    a.ylast = n % 32 == 31 ? 0xFFFFFFFFu : (2u << (n % 32)) - 1u;
    a.ystride = (a.Y + 1) | 1u;
    static void (*const kernels[6])(const uint32_t *, uint32_t *, EncShortArgs) = {k_encode_short<0>, k_encode_short<1>, k_encode_short<2>,
                                                     k_encode_short<3>, k_encode_short<4>, k_encode_short<5>};
    const uint64_t ctas = (uint64_t)num_sms();
    const EncShape shape = encode_shape(n, k, a.ystride, num_cw, ctas);
    a.g = shape.g;
    a.ntiles = (num_cw + a.g - 1) / a.g;
    a.off_area = area_offset(k, a.g);
    a.warp_bytes = warp_smem(k, a.ystride, a.g);
    const auto kern = kernels[shape.tlog];
    if (stream_blocks_per_sm(reinterpret_cast<const void *>(kern), kWarps * 32, kSmemPerCta) <= 0)
        return cudaErrorInvalidConfiguration;
    // at most one tile per warp: the warps spread over all SMs
    const uint32_t W = (uint32_t)std::min<uint64_t>(shape.warps, (a.ntiles + ctas - 1) / ctas);
    const int grid = decode_grid((a.ntiles + W - 1) / W, ctas);
    return launch_kernel(kern, dim3((unsigned)grid), dim3(W * 32), W * a.warp_bytes, st, true, data, stream, a);
}

}  // namespace hd
