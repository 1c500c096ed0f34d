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
// Bound: the issue slots, about 30 instructions per 32 output words beside 23
// bytes a clock of HBM.  Message words are read by plain loads, eight in flight
// a lane: a segment's windows start at any bit, every word is read twice within
// a few instructions (the second time from L1), and 48 warps an SM hide the
// rest, so that stages and barriers would only cost shared memory.
#include <algorithm>
#include <cstdint>

#include "hd_device.cuh"
#include "hd_internal.h"
#include "hd_lane.cuh"

namespace hd {
namespace {

constexpr int kWarps = 8;
constexpr uint32_t kAreaWords = 1056;  // position-domain words a warp holds: 48 warps an SM, and n = 32767 fits
constexpr uint32_t kMaxTile = 256;     // segments per tile

struct EncShortArgs {
    const uint32_t *data;
    uint32_t *stream;
    uint64_t data_words, num_cw, ntiles;
    uint32_t n, k, g;          // segment length, message bits, segments per tile
    uint32_t Y, ylast;         // position-domain words per segment, valid bits of the last one
    uint32_t ystride;          // words between two segments' position domains (odd, at least Y + 1)
    uint32_t tlog;             // log2 of the team size
    uint32_t step_cw, step_bits;  // 1024 stream bits (32 words) further: segments and bits
};

__device__ __forceinline__ uint32_t low_bits(uint32_t b) { return b >= 32 ? 0xFFFFFFFFu : (1u << b) - 1u; }

// Pass 1 for one segment per team: the lane's position-domain words tl + T*i
// into `y` and their fold.  x is the XOR of the words; h the XOR of the
// indices i of the odd-parity words.  Four words at a time: the two low index
// bits come from XORs of the words that have them, so one popcount serves four
// words.  SAFE: every window lies inside the message buffer.
template <bool SAFE>
__device__ __forceinline__ void fold_segment(const EncShortArgs &a, const uint32_t *src, int32_t bit0, uint32_t tl,
                                             uint32_t *y, uint32_t &x_out, uint32_t &h_out)
{
    const uint32_t tlog = a.tlog, T = 1u << tlog, Y = a.Y, last = Y - 1u;
    const uint32_t *end = a.data + a.data_words;
    auto ld = [&](const uint32_t *p) { return SAFE || p < end ? __ldg(p) : 0u; };
    // window of word j (>= 1, floor(log2(32 j)) = J): message bit 32 j - J - 2
    auto window = [&](uint32_t j, uint32_t J) {
        const int32_t b = bit0 - (int32_t)J - 2;
        const uint32_t *p = src + (b >> 5) + (int32_t)j;
        return __funnelshift_r(ld(p), ld(p + 1), (uint32_t)b & 31u);
    };
    uint32_t x = 0, A = 0, B = 0, hq = 0;
    // words past the segment are 0, the last one holds positions up to n only
    auto trim = [&](uint32_t j, uint32_t v) { return j < last ? v : j == last ? v & a.ylast : 0u; };
    auto take = [&](const uint32_t (&v)[4], uint32_t q) {
        A ^= v[1] ^ v[3];
        B ^= v[2] ^ v[3];
        const uint32_t b = v[0] ^ v[1] ^ v[2] ^ v[3];
        x ^= b;
        hq ^= q & (0u - parity32(b));
    };
    {  // i = 0..3
        uint32_t v[4];
        if (tl == 0)
            v[0] = trim(0, expand_runs<5>(__funnelshift_r(ld(src + (bit0 >> 5)), ld(src + (bit0 >> 5) + 1),
                                                          (uint32_t)bit0 & 31u)));
        else
            v[0] = tl < Y ? trim(tl, window(tl, 36u - __clz(tl)) & ((tl & (tl - 1u)) == 0 ? ~1u : ~0u)) : 0u;
#pragma unroll
        for (uint32_t u = 1; u < 4; ++u) {
            const uint32_t j = tl + (u << tlog);
            v[u] = j < Y ? trim(j, window(j, 5u + tlog + (u >> 1)) & (tl == 0 && u < 3 ? ~1u : ~0u)) : 0u;
        }
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
            if (tl + (u << tlog) < Y) y[tl + (u << tlog)] = v[u];
        take(v, 0);
    }
    for (uint32_t q = 1, J = 7u + tlog; (q << (tlog + 2)) < Y; ++q) {
        const bool octave = (q & (q - 1u)) == 0;  // i = 4q is a power of two: J goes up (q = 1 starts at its own)
        if (octave && q > 1) ++J;
        const int32_t b = bit0 - (int32_t)J - 2;
        const uint32_t j0 = tl + (q << (tlog + 2)), sh = (uint32_t)b & 31u;
        const uint32_t *p = src + (b >> 5) + (int32_t)j0;
        uint32_t v[4];
        if (j0 + 3u * T < last) {
            uint32_t lo[4], hi[4];
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                lo[u] = ld(p + u * T);
                hi[u] = ld(p + u * T + 1);
            }
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) v[u] = __funnelshift_r(lo[u], hi[u], sh);
            if (octave && tl == 0) v[0] &= ~1u;
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) y[j0 + u * T] = v[u];
        } else {
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                const uint32_t j = j0 + u * T;
                v[u] = j < Y ? trim(j, __funnelshift_r(ld(p + u * T), ld(p + u * T + 1), sh)) : 0u;
                if (u == 0 && octave && tl == 0) v[0] &= ~1u;
                if (j < Y) y[j] = v[u];
            }
        }
        take(v, q);
    }
    x_out = x;
    h_out = hq << 2 | parity32(B) << 1 | parity32(A);
}

__global__ void __launch_bounds__(kWarps * 32) k_encode_short(const EncShortArgs a)
{
    extern __shared__ uint32_t s_area[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *area = s_area + warp * kAreaWords;
    const uint32_t tlog = a.tlog, T = 1u << tlog, tl = lane & (T - 1u), team = lane >> tlog, G = 32u >> tlog;
    const uint32_t n = a.n, k = a.k, Y = a.Y, ys = a.ystride;
    grid_dep_launch_dependents();
    grid_dep_wait();
    for (uint64_t t = (uint64_t)blockIdx.x * kWarps + warp; t < a.ntiles; t += (uint64_t)gridDim.x * kWarps) {
        const uint64_t c0 = t * a.g;
        const uint32_t gcnt = (uint32_t)min((uint64_t)a.g, a.num_cw - c0);
        const uint64_t bit_in = c0 * k, bit_out = c0 * n;
        const uint32_t *src = a.data + (bit_in >> 5);
        const uint32_t off = (uint32_t)bit_in & 31u;
        // windows reach at most 63 bits past the tile's messages
        const bool safe = ((bit_in + (uint64_t)gcnt * k + 95u) >> 5) < a.data_words;

        for (uint32_t cb = 0; cb < gcnt; cb += G) {
            const uint32_t c = cb + team;
            uint32_t *y = area + c * ys;
            uint32_t x = 0, h = 0;
            if (c < gcnt) {
                if (safe)
                    fold_segment<true>(a, src, (int32_t)(off + c * k), tl, y, x, h);
                else
                    fold_segment<false>(a, src, (int32_t)(off + c * k), tl, y, x, h);
                if (tl == 0) y[Y] = 0u;
            }
            // index j = tl + T*i: the team's XOR gives the high checksum bits
            h = (h << tlog) ^ (parity32(x) ? tl : 0u);
            for (uint32_t o = T >> 1; o > 0; o >>= 1) {  // stays inside aligned groups of T lanes
                x ^= __shfl_xor_sync(0xFFFFFFFFu, x, o);
                h ^= __shfl_xor_sync(0xFFFFFFFFu, h, o);
            }
            __syncwarp();  // the team's words are in place
            if (c < gcnt) {
                // checksum positions 1, 2, 4, 8, 16 lie in word 0 (those past n do not exist and
                // their parities are 0: no position has such a bit), 32 * 2^b in word 2^b
                if (tl == 0) y[0] |= superset_xor<5>(x) & 0x00010116u;
                for (uint32_t b = tl; b < 10u && (1u << b) < Y; b += T) y[1u << b] |= (h >> b) & 1u;
            }
        }
        __syncwarp();

        // pass 2: stream words, counted from the word holding the tile's first bit
        const uint32_t ob = (uint32_t)bit_out & 31u, total = gcnt * n;
        uint32_t *out = a.stream + (bit_out >> 5);
        const bool last_tile = c0 + gcnt == a.num_cw;
        if (ob != 0 && lane == 0) {  // the first word's low bits belong to the tile before
            uint32_t v = area[0] >> 1, avail = n;
            for (uint32_t c = 1; avail < 32u && c < gcnt; ++c, avail += n) v |= (area[c * ys] >> 1) << avail;
            v <<= ob;
            uint32_t own = ~low_bits(ob);
            if (ob + total < 32u && !last_tile) own &= low_bits(ob + total);
            atomicAnd(out, v | ~own);
            atomicOr(out, v & own);
        }
        // the lane's first whole word, as (segment, bits before it), then 32 words on at a time
        uint32_t w = (uint32_t)lane + (ob != 0 ? 1u : 0u);
        const uint32_t bit = 32u * w - ob;
        uint32_t c = bit / n, r = bit - c * n;
        for (; 32u * w < ob + total; w += 32) {
            const uint32_t *y = area + c * ys;
            const uint32_t q = r + 1u;  // position of the word's first bit
            uint32_t v = __funnelshift_r(y[q >> 5], y[(q >> 5) + 1], q & 31u);
            uint32_t avail = n - r;
            if (avail < 32u) {  // heads of the segments that begin in this word
                for (uint32_t e = c + 1; avail < 32u && e < gcnt; ++e, avail += n) v |= (area[e * ys] >> 1) << avail;
            }
            if (avail < 32u && !last_tile) {
                atomicAnd(&out[w], v | ~low_bits(avail));
                atomicOr(&out[w], v);
            } else {
                out[w] = v;
            }
            c += a.step_cw;
            r += a.step_bits;
            if (r >= n) {
                r -= n;
                ++c;
            }
        }
        __syncwarp();  // the next tile overwrites the area
    }
}

}  // namespace

cudaError_t launch_encode_short(const uint32_t *data, uint32_t n, uint32_t k, uint64_t num_cw, uint32_t *stream,
                                cudaStream_t st)
{
    EncShortArgs a{};
    a.data = data;
    a.stream = stream;
    a.data_words = words_for_bits(num_cw * k);
    a.num_cw = num_cw;
    a.n = n;
    a.k = k;
    a.Y = (n + 32) / 32;
    a.ylast = n % 32 == 31 ? 0xFFFFFFFFu : (2u << (n % 32)) - 1u;
    a.ystride = (a.Y + 1) | 1u;
    constexpr uint32_t smem = kWarps * kAreaWords * 4;
    const int bps = stream_blocks_per_sm(reinterpret_cast<const void *>(k_encode_short), kWarps * 32, smem);
    if (bps <= 0) return cudaErrorInvalidConfiguration;
    const uint64_t cap = (uint64_t)num_sms() * (uint64_t)bps;
    // segments per tile: what the area holds, fewer when the stream then has
    // less than one tile per resident warp
    const uint64_t share = (num_cw + cap * kWarps - 1) / (cap * kWarps);
    a.g = (uint32_t)std::min<uint64_t>({kAreaWords / a.ystride, kMaxTile, share});
    // team size: a round of 32 / T segments costs a lane its ceil(Y / 4T) blocks of
    // four words and a fixed chain (the reduction, the butterfly, the inserts)
    uint64_t best = ~0ull;
    for (uint32_t lg = 0; lg <= 5; ++lg) {
        const uint32_t T = 1u << lg, G = 32u >> lg;
        const uint64_t cost = (uint64_t)((a.g + G - 1) / G) * ((a.Y + 4 * T - 1) / (4 * T) * 40 + 60 + 8 * lg);
        if (cost < best) {
            best = cost;
            a.tlog = lg;
        }
    }
    a.step_cw = 1024 / n;
    a.step_bits = 1024 % n;
    a.ntiles = (num_cw + a.g - 1) / a.g;
    const int grid = decode_grid((a.ntiles + kWarps - 1) / kWarps, cap);
    return launch_kernel(k_encode_short, dim3((unsigned)grid), dim3(kWarps * 32), smem, st, true, a);
}

}  // namespace hd
