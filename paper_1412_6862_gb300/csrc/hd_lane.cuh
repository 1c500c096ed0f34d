// hd_lane.cuh -- one codeword per lane: a warp takes a tile of 32 consecutive
// codewords of a compile-time length straight from global memory, with bounds
// checks, so it covers ragged tails and streams too short for whole chunks.
// 32 codewords of n bits fill n words (32 messages k words), so a tile starts
// on a word boundary on both sides.  Also the checksum arithmetic of the
// encoders.
#pragma once

#include "hd_device.cuh"
#include "hd_tile.cuh"

namespace hd {

// Words a lane's slot holds in a tile's merge area: the codeword's words, a
// zero spare for the two-word reads, and an odd stride against bank conflicts.
__host__ __device__ constexpr int lane_slot_words(int words) { return (words + 1) | 1; }

// v repeated in every field of 2^M bits of a word.
template <int M>
__host__ __device__ constexpr uint32_t in_fields(uint32_t v)
{
    uint32_t r = 0;
    for (int f = 0; f < 32; f += 1 << M) r |= v << f;
    return r;
}

// Redundancy insertion, the inverse of compress_runs: in every 2^M-bit field
// the data bits 0 .. go up to positions 3, 5..7, 9..15, 17..31, checksum
// positions and bit 0 become 0.
template <int M>
__device__ __forceinline__ uint32_t expand_runs(uint32_t d)
{
    constexpr uint32_t data = M >= 5 ? 0xFFFEFEE8u : M == 4 ? 0xFEE8FEE8u : 0xE8E8E8E8u;
    if constexpr (M >= 4) d = bitsel(in_fields<M>(0x0000000Fu), d, d << 2);  // runs 3, 4 two bits up
    d = bitsel(in_fields<M>(M >= 4 ? 0x00001FC1u : 0x01u), d, d << 1);       // runs 2, 4 one more
    return (d << 3) & data;
}

// Parity of a word, 0 or 1.
__device__ __forceinline__ uint32_t parity32(uint32_t v) { return (uint32_t)__popc(v) & 1u; }

// Every third bit of a word from the low 11 bits of x (bit i to bit 3i).
__device__ __forceinline__ uint32_t spread3(uint32_t x)
{
    x = (x | x << 16) & 0xFF0000FFu;
    x = (x | x << 8) & 0x0F00F00Fu;
    x = (x | x << 4) & 0xC30C30C3u;
    return (x | x << 2) & 0x49249249u;
}

// 32 bits of the message words r from bit `start` on (a constant once the
// callers' loops are unrolled); bits past the array read as 0.
template <int R>
__device__ __forceinline__ uint32_t bits_at(const uint32_t (&r)[R], int start)
{
    const int a = start >> 5, sh = start & 31;
    const uint32_t lo = a < R ? r[a] : 0u;
    if (sh == 0) return lo;
    const uint32_t hi = a + 1 < R ? r[a + 1] : 0u;
    return __funnelshift_r(lo, hi, sh);
}

// The position-domain words of a codeword of at least one word (n >= 31) from
// its message at bit `start` of r: bit p of y is position p, the checksum bits
// in place, and with XH the overall parity at position 0.
template <int N_, bool XH, int R>
__device__ __forceinline__ void encode_words(const uint32_t (&r)[R], int start, uint32_t (&y)[Code<N_>::Wy])
{
    using C = Code<N_>;
    y[0] = expand_runs<5>(bits_at(r, start));
    uint32_t f = y[0];
    int at = start + 26;
#pragma unroll
    for (int w = 1; w < C::Wy; ++w) {
        if ((w & (w - 1)) == 0) {
            y[w] = bits_at(r, at - 1) & ~1u;  // position 32w is a checksum position
            at += 31;
        } else {
            y[w] = bits_at(r, at);
            at += 32;
        }
        f ^= y[w];
    }
    y[0] |= superset_xor<5>(f) & 0x00010116u;
#pragma unroll
    for (int t = 0; (1 << t) < C::Wy; ++t) {
        uint32_t g = 0;
#pragma unroll
        for (int w = 0; w < C::Wy; ++w)
            if ((w >> t) & 1) g ^= y[w];
        y[1 << t] |= parity32(g);
    }
    if constexpr (XH) {
        uint32_t all = 0;
#pragma unroll
        for (int w = 0; w < C::Wy; ++w) all ^= y[w];
        y[0] |= parity32(all);
    }
}

// The codewords of n = 3, 7 or 15 that fit one word (fields of n + 1 bits,
// bit p of a field is position p), from their messages in the low bits of d.
template <int N_, bool XH>
__device__ __forceinline__ uint32_t encode_fields(uint32_t d)
{
    using C = Code<N_>;
    if constexpr (N_ == 3) {
        d &= 0xFFu;  // a data bit and its two copies (and, with XH, a third)
        d = (d | d << 12) & 0x000F000Fu;
        d = (d | d << 6) & 0x03030303u;
        d = (d | d << 3) & 0x11111111u;
        return d * (XH ? 15u : 14u);
    } else {
        if constexpr (N_ == 7) {
            d = (d | d << 8) & 0x00FF00FFu;
            d = (d | d << 4) & 0x0F0F0F0Fu;
        } else {
            d = (d & 0x7FFu) | ((d << 5) & 0x07FF0000u);
        }
        const uint32_t y = expand_runs<C::m>(d);
        const uint32_t z = superset_xor<C::m>(y);
        uint32_t r = y | (z & in_fields<C::m>(0x0116u & ((1u << (1 << C::m)) - 1u)));
        if constexpr (XH) {
            // overall parity: bit 0 of z (the data's) and the checksum bits 1, 2, 4, 8
            uint32_t p = z & in_fields<C::m>(0x0117u & ((1u << (1 << C::m)) - 1u));
            if constexpr (C::m == 4) p ^= p >> 8;
            p ^= p >> 4;
            p ^= (p >> 1) ^ (p >> 2);
            r |= p & in_fields<C::m>(1u);
        }
        return r;
    }
}

// Codewords encode_fields makes at once.
template <int N_>
constexpr int kFieldCodewords = 32 / (N_ + 1);

// Without the overall parity bit the fields lose their bit 0: n bits each.
template <int N_>
__device__ __forceinline__ uint32_t close_fields(uint32_t y)
{
    if constexpr (N_ == 15) return ((y & 0x0000FFFEu) >> 1) | ((y & 0xFFFE0000u) >> 2);
    y = ((y & 0x00FE00FEu) >> 1) | ((y & 0xFE00FE00u) >> 2);
    return (y & 0x3FFFu) | ((y >> 2) & 0x0FFFC000u);
}

// Encode a part of G codewords whose messages are r[] (bit 0 of r[0] is the
// first codeword's data bit 0), appending n bits per codeword to `op`.
template <int N_, int G, int R, class OP>
__device__ __forceinline__ void encode_part(const uint32_t (&r)[R], OP &op)
{
    using C = Code<N_>;
    if constexpr (N_ == 3) {
        // 32 codewords of three equal bits are three words
        static_assert(G == 32, "one thread per 32-codeword tile");
        const uint32_t d = r[0];
        op.append(spread3(d & 0x7FFu) * 7u, 32);
        op.append(spread3((d >> 11) & 0x7FFu) * 14u + ((d >> 10) & 1u), 32);
        op.append(spread3(d >> 22) * 28u + ((d >> 21) & 1u) * 3u, 32);
    } else if constexpr (C::Wy == 1 && N_ < 31) {
        constexpr int F = kFieldCodewords<N_>;
#pragma unroll
        for (int c = 0; c < G; c += F) {
            uint32_t d = bits_at(r, c * C::k);
            if constexpr (F * C::k < 32) d &= (1u << (F * C::k)) - 1u;
            op.append(close_fields<N_>(encode_fields<N_, false>(d)), F * N_);
        }
    } else {
#pragma unroll
        for (int c = 0; c < G; ++c) {
            uint32_t y[C::Wy];
            encode_words<N_, false>(r, c * C::k, y);
            op.append(y[0] >> 1, 31);
#pragma unroll
            for (int w = 1; w < C::Wy; ++w) op.append(y[w], 32);
        }
    }
    op.finish();
}

// Words [0, words) of a tile of 32 pieces of LEN bits each, piece c at bit
// `first` of slot c, back to back: lane q writes words q, q + 32, ...
template <int LEN, int SLOT>
__device__ __forceinline__ void merge_tile(const uint32_t *slots, int first, uint32_t *__restrict__ out,
                                           uint32_t words, int lane)
{
#pragma unroll
    for (int q0 = 0; q0 < LEN; q0 += 32) {
        const uint32_t q = (uint32_t)q0 + (uint32_t)lane;
        if (q >= words) break;  // words <= LEN
        uint32_t c = (32u * q) / (uint32_t)LEN, o = 32u * q - c * (uint32_t)LEN, v = 0, filled = 0;
#pragma unroll
        for (int step = 0; step < 31 / LEN + 2; ++step) {
            if (filled < 32u && c < 32u) {
                const uint32_t *s = slots + c * SLOT;
                const uint32_t b = o + (uint32_t)first, left = (uint32_t)LEN - o;
                uint32_t x = __funnelshift_r(s[b >> 5], s[(b >> 5) + 1], b & 31u);
                if (left < 32u) x &= (1u << left) - 1u;
                v |= x << filled;
                filled += left;  // past 32 once the piece has more bits than the word takes
                ++c;
                o = 0;
            }
        }
        out[q] = v;
    }
}

// Encode tile t (codewords 32t .. 32t + 31, those below num_cw) of the plain
// code: `slots` holds 32 * lane_slot_words(Wy) words of this warp's shared
// memory.  Every lane of the warp calls it.
template <int N_>
__device__ __forceinline__ void encode_lane_tile(const uint32_t *__restrict__ data, uint64_t data_words,
                                                 uint64_t num_cw, uint64_t t, uint32_t *__restrict__ stream,
                                                 uint64_t stream_words, uint32_t *slots, int lane)
{
    using C = Code<N_>;
    constexpr int SLOT = lane_slot_words(C::Wy), R = (C::k + 31) / 32;
    const uint32_t *src = data + t * C::k;
    const uint32_t have = (uint32_t)min((uint64_t)C::k, data_words - t * C::k);  // words of the tile
    const uint32_t bit = (uint32_t)lane * C::k, a = bit >> 5, sh = bit & 31u;
    const bool valid = t * 32 + lane < num_cw;
    uint32_t d[R];
    uint32_t lo = valid && a < have ? src[a] : 0u;
#pragma unroll
    for (int w = 0; w < R; ++w) {
        const uint32_t hi = valid && a + w + 1 < have ? src[a + w + 1] : 0u;
        d[w] = __funnelshift_r(lo, hi, sh);
        lo = hi;
    }
    if constexpr (C::k % 32 != 0) d[R - 1] &= (1u << (C::k % 32)) - 1u;
    uint32_t *mine = slots + lane * SLOT;
    if constexpr (N_ < 31) {
        mine[0] = encode_fields<N_, false>(d[0]) & ((2u << N_) - 1u);
    } else {
        uint32_t y[C::Wy];
        encode_words<N_, false>(d, 0, y);
#pragma unroll
        for (int w = 0; w < C::Wy; ++w) mine[w] = y[w];
    }
    mine[C::Wy] = 0u;
    __syncwarp();
    merge_tile<N_, SLOT>(slots, 1, stream + t * N_, (uint32_t)min((uint64_t)N_, stream_words - t * N_), lane);
    __syncwarp();
}

// Decode tile t (codewords 32t .. 32t + 31, those below num_cw) of the plain
// code, or with XH of its SECDED extension (decode_part's conventions):
// `slots` holds 32 * lane_slot_words(ceil(k / 32)) words of this warp's shared
// memory.  syn_type 0 (none), 1 (u8) or 2 (u16); the nonzero and detected
// syndromes of the tile are added to errs and dets (the same in every lane).
// Every lane of the warp calls it.
template <int N_>
constexpr int kLaneDataSlot = lane_slot_words((Code<N_>::k + 31) / 32);

template <int N_, bool XH>
__device__ __forceinline__ void decode_lane_tile(const uint32_t *__restrict__ in, uint64_t in_words, uint64_t num_cw,
                                                 uint64_t t, uint32_t *__restrict__ out, uint64_t out_words,
                                                 void *__restrict__ syn, int syn_type, uint32_t *slots, int lane,
                                                 uint32_t &errs, uint32_t &dets)
{
    using C = Code<N_>;
    constexpr int L = N_ + (XH ? 1 : 0), D = (C::k + 31) / 32, SLOT = kLaneDataSlot<N_>;
    const uint32_t *src = in + t * L;
    const uint32_t have = (uint32_t)min((uint64_t)L, in_words - t * L);  // words of the tile
    const uint64_t i = t * 32 + lane;
    const bool valid = i < num_cw;
    // position p is tile bit lane * L + p (XH), lane * L + p - 1 (lane 0's position 0 would be word -1)
    const int32_t bit = lane * L - (XH ? 0 : 1), a = bit >> 5;
    const uint32_t sh = (uint32_t)bit & 31u;
    uint32_t y[C::Wy];
    auto word = [&](int32_t w) { return valid && (uint32_t)w < have ? src[w] : 0u; };
    uint32_t lo = word(a);
#pragma unroll
    for (int w = 0; w < C::Wy; ++w) {
        // SECDED codewords never straddle a word
        const uint32_t hi = XH ? (w + 1 < C::Wy ? word(a + w + 1) : 0u) : word(a + w + 1);
        y[w] = XH && L >= 32 ? lo : __funnelshift_r(lo, hi, sh);
        lo = hi;
    }
    if constexpr (!XH) y[0] &= ~1u;
    if constexpr (N_ < 31) y[0] &= (2u << N_) - 1u;
    const uint32_t s = part_syndrome<N_>(y);
    uint32_t sf = s, val = s;
    bool nonzero = s != 0u;
    if constexpr (XH) {
        uint32_t f = 0;
#pragma unroll
        for (int w = 0; w < C::Wy; ++w) f ^= y[w];
        const uint32_t P = parity32(f);
        sf = P ? s : 0xFFFFFFFFu;
        val = s | P << C::m;
        nonzero = val != 0u;
        dets += __popc(__ballot_sync(0xFFFFFFFFu, valid && P == 0u && s != 0u));
    }
    errs += __popc(__ballot_sync(0xFFFFFFFFu, valid && nonzero));
    if (valid) {
        if (syn_type == 1) static_cast<uint8_t *>(syn)[i] = (uint8_t)val;
        if (syn_type == 2) static_cast<uint16_t *>(syn)[i] = (uint16_t)val;
    }
#pragma unroll
    for (int w = 0; w < C::Wy; ++w) y[w] ^= shl_clamp(1u, sf - 32u * (uint32_t)w);
    if constexpr (N_ == 3) {
        const uint32_t v = __ballot_sync(0xFFFFFFFFu, (y[0] >> 3) & 1u);  // one data bit each: the tile's word
        if (lane == 0) out[t] = v;
    } else {
        // the data bits, packed: 26, then 31 or 32 per word
        uint32_t d[D];
        d[0] = compress_runs<(C::m < 5 ? C::m : 5)>(y[0]);
        if constexpr (C::m < 5) d[0] &= (1u << C::k) - 1u;
        int at = 26;
#pragma unroll
        for (int w = 1; w < C::Wy; ++w) {
            const bool chk = (w & (w - 1)) == 0;  // position 32w is a checksum position
            const uint32_t v = chk ? y[w] >> 1 : y[w];
            d[at / 32] |= v << (at % 32);
            const int end = at + (chk ? 31 : 32);
            if (end > (at / 32 + 1) * 32 || (end == (at / 32 + 1) * 32 && at / 32 + 1 < D))
                d[at / 32 + 1] = at % 32 == 0 ? 0u : v >> (32 - at % 32);
            at = end;
        }
        uint32_t *mine = slots + lane * SLOT;
#pragma unroll
        for (int w = 0; w < D; ++w) mine[w] = d[w];
        mine[D] = 0u;
        __syncwarp();
        merge_tile<C::k, SLOT>(slots, 0, out + t * C::k, (uint32_t)min((uint64_t)C::k, out_words - t * C::k), lane);
        __syncwarp();
    }
}

}  // namespace hd
