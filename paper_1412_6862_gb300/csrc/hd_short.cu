// hd_short.cu -- shortened Hamming codes: segments of any length n.
//
// The paper's decoder splits a packet of M bytes into t segments (Sec. II,
// Fig. 1; the evaluation of Sec. IV-A sweeps M = 400..2000 bytes and
// t = 2..6), and each segment carries its own checksum bits, so a segment is
// a codeword of a shortened code: n = k + r bits, r the smallest count with
// 2^r >= n + 1, checksum bits at the power-of-two positions 1..2^(r-1), data at
// the other positions.  A syndrome s <= n names the position to flip; a
// syndrome past n names none, and the codeword is counted as detected and
// left as received.
//
// Two decoders:
//  * k_short_tiles (n >= 960, large streams from n = 768; any k >= 64 where a configuration is chosen): each warp
//    takes tiles of g whole codewords, one at a time, into a shared-memory stage of its
//    own filled by a 1-D bulk copy (the next tile goes to L2 meanwhile).  Per tile:
//    (1) syndromes, teams of T lanes per codeword (g, T and the warps from a cost model),
//    each lane folding its stage words four at a time, then one XOR over the team; the
//    corrections flip bits in the stage.  (3) Every output word from a per-length table of
//    output-word offsets: a funnel shift (and, for short codewords, a merge at
//    the word's checksum position), lane-strided so stage reads are
//    conflict-free and stores coalesced.  (4) The words that hold a codeword's
//    first 26 data bits or cross into the next codeword, per codeword.  (5) For
//    long codewords, the few words that hold a checksum position.
//  * k_short_small (below): warp tiles of 32 codewords straight from global
//    memory, one codeword per lane.
// The encoder is in hd_short_encode.cu.
#include <algorithm>
#include <array>
#include <cstdint>
#include <mutex>
#include <new>
#include <type_traits>
#include <utility>
#include <vector>

#include "hd_device.cuh"
#include "hd_internal.h"
#include "hd_lane.cuh"

namespace hd {

// It depends on the distance modulo 32 words.
const BankWays &bank_ways(uint32_t bits)
{
    static const std::array<BankWays, 1024> table = [] {
        std::array<BankWays, 1024> t{};
        for (uint32_t m = 0; m < 1024; ++m)
            for (uint32_t lg = 0; lg <= 5; ++lg) {
                uint8_t words[32] = {}, most = 0;
                for (uint32_t l = 0; l < 32; ++l)
                    most = std::max(most, ++words[(((l >> lg) * (1024 + m) >> 5) + (l & ((1u << lg) - 1u))) & 31u]);
                t[m][lg] = most;
            }
        return t;
    }();
    return table[bits % 1024];
}

namespace {

constexpr uint32_t kShortMaxN = 32767;  // r <= 15: syndromes fit 16 bits
constexpr uint32_t kLongMinK = 64;      // k_short_tiles needs the first 58 data bits inside one codeword
// Lengths below kLaneMaxN are decoded one codeword per lane, except large streams from
// kLaneTileN on.  On GB300 with u16 syndromes, lanes against tiles: 1 Gbit of n = 400 55/76 us,
// 544 58/68, 650 63/61, 700 60/66, 768 74/66, 850 67/62, 959 71/60; 256 Mbit of n = 768 24.5/23.5, 850
// 23.0/21.5, 959 24.0/22.7; 32 Mbit of n = 900 5.8/6.6; 20,000 bits of n = 850 3.6/4.8.
constexpr uint32_t kLaneMaxN = 960;
constexpr uint32_t kLaneTileN = 768;
constexpr uint64_t kLaneTileBits = 1ull << 28;

__host__ __device__ inline uint32_t short_r(uint32_t n)
{
    uint32_t r = 0;
    while ((1u << r) < n + 1u) ++r;
    return r;
}

__device__ __forceinline__ uint32_t lowmask(uint32_t b) { return b >= 32 ? 0xFFFFFFFFu : (1u << b) - 1u; }

struct ShortArgs {
    uint32_t *status;
    uint64_t num_cw;
    uint64_t in_words;
    uint64_t bulk_end;  // bytes of the input that 16-byte bulk copies may read
    uint64_t ntiles;
    uint32_t n, k, g;   // code length, data bits, codewords per tile
    uint32_t tlog;      // log2 of the team size of the syndrome pass
    int syn_type;
    bool direct;        // one CTA that overwrites the counters
    uint32_t tab_len;       // entries of the output-word table (see output_table), 2 or 4 bytes each
    uint32_t nJ;            // data runs J >= 5 that end inside the codeword's data (D_J < k)
    uint32_t nJ_magic;      // ceil(2^32 / nJ) for nJ > 1: f / nJ = umulhi(f, nJ_magic) for the small f used
    uint32_t stage;         // bytes of a warp's stage: the longest tile with its 16-byte rounding
};

// A warp's shared memory: a 16-byte guard area (its last word is read as word -1), the
// stage, 16 bytes of slack behind it, and the mbarrier.
constexpr uint32_t kStageExtra = 48;
constexpr uint32_t kMaxStage = 8192;
constexpr int kTileWarps = 24;  // most warps of a CTA
constexpr uint32_t kMaxTileCw = 256;

// Codewords per tile: the tile's input plus 16-byte rounding at both ends fits a stage.
inline uint32_t tile_codewords(uint32_t stage, uint32_t n)
{
    return std::min<uint32_t>((8u * stage - 256u) / n, kMaxTileCw);
}

// The stage of g codewords: their bits behind up to 127 others, in whole 16-byte pieces.
inline uint32_t stage_bytes(uint32_t n, uint32_t g) { return (g * n + 254u) / 128u * 16u; }

// Bytes of tile t that a bulk copy brings in, and where they start.
__device__ __forceinline__ void tile_span(const ShortArgs &a, uint64_t t, uint64_t &byte0, uint32_t &bytes,
                                          uint32_t &gcnt)
{
    const uint64_t c0 = t * a.g;
    gcnt = (uint32_t)min((uint64_t)a.g, a.num_cw - c0);
    const uint64_t bit0 = c0 * a.n, bit1 = (c0 + gcnt) * a.n;
    byte0 = (bit0 >> 7) << 4;
    uint64_t byte1 = ((bit1 + 127) >> 7) << 4;
    if (byte1 > a.bulk_end) byte1 = a.bulk_end;
    bytes = byte1 > byte0 ? (uint32_t)(byte1 - byte0) : 0u;
}

__device__ __forceinline__ void issue_tile(const ShortArgs &a, const uint32_t *in, uint64_t t, uint8_t *stage,
                                           uint64_t *bar)
{
    uint64_t byte0;
    uint32_t bytes, gcnt;
    tile_span(a, t, byte0, bytes, gcnt);
    mbar_arrive_expect_tx(bar, bytes);
    if (bytes) bulk_g2s(stage + 16, reinterpret_cast<const uint8_t *>(in) + byte0, bytes, bar);
}

// The first 32 data bits of the codeword whose position 1 is stage bit cb
// (positions 3, 5-7, 9-15, 17-31, 33-38).
__device__ __forceinline__ uint32_t head_word(const uint32_t *st, uint32_t cb)
{
    const int32_t q = (int32_t)cb - 1;
    const int32_t wi = q >> 5;  // -1 reads the guard word
    const uint32_t sh = (uint32_t)q & 31u;
    const uint32_t y0 = __funnelshift_r(st[wi], st[wi + 1], sh);
    const uint32_t y1 = __funnelshift_r(st[wi + 1], st[wi + 2], sh);
    return ((y0 >> 3) & 1u) | ((y0 >> 4) & 0xEu) | ((y0 >> 5) & 0x7F0u) | ((y0 >> 6) & 0x3FFF800u) |
           ((y1 << 25) & 0xFC000000u);
}

// 32 data bits of the codeword whose position 1 is stage bit cb, from data bit
// d >= 26 on (so at most one checksum position falls inside).
__device__ __forceinline__ uint32_t run_word(const uint32_t *st, uint32_t cb, uint32_t d)
{
    const uint32_t J1 = 31u - __clz(d);
    const uint32_t J = J1 + ((d + J1 + 2u) >> (J1 + 1u));  // data run of bit d
    const uint32_t q = cb + d + J + 1u;
    const uint32_t lo = st[q >> 5], hi = st[(q >> 5) + 1], sh = q & 31u;
    const uint32_t m = lowmask((2u << J) - J - 2u - d);
    return (__funnelshift_r(lo, hi, sh) & m) | (__funnelshift_rc(lo, hi, sh + 1u) & ~m);
}

// End of a decode kernel: the lanes' counts to the counters.  direct: this CTA is
// the whole grid and overwrites them (nothing cleared them); else they are added
// to.  Warp w leaves its counts at base + w * stride (two words of shared memory of
// its own).  Every thread of the CTA calls it.
__device__ __forceinline__ void add_counts(bool direct, unsigned long long *err, unsigned long long *det, uint32_t errs,
                                           uint32_t dets, uint32_t *base, uint32_t stride)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    errs = __reduce_add_sync(0xFFFFFFFFu, errs);
    dets = __reduce_add_sync(0xFFFFFFFFu, dets);
    if (!direct) {
        if (lane == 0) {
            grid_dep_wait();  // the counters' clear ahead of a programmatic dependent launch
            if (err && errs) atomicAdd(err, (unsigned long long)errs);
            if (det && dets) atomicAdd(det, (unsigned long long)dets);
        }
        return;
    }
    if (lane == 0) {
        base[warp * stride] = errs;
        base[warp * stride + 1] = dets;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long e = 0, d = 0;
        for (uint32_t w = 0; w < blockDim.x / 32; ++w) {
            e += base[w * stride];
            d += base[w * stride + 1];
        }
        if (err) *err = e;
        if (det) *det = d;
    }
}

template <bool TAB_SMEM, bool SPLIT>
__global__ void __launch_bounds__(kTileWarps * 32, 1)
    k_short_tiles(const uint32_t *__restrict__ in, uint32_t *__restrict__ out, void *__restrict__ syn,
                  unsigned long long *__restrict__ err, unsigned long long *__restrict__ det,
                  const void *__restrict__ table, const ShortArgs a)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t warp_bytes = a.stage + kStageExtra, W = blockDim.x >> 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the output-word table, copied once per CTA when it fits next to the stages
    // SPLIT: 32-bit entries that also say where a word's checksum position falls, resolved
    // in pass 3; otherwise 16-bit entries and pass 5 rewrites those words
    using Entry = typename std::conditional<SPLIT, uint32_t, uint16_t>::type;
    const Entry *tab = static_cast<const Entry *>(table);
    uint8_t *wbase = smem + warp * warp_bytes;
    uint64_t *bar = reinterpret_cast<uint64_t *>(wbase + a.stage + 32);
    uint32_t *st = reinterpret_cast<uint32_t *>(wbase + 16);
    const uint64_t gw = (uint64_t)blockIdx.x * W + warp, tw = (uint64_t)gridDim.x * W;

    if (lane == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
        if (gw < a.ntiles) issue_tile(a, in, gw, wbase, bar);
    }
    // the output-word table next to the stages where it fits: one bulk copy per CTA, behind the
    // first tiles and waited for before the first output words
    uint64_t *tbar = nullptr;
    if constexpr (TAB_SMEM) {
        uint8_t *s_tab = smem + W * warp_bytes;
        const uint32_t tab_bytes = (a.tab_len * (uint32_t)sizeof(Entry) + 15u) & ~15u;
        tbar = reinterpret_cast<uint64_t *>(s_tab + tab_bytes);
        if (threadIdx.x == 0) {
            mbar_init(tbar, 1);
            fence_mbar_init();
            mbar_arrive_expect_tx(tbar, tab_bytes);
            bulk_g2s(s_tab, table, tab_bytes, tbar);
        }
        __syncthreads();
        tab = reinterpret_cast<const Entry *>(s_tab);
    }
    __syncwarp();

    // syndrome teams: T lanes per codeword, G codewords per round
    const uint32_t tlog = a.tlog, T = 1u << tlog, tl = lane & (T - 1u), team = lane >> tlog, G = 32u >> tlog;
    const uint32_t n = a.n, k = a.k;
    const int32_t stage_bits = 8 * (int32_t)a.stage;  // reads past the data stay inside the stage's slack
    uint32_t errs = 0, dets = 0, it = 0;
    bool aborted = false;
    for (uint64_t t = gw; t < a.ntiles; t += tw, ++it) {
        bool ok = mbar_wait_bounded(bar, it & 1u);
        if (TAB_SMEM && it == 0) ok = ok && mbar_wait_bounded(tbar, 0);
        if (__any_sync(0xFFFFFFFFu, !ok)) {
            aborted = true;
            break;
        }
        uint64_t byte0;
        uint32_t bytes, gcnt;
        tile_span(a, t, byte0, bytes, gcnt);
        if (TAB_SMEM && lane == 0 && t + tw < a.ntiles) {
            // the warp's next tile comes into the one stage when this one is done: into L2 meanwhile
            // (n = 8013, 1 Gbit 45.3 -> 43.1 us; no gain with the table in global memory, 54.1/55.4)
            uint64_t nb;
            uint32_t nbytes, ncw;
            tile_span(a, t + tw, nb, nbytes, ncw);
            if (nbytes) bulk_prefetch_l2(reinterpret_cast<const uint8_t *>(in) + nb, nbytes);
        }
        const uint64_t c0 = t * a.g;
        const uint32_t off0 = (uint32_t)((c0 * n) & 127u);
        {  // words past the last 16-byte boundary of the input arrive by plain loads
            const uint64_t w0 = byte0 >> 2, wb = (byte0 + bytes) >> 2;
            const uint64_t we = min(((c0 + gcnt) * n + 31) >> 5, a.in_words);
            if (wb < we) {
                for (uint64_t w = wb + lane; w < we; w += 32) st[w - w0] = in[w];
                __syncwarp();
            }
        }

        // 1. syndromes.  Lane tl of a team reads stage words r = tl + T*i of its codeword, four
        //    at a time (i = 4q + u), as they lie: bit b of word r is position 32*r + b - sh, so the
        //    word's bits from sh up belong to position-domain word r and those below to r - 1.
        //    x is the XOR of all of the lane's words (rotated by sh at the end: every word's
        //    rotation is the same), A and B the XORs of those with bit 0 and bit 1 of u set, hq
        //    the XOR of the q whose four words have odd parity, so that one popcount serves four
        //    words.  For tl > 0 word r - 1 has the same i, and only the low part of the index
        //    differs; for tl = 0 the bits below sh count for i - 1 (mask lm).  The low syndrome
        //    bits are parities of x, the high ones the XOR of the indices of the odd-parity words.
        //    One load and no shift per word: with two loads and a funnel shift (position-domain
        //    words) 900 Mbit of n = 3212 took 52.2 us, 49.6 so.
        for (uint32_t cbase = 0; cbase < gcnt; cbase += G) {
            const uint32_t c = cbase + team;
            uint32_t x = 0, A = 0, B = 0, hq = 0, lo = 0, lm = 0, sh = 0;
            if (c < gcnt) {
                const int32_t q0 = (int32_t)(off0 + c * n) - 1;  // position 0 is bit -1 of c (the guard word for c = 0)
                sh = (uint32_t)q0 & 31u;
                lo = (1u << sh) - 1u;
                lm = tl == 0 ? lo : 0u;
                const uint32_t rl = (n + sh) >> 5, last = 0xFFFFFFFFu >> (31u - ((n + sh) & 31u));  // last word, its bits
                const uint32_t *ad = st + (q0 >> 5) + (int32_t)tl;
                auto take = [&](uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3, uint32_t v4, uint32_t q) {
                    A ^= v1 ^ v3;
                    B ^= v2 ^ v3;
                    const uint32_t b = v0 ^ v1 ^ v2 ^ v3;
                    x ^= b;
                    hq ^= q & (0u - (__popc(b ^ ((v0 ^ v4) & lm)) & 1u));
                };
                // word r without the bits past position n
                auto end = [&](uint32_t r, const uint32_t *p) { return r < rl ? *p : r == rl ? *p & last : 0u; };
                uint32_t r = tl, q = 0;
                uint32_t v0 = end(r, ad) & ~lm;  // not the bits before the codeword
                // plain shared-memory loads, so that the compiler issues an unrolled
                // iteration's loads ahead of their uses
#pragma unroll 2
                for (; r + 4u * T < rl; r += 4u * T, ++q, ad += 4u * T) {
                    const uint32_t v1 = ad[T], v2 = ad[2u * T], v3 = ad[3u * T], v4 = ad[4u * T];
                    take(v0, v1, v2, v3, v4, q);
                    v0 = v4;
                }
                const uint32_t v1 = end(r + T, ad + T), v2 = end(r + 2u * T, ad + 2u * T);
                const uint32_t v3 = end(r + 3u * T, ad + 3u * T), v4 = end(r + 4u * T, ad + 4u * T);
                take(v0, v1, v2, v3, v4, q);
                take(v4, 0u, 0u, 0u, 0u, q + 1u);
            }
            // the lane's share in one word: the low bits' parities on bits 1, 2, 4, 8, 16 of x's
            // transform, the index bits from 17 up; XOR over the team (butterfly steps stay
            // inside aligned groups of T lanes)
            const uint32_t hi = hq << 2 | (__popc(B ^ ((x ^ A) & lm)) & 1u) << 1 | (__popc(A ^ (x & lm)) & 1u);
            const uint32_t tsum = (0u - (__popc(x & ~lo) & 1u) & tl) ^ (0u - (__popc(x & lo) & 1u) & (tl - 1u) & (T - 1u));
            uint32_t z = (superset_xor<5>(__funnelshift_r(x, x, sh)) & 0x00010116u) | ((hi << tlog) ^ tsum) << 17;
            if (T == 32u)
                z = __reduce_xor_sync(0xFFFFFFFFu, z);
            else
                for (uint32_t o = T >> 1; o > 0; o >>= 1) z ^= __shfl_xor_sync(0xFFFFFFFFu, z, o);
            if (tl == 0 && c < gcnt) {
                const uint32_t sv = (z >> 17) << 5 | ((z >> 1) & 3u) | ((z >> 2) & 4u) | ((z >> 5) & 8u) | ((z >> 12) & 16u);
                if (sv != 0) {
                    ++errs;
                    if (sv <= n) {
                        const uint32_t b = off0 + c * n + sv - 1u;
                        atomicXor(&st[b >> 5], 1u << (b & 31u));
                    } else {
                        ++dets;
                    }
                }
                if (a.syn_type == 1) static_cast<uint8_t *>(syn)[c0 + c] = (uint8_t)sv;
                if (a.syn_type == 2) static_cast<uint16_t *>(syn)[c0 + c] = (uint16_t)sv;
            }
        }
        __syncwarp();

        // 3. output words, lane-strided (conflict-free stage reads, coalesced stores).  The table
        //    describes output word idx of a 32-codeword period (k words): the distance from bit
        //    32*idx to the stage bit of the word's first data bit (counted from position 1 of the
        //    period's first codeword) and how many data bits precede its one checksum position.
        //    Words holding a codeword's head or a crossing are rewritten by pass 4.
        const uint64_t ob0 = c0 * k, ob1 = (c0 + gcnt) * k;
        const uint64_t F = ob0 >> 5, L = (ob1 - 1) >> 5;
        const bool fs = (ob0 & 31u) != 0, last_tile = (c0 + gcnt) == a.num_cw;
        const bool ls = (ob1 & 31u) != 0 && !last_tile;
        const int32_t nW = (int32_t)(L - F) + 1;                       // words of this tile
        const int32_t wlo = fs ? 1 : 0, whi = nW - 1 - (ls ? 1 : 0);  // words it writes whole
        {
            // the table runs past one period, so a tile's words never wrap: word w of the tile is
            // entry idxF + w, whose first data bit is at stage bit sb0 + 32 * (idxF + w) + delta
            const uint32_t cr = (uint32_t)(c0 & 31u);
            const int32_t idx0 = (int32_t)((cr * k) >> 5) + lane;
            int32_t sbw = (int32_t)off0 - (int32_t)(cr * n) + 32 * idx0;
            const Entry *tp = tab + idx0;
            uint32_t *outp = out + F + lane;
            // four words per lane per iteration, 32 apart.  Words past the tile come from
            // in-range entries and clamped stage bits and are never stored.
            for (int32_t w0 = lane; w0 <= whi; w0 += 128, outp += 128, tp += 128, sbw += 4096) {
                uint32_t e[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) e[u] = tp[32 * u];
                if (w0 - lane >= wlo && w0 - lane + 127 <= whi) {
                    // all 128 words of this step are the tile's own (warp-uniform): their first
                    // data bits lie inside the stage, so neither the clamp nor the store test
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int32_t q = sbw + 1024 * u + (int32_t)(e[u] & 0xFFFFu);
                        const uint32_t lo = st[q >> 5], hi = st[(q >> 5) + 1], sh = (uint32_t)q & 31u;
                        uint32_t v = __funnelshift_r(lo, hi, sh);
                        if constexpr (SPLIT) {
                            const uint32_t m = shl_clamp(1u, e[u] >> 16) - 1u;
                            v = (v & m) | (__funnelshift_rc(lo, hi, sh + 1u) & ~m);
                        }
                        outp[32 * u] = v;
                    }
                    continue;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int32_t q = max(0, min(sbw + 1024 * u + (int32_t)(e[u] & 0xFFFFu), stage_bits));
                    const uint32_t lo = st[q >> 5], hi = st[(q >> 5) + 1], sh = (uint32_t)q & 31u;
                    uint32_t v = __funnelshift_r(lo, hi, sh);
                    if constexpr (SPLIT) {
                        const uint32_t m = shl_clamp(1u, e[u] >> 16) - 1u;
                        v = (v & m) | (__funnelshift_rc(lo, hi, sh + 1u) & ~m);
                    }
                    const int32_t w = w0 + 32 * u;
                    if (w >= wlo && w <= whi) outp[32 * u] = v;
                }
            }
        }
        __syncwarp();  // orders pass 3's stores before pass 4 rewrites some of the same words

        // 4. per codeword: the word where its data starts (crossing from the previous codeword,
        //    or the tile's first word), the next word if it still holds head bits, and for the
        //    last codeword the tile's last word.  Word indices are tile-relative.
        for (uint32_t c = lane; c < gcnt; c += 32) {
            const uint32_t b = (uint32_t)(ob0 & 31u) + c * k;  // tile bit of the codeword's data bit 0
            const int32_t ws = (int32_t)(b >> 5);
            const uint32_t al = b & 31u;
            const uint32_t cb = off0 + c * n;  // stage bit of position 1
            const uint32_t head = head_word(st, cb);
            uint32_t *o = out + F + ws;
            if (c == 0 && fs) {
                const uint32_t own = ~lowmask(al), v = head << al;
                atomicAnd(o, v | ~own);
                atomicOr(o, v & own);
            } else if (ws <= whi) {
                *o = al == 0 ? head : (run_word(st, cb - n, k - al) & lowmask(al)) | (head << al);
            }
            if (al > 6 && ws + 1 <= whi) {
                // data bits 32 - al .. 63 - al: the head word's top bits, then data bits 32.. (positions
                // 39..63 of run 5, then run 6 after position 64)
                const uint32_t q = cb + 38u;
                const uint32_t lo = st[q >> 5], hi = st[(q >> 5) + 1], sh = q & 31u;
                const uint32_t x2 = (__funnelshift_r(lo, hi, sh) & 0x1FFFFFFu) |
                                    (__funnelshift_rc(lo, hi, sh + 1u) & ~0x1FFFFFFu);
                o[1] = (head >> (32u - al)) | (x2 << al);
            }
            if (c == gcnt - 1 && (ob1 & 31u) != 0) {
                const uint32_t rem = (uint32_t)(ob1 & 31u);
                const uint32_t v = run_word(st, cb, k - rem) & lowmask(rem);
                uint32_t *ol = out + L;
                if (ls) {
                    atomicAnd(ol, v | ~lowmask(rem));
                    atomicOr(ol, v);
                } else {
                    *ol = v;
                }
            }
        }
        // 5. words with a checksum position inside (data run J ends at data bit D_J = 2^(J+1) - J - 2,
        //    J >= 5): pass 3 read them with one shift; lanes take (codeword, J) pairs
        for (uint32_t f = lane; !SPLIT && f < gcnt * a.nJ; f += 32) {
            const uint32_t c = a.nJ == 1 ? f : __umulhi(f, a.nJ_magic), J = 5u + (f - c * a.nJ);
            const uint32_t b0 = (uint32_t)(ob0 & 31u) + c * k;   // tile bit of the codeword's data bit 0
            const uint32_t bd = b0 + (2u << J) - J - 2u;          // tile bit of data bit D_J
            const uint32_t dw = (bd & ~31u) - b0;                 // data bit at the start of its word (>= 26)
            if ((bd & 31u) != 0 && dw + 32u <= k) out[F + (bd >> 5)] = run_word(st, off0 + c * n, dw);
        }
        // the corrections wrote the stage through the generic proxy; the refill writes it through the async one
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
            const uint64_t tn = t + tw;
            if (tn < a.ntiles) issue_tile(a, in, tn, wbase, bar);
        }
        __syncwarp();
    }
    if (lane == 0 && aborted) {
        atomicOr(a.status, (uint32_t)HD_ERR_TIMEOUT);
        (void)mbar_wait_bounded(bar, it & 1u);  // the copies in flight
        if (TAB_SMEM) (void)mbar_wait_bounded(tbar, 0);
    }
    add_counts(a.direct, err, det, errs, dets, reinterpret_cast<uint32_t *>(smem), warp_bytes / 4);
}

// ---------------------------------------------------------------------------
// Segments of at most WY position-domain words (n < 32 * WY): warp tiles of 32
// codewords, one per lane, straight from global memory.  32 codewords of any
// length n fill exactly n input words and k output words.  The data runs move to
// constant places (positions past n are 0); the lanes OR theirs into the tile's k
// output words in shared memory, which costs neither a division nor a loop over a
// word's pieces.
// Bound: the integer ALU (61 % busy at n = 70, 170 instructions a tile) below n = 150,
// then the L1's wavefronts of the lanes' strided reads.  The per-lane kernel it
// replaces (k < 64 only; bits moved a run at a time through shared memory) took 1296
// us at n = 16 and 427 at n = 70 for 1 Gbit, this one 312 and 109; from n = 71 on see
// kLaneMaxN.
// ---------------------------------------------------------------------------
constexpr int kSmallWarps = 8;

template <int WY>
__global__ void __launch_bounds__(kSmallWarps * 32)
    k_short_small(const uint32_t *__restrict__ in, uint64_t in_words, uint32_t n, uint32_t r, uint64_t num_cw,
                  uint32_t *__restrict__ out, uint64_t out_words, void *__restrict__ syn, int syn_type,
                  unsigned long long *__restrict__ err, unsigned long long *__restrict__ det, bool direct)
{
    constexpr uint32_t kMerged = 32u * WY + WY + 1u;  // k words, and spill words for the last lane
    __shared__ uint32_t merged[kSmallWarps][kMerged];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    uint32_t *m = merged[wp];
    const uint32_t k = n - r;
    const uint64_t tiles = (num_cw + 31) / 32;
    // position p of the lane's codeword is tile bit lane * n + p - 1
    const int32_t bit = lane * (int32_t)n - 1, a0 = bit >> 5;
    const uint32_t sh = (uint32_t)bit & 31u;
    const uint32_t ob = (uint32_t)lane * k, os = ob & 31u, oe = (os + k + 31u) >> 5;  // the data bits' place in the tile
    uint32_t *mine = m + (ob >> 5);
    uint32_t mask[WY];  // valid positions (bit 0 of the first word is none)
#pragma unroll
    for (uint32_t w = 0; w < WY; ++w) mask[w] = n >= 32u * w ? lowmask(n + 1u - 32u * w) : 0u;
    mask[0] &= ~1u;
    uint32_t errs = 0, dets = 0;
    for (uint64_t t = (uint64_t)blockIdx.x * kSmallWarps + wp; t < tiles; t += (uint64_t)gridDim.x * kSmallWarps) {
        const uint64_t i = t * 32 + lane;
        const bool valid = i < num_cw;
        const uint32_t *src = in + t * n;
        const uint32_t have = (uint32_t)min((uint64_t)n, in_words - t * n);  // words of the tile
        uint32_t raw[WY + 1], y[WY];
#pragma unroll
        for (int w = 0; w <= WY; ++w) raw[w] = valid && (uint32_t)(a0 + w) < have ? src[a0 + w] : 0u;
#pragma unroll
        for (uint32_t w = 0; w <= WY; ++w)
            if (32u * w + lane < kMerged) m[32u * w + lane] = 0u;
        uint32_t x = 0, s = 0;
#pragma unroll
        for (int w = 0; w < WY; ++w) {
            y[w] = __funnelshift_r(raw[w], raw[w + 1], sh) & mask[w];
            x ^= y[w];
        }
#pragma unroll
        for (int b = 0; (1 << b) < WY; ++b) {
            uint32_t g = 0;
#pragma unroll
            for (int w = 0; w < WY; ++w)
                if ((w >> b) & 1) g ^= y[w];
            s |= (__popc(g) & 1u) << (5 + b);
        }
        const uint32_t z = superset_xor<5>(x);
        s |= ((z >> 1) & 3u) | ((z >> 2) & 4u) | ((z >> 5) & 8u) | ((z >> 12) & 16u);
        const uint32_t fix = s <= n ? s : 0u;  // a syndrome past n names no position; bit 0 is dropped again
#pragma unroll
        for (int w = 0; w < WY; ++w) y[w] ^= shl_clamp(1u, fix - 32u * (uint32_t)w);
        // the data bits, packed: 26 of the first word, then 31 or 32 a word
        uint32_t d[WY + 1];
        d[0] = compress_runs<5>(y[0] & ~1u);
#pragma unroll
        for (int w = 1; w <= WY; ++w) d[w] = 0u;
        int at = 26;
#pragma unroll
        for (int w = 1; w < WY; ++w) {
            const bool chk = (w & (w - 1)) == 0;  // position 32w is a checksum position
            const uint32_t v = chk ? y[w] >> 1 : y[w];
            d[at / 32] |= v << (at % 32);
            if (at % 32 != 0) d[at / 32 + 1] |= v >> (32 - at % 32);
            at += chk ? 31 : 32;
        }
        __syncwarp();  // the tile's words are cleared
        if (valid) {
            uint32_t lo = 0;
#pragma unroll
            for (uint32_t w = 0; w <= WY; ++w) {
                if (w < oe) atomicOr(&mine[w], __funnelshift_l(lo, d[w], os));
                lo = d[w];
            }
            if (syn_type == 1) static_cast<uint8_t *>(syn)[i] = (uint8_t)s;
            if (syn_type == 2) static_cast<uint16_t *>(syn)[i] = (uint16_t)s;
        }
        errs += __popc(__ballot_sync(0xFFFFFFFFu, valid && s != 0));
        dets += __popc(__ballot_sync(0xFFFFFFFFu, valid && s > n));
        __syncwarp();
        uint32_t *o = out + t * k;
        const uint32_t words = (uint32_t)min((uint64_t)k, out_words - t * k);
#pragma unroll
        for (uint32_t w = 0; w < WY; ++w)
            if (32u * w + lane < words) o[32u * w + lane] = m[32u * w + lane];
        __syncwarp();  // the next tile clears the words
    }
    add_counts(direct, err, det, lane == 0 ? errs : 0u, lane == 0 ? dets : 0u, merged[0], kMerged);
}

// ---------------------------------------------------------------------------
// Variant table of the tile kernel (compiled configurations).
// ---------------------------------------------------------------------------
struct ShortVariant {
    uint32_t warps, stage;  // per CTA (fewer where shared memory does not hold them); bytes of a warp's stage
};

// [0]: the built-in choice.  One CTA of 24 warps shares one output-word table; where that stays in
// global memory (n > about 18,500) two CTAs of 16 warps (n = 24,000, 900 Mbit: 54.5 us with 24
// warps in one CTA, 49.4 with 16 in two).
// A warp's tile costs the same few chains (wait, transform, butterfly, heads) whatever its
// size, so one 8 KB stage beats two of 4 KB: 900 Mbit of n = 3212 in 52.2 us with two, n = 8013
// in 55.9, n = 12,000 in 68.6, against 43.6, 44.5 and 51.1 with one.
const ShortVariant kShortVariants[] = {{0, 0}, {24, 8192}, {24, 6144}, {16, 6144}, {16, 4096}, {12, 4096}, {8, 8192}};
const ShortVariant kSharedTable = {24, 8192}, kGlobalTable = {16, 7168};
constexpr int kNumShortVariants = sizeof(kShortVariants) / sizeof(kShortVariants[0]);
constexpr int kLanes = kNumShortVariants;  // the configuration behind them: one codeword per lane, n < kLaneMaxN

using TileKernel = void (*)(const uint32_t *, uint32_t *, void *, unsigned long long *, unsigned long long *,
                            const void *, ShortArgs);
// [0]: table in global memory; [1]: table in shared memory; [2]: shared, splits in pass 3
const TileKernel kTileKernels[3] = {k_short_tiles<false, false>, k_short_tiles<true, false>, k_short_tiles<true, true>};

constexpr uint32_t kSmemPerCta = 227u << 10;
constexpr uint32_t kTabSmemMax = 40u << 10;  // larger tables stay in global memory

std::mutex g_short_mu;
int g_short_choice[64] = {};  // variant pinned for every length on a device (index + 1; 0 = none)
struct TunedEntry {
    uint32_t n = 0;
    int v = -1;
};
TunedEntry g_short_tuned[64][64];  // per device: the autotuner's choice per length

struct OccEntry {
    int tsm = -1;
    uint32_t warps = 0, smem = 0;
    int bps = 0;
};
OccEntry g_occ[64][32];

// Resident CTAs per SM of tile kernel tsm with `warps` warps and `smem` bytes of dynamic shared memory.
int short_blocks_per_sm(int tsm, uint32_t warps, uint32_t smem)
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    std::lock_guard<std::mutex> lk(g_short_mu);
    for (const OccEntry &e : g_occ[dev])
        if (e.tsm == tsm && e.warps == warps && e.smem == smem) return e.bps;
    const void *kern = reinterpret_cast<const void *>(kTileKernels[tsm]);
    // the attribute is per kernel: allow the device's largest opt-in size once, never a smaller one
    int optin = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        (uint32_t)optin < smem ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin) != cudaSuccess)
        return -1;
    int bps = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, (int)warps * 32, smem) != cudaSuccess || bps <= 0)
        return -1;
    for (OccEntry &e : g_occ[dev])
        if (e.tsm < 0) {
            e = OccEntry{tsm, warps, smem, bps};
            break;
        }
    return bps;
}

// The configuration chosen for length n: a pinned one, else the autotuner's, else -1.
int chosen_short_variant(uint32_t n)
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    std::lock_guard<std::mutex> lk(g_short_mu);
    if (g_short_choice[dev] > 0) return g_short_choice[dev] - 1;
    for (const TunedEntry &e : g_short_tuned[dev])
        if (e.n == n && e.v >= 0) return e.v;
    return -1;
}

void remember_short_variant(uint32_t n, int v)
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    std::lock_guard<std::mutex> lk(g_short_mu);
    TunedEntry *slot = nullptr;
    for (TunedEntry &e : g_short_tuned[dev]) {
        if (e.n == n) {
            slot = &e;
            break;
        }
        if (!slot && e.v < 0) slot = &e;
    }
    if (!slot) slot = &g_short_tuned[dev][n % 64];  // table full: overwrite one entry
    slot->n = n;
    slot->v = v;
}

// Syndrome pass of a tile of g codewords: a team of T = 2^lg lanes reads a codeword's Y
// words, ceil(Y / 4T) blocks of four per lane, and the tile's codewords take
// ceil(g / (32 / T)) rounds, each of which ends in a chain of dependent steps (the
// transform, the butterfly over the team, the correction).  The weights follow the times
// of every T at 18 lengths on GB300 (1 Gbit, T = 1 .. 16: n = 1078 65/73/87/107/146 us,
// n = 3212 71/59/64/67/76, n = 8013 128/91/73/66/75); the least cost is the fastest at all
// of them.
// A block's loads cost more than its arithmetic where the warp's 32 words share few banks
// (codewords a multiple of 32 words apart): weight 10 per word of the fullest bank, fitted
// to every T at 25 lengths, four of them so (1 Gbit of n = 1024: 171 us without the term, 89 with
// it, 2047 134 / 73, 4095 99 / 58; lengths whose fullest bank has up to four words keep their T).
uint64_t team_cost(uint32_t n, uint32_t g, uint32_t *tlog)
{
    const uint32_t Y = (n + 32) / 32;
    const BankWays &ways = bank_ways(n);
    uint64_t best = ~0ull;
    for (uint32_t lg = 0; lg <= 5; ++lg) {
        const uint32_t rounds = (g + (32u >> lg) - 1) >> (5 - lg), blocks = (Y + (4u << lg) - 1) >> (lg + 2);
        const uint64_t cost = (uint64_t)rounds * (blocks * std::max(40u, 10u * ways[lg]) + 160 + 20 * lg);
        if (cost < best) {
            best = cost;
            *tlog = lg;
        }
    }
    return best;
}

// How a stream is cut: codewords per tile (at most gmax), the team size for them, and the
// warps per CTA (W, at most the configuration's; lowered in steps of two to w_min).  All
// warps work through their tiles in step, so the last of the R rounds of tiles should be as
// full as the others, g = ceil(num_cw / (R * warps)), and the g codewords should fill the
// lanes of the syndrome teams (n = 3212: g = 20 takes two rounds of T = 2, g = 16 one).
// The cost is R times a tile's, which grows with the warps that share the SM (0.2 + 0.8 W /
// 24, fitted).  On GB300 at nine lengths of 961 .. 3212 and four sizes of 0.2 .. 0.5 Gbit the
// pick is 5 % faster on average than 24 warps in the smallest R (n = 1100, 244,032
// codewords: 24.9 -> 21.6 us; n = 1611, 124,146: 16.7 -> 14.2; at worst 1.8 % slower), and
// the fastest choice of W and R 5.7 %.  A stream of one codeword per warp or less spreads over
// the whole GPU.
struct TileShape {
    uint32_t g, tlog, warps;
};

TileShape tile_shape(uint32_t n, uint32_t gmax, uint64_t num_cw, uint64_t ctas, uint32_t w_max, uint32_t w_min)
{
    TileShape pick{1, 0, w_max};
    if (num_cw <= ctas * w_max) {
        team_cost(n, 1, &pick.tlog);
        return pick;
    }
    uint64_t best = ~0ull;
    for (int w = (int)w_max; w >= (int)w_min; w -= 2) {
        const uint64_t warps = ctas * (uint32_t)w, r0 = (num_cw + gmax * warps - 1) / (gmax * warps);
        for (uint64_t R = r0; R < r0 + 3; ++R) {
            const uint32_t g = (uint32_t)((num_cw + R * warps - 1) / (R * warps));
            uint32_t lg = 0;
            const uint64_t cost = R * (team_cost(n, g, &lg) + 100) * (uint32_t)(w + 6);
            if (cost < best) {
                best = cost;
                pick = TileShape{g, lg, (uint32_t)w};
            }
        }
    }
    return pick;
}

// Output-word offsets: entry idx describes output word idx of a run of
// codewords that starts at a multiple of 32 (32 codewords fill k words, so a
// tile's first word is entry (c0 mod 32) * k / 32).  The table covers one
// period of k words plus the longest tile and a lane's last group of reads,
// so no tile wraps.  Entry = delta: the word's first data bit is at bit
// 32*idx + delta counted from position 1 of the run's first codeword
// (delta = c*r + J + 1 for data bit d of codeword c in data run J).  Words
// holding a codeword's first 26 data bits, crossing into the next codeword or
// holding a checksum position are rewritten by the kernel's per-codeword
// passes; the first two kinds only point inside their codeword.
std::vector<uint32_t> output_table(uint32_t n, uint32_t k, uint32_t max_tile_words)
{
    const uint32_t r = n - k;
    const uint32_t len = k + max_tile_words + 128;
    std::vector<uint32_t> t(len, 0);
    for (uint32_t idx = 0; idx < len; ++idx) {
        const uint64_t e = 32ull * idx;
        const uint32_t c = (uint32_t)(e / k), d = (uint32_t)(e % k);
        uint32_t delta = c * r + 1u, split = 32;
        if (d >= 26 && k - d >= 32) {
            uint32_t J = 5;
            while (d >= (2u << J) - J - 2u) ++J;  // data run J holds data bits 2^J - J - 1 .. 2^(J+1) - J - 3
            delta = c * r + J + 1u;
            split = std::min<uint32_t>(32u, (2u << J) - J - 2u - d);
        }
        t[idx] = delta | (split << 16);
    }
    return t;
}

// Where the words holding a checksum position are resolved: per word in the
// output pass (32-bit entries) when k is small, so that codewords have few
// words and such words are common; else in a per-codeword pass (16-bit
// entries, half the table).
bool split_in_pass3(uint32_t k) { return k < 1280; }

// Build the output-word table of length n on the current device: cudaMalloc
// and a synchronous copy (the only allocation of the shortened-code path).
cudaError_t build_short_table(uint32_t n, uint32_t k, void **dev, uint32_t *len)
{
    // the longest tile of any configuration: the largest stage's codewords, plus a partial word
    const uint32_t max_words = (uint32_t)(((uint64_t)tile_codewords(kMaxStage, n) * k + 31) / 32) + 1;
    std::vector<uint32_t> full = output_table(n, k, max_words);
    full.resize((full.size() + 7) / 8 * 8, 0);  // whole 16-byte pieces for the kernels' bulk copy
    const bool wide = split_in_pass3(k);
    std::vector<uint16_t> narrow;
    if (!wide)
        for (uint32_t e : full) narrow.push_back((uint16_t)(e & 0xFFFFu));
    const size_t bytes = wide ? full.size() * 4 : narrow.size() * 2;
    const void *src = wide ? static_cast<const void *>(full.data()) : static_cast<const void *>(narrow.data());
    void *d = nullptr;
    cudaError_t e = cudaMalloc(&d, bytes);
    if (e != cudaSuccess) return e;
    e = cudaMemcpy(d, src, bytes, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(d);
        return e;
    }
    *dev = d;
    *len = (uint32_t)full.size();
    return cudaSuccess;
}

// The tables that hd_decode_short builds on first use of a length, per
// device, least recently used first out.  Each table's last use is an event on
// the stream that used it, so evicting a table waits for that use only; a
// table used while its stream was capturing may be read by any later replay
// of that graph and is never evicted.
struct TableEntry {
    uint32_t n = 0;
    void *dev = nullptr;
    uint32_t len = 0;
    uint64_t used = 0;
    cudaEvent_t last = nullptr;  // recorded after each uncaptured use
    bool pinned = false;         // used inside a stream capture
};
constexpr int kMaxTables = 32;
TableEntry g_tables[64][kMaxTables];
uint64_t g_table_clock = 0;

// The cached table of length n for a launch on `st` (built on a miss, which a
// capturing stream may not do: cudaErrorStreamCaptureUnsupported).
cudaError_t table_for(uint32_t n, uint32_t k, cudaStream_t st, TableEntry **entry)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const bool capturing = stream_capturing(st);
    std::lock_guard<std::mutex> lk(g_short_mu);
    TableEntry *slot = nullptr;
    for (TableEntry &e : g_tables[dev]) {
        if (e.n == n && e.dev) {
            e.used = ++g_table_clock;
            *entry = &e;
            return cudaSuccess;
        }
        if (e.pinned) continue;
        if (!slot || (!e.dev && slot->dev) || (e.dev && slot->dev && e.used < slot->used)) slot = &e;
    }
    if (capturing) return cudaErrorStreamCaptureUnsupported;
    if (!slot) return cudaErrorMemoryAllocation;  // every slot is held by a captured graph
    if (slot->dev) {  // evict once its last use has finished
        if (slot->last && cudaEventSynchronize(slot->last) != cudaSuccess) return cudaErrorUnknown;
        cudaFree(slot->dev);
        slot->dev = nullptr;
        slot->n = 0;
    }
    void *d = nullptr;
    uint32_t len = 0;
    cudaError_t e = build_short_table(n, k, &d, &len);
    if (e != cudaSuccess) return e;
    if (!slot->last && cudaEventCreateWithFlags(&slot->last, cudaEventDisableTiming) != cudaSuccess) {
        cudaFree(d);
        return cudaErrorUnknown;
    }
    slot->n = n;
    slot->dev = d;
    slot->len = len;
    slot->used = ++g_table_clock;
    *entry = slot;
    return cudaSuccess;
}

// Mark a cached table's use by a launch just enqueued on `st`.
void table_used(TableEntry *e, cudaStream_t st)
{
    std::lock_guard<std::mutex> lk(g_short_mu);
    if (stream_capturing(st)) e->pinned = true;
    else cudaEventRecord(e->last, st);
}

// Launch a decode whose counts start from zero: a grid of one CTA overwrites the
// counters (*direct), any other is the programmatic dependent of their clear.
// bare: the decode alone, added to counters nobody cleared (timing).
template <class Launch>
cudaError_t launch_counted(bool &direct, unsigned long long *err, unsigned long long *det, int grid, bool bare,
                           cudaStream_t st, Launch launch)
{
    direct = grid == 1 && !bare;
    const bool clear = (err || det) && !direct && !bare;
    if (clear) {
        const cudaError_t e = launch_zero_counts(err, det, st);
        if (e != cudaSuccess) return e;
    }
    return launch(clear);
}

cudaError_t launch_short_tiles(int vi, const uint32_t *in, uint32_t n, uint64_t num_cw, uint32_t *out, void *syn,
                               int syn_type, unsigned long long *err, unsigned long long *det, cudaStream_t st,
                               const void *table, uint32_t tab_len, bool bare)
{
    const uint32_t r = short_r(n), k = n - r;
    ShortArgs a{};
    a.status = status_ptr();
    if (!a.status) return cudaErrorUnknown;
    if (!table) return cudaErrorInvalidValue;
    a.num_cw = num_cw;
    a.in_words = words_for_bits(num_cw * n);
    a.bulk_end = (a.in_words * 4) >> 4 << 4;
    a.n = n;
    a.k = k;
    a.tab_len = tab_len;
    a.syn_type = syn ? syn_type : 0;
    a.nJ = 0;
    for (uint32_t J = 5; (2u << J) - J - 2u < k; ++J) ++a.nJ;
    a.nJ_magic = a.nJ > 1 ? (uint32_t)((0x100000000ull + a.nJ - 1) / a.nJ) : 0u;
    const bool split = split_in_pass3(k);
    const uint32_t tab_bytes = (a.tab_len * (split ? 4u : 2u) + 15) & ~15u;
    const int tsm = split ? 2 : (tab_bytes <= kTabSmemMax ? 1 : 0);  // split tables are small
    if (split) a.nJ = 0;  // no per-codeword pass for checksum words
    const uint32_t tab_smem = tsm ? tab_bytes + 16u : 0u;  // with its mbarrier
    const ShortVariant v = vi > 0 ? kShortVariants[vi] : tsm ? kSharedTable : kGlobalTable;
    const uint32_t gmax = tile_codewords(v.stage, n);
    if (gmax == 0) return cudaErrorInvalidValue;  // the caller picks a configuration whose stage holds a codeword
    a.stage = stage_bytes(n, gmax);
    const uint32_t w_max = std::min(v.warps, (kSmemPerCta - tab_smem) / (a.stage + kStageExtra));
    const int bps = short_blocks_per_sm(tsm, w_max, w_max * (a.stage + kStageExtra) + tab_smem);
    if (bps <= 0) return cudaErrorInvalidConfiguration;
    const uint64_t cap = (uint64_t)num_sms() * (uint64_t)bps;
    // the built-in choice for shared tables varies the warps, a pinned configuration does not
    const TileShape shape = tile_shape(n, gmax, num_cw, cap, w_max, vi > 0 || !tsm ? w_max : std::min(w_max, 14u));
    uint32_t W = shape.warps;
    a.g = shape.g;
    a.tlog = shape.tlog;
    a.ntiles = (num_cw + a.g - 1) / a.g;
    a.stage = stage_bytes(n, a.g);
    // at most one tile per warp: the warps spread over all SMs, or stay in one CTA (direct counts)
    if (a.ntiles > W) W = (uint32_t)std::min<uint64_t>(W, (a.ntiles + cap - 1) / cap);
    const uint32_t smem = W * (a.stage + kStageExtra) + tab_smem;
    const int grid = decode_grid((a.ntiles + W - 1) / W, cap);
    return launch_counted(a.direct, err, det, grid, bare, st, [&](bool pdl) {
        return launch_kernel(kTileKernels[tsm], dim3((unsigned)grid), dim3(W * 32), smem, st, pdl, in, out, syn, err,
                             det, table, a);
    });
}

// One codeword per lane: n < kLaneMaxN.  The kernel of the first word count that
// holds n (even counts above 16).
template <size_t... I>
void (*lane_kernel(uint32_t words, std::index_sequence<I...>))(const uint32_t *, uint64_t, uint32_t, uint32_t, uint64_t,
                                                               uint32_t *, uint64_t, void *, int, unsigned long long *,
                                                               unsigned long long *, bool)
{
    static const decltype(&k_short_small<1>) kernels[] = {&k_short_small<(int)(I < 16 ? I + 1 : (I + 2) / 2 * 2)>...};
    return kernels[words - 1];
}

cudaError_t launch_short_lanes(const uint32_t *in, uint32_t n, uint64_t num_cw, uint32_t *out, void *syn, int syn_type,
                               unsigned long long *err, unsigned long long *det, cudaStream_t st, bool bare)
{
    const uint32_t r = short_r(n);
    const auto kern = lane_kernel(n / 32 + 1, std::make_index_sequence<kLaneMaxN / 32>());
    const uint64_t tiles = (num_cw + 31) / 32;
    const int bps = stream_blocks_per_sm(reinterpret_cast<const void *>(kern), kSmallWarps * 32, 0);
    if (bps <= 0) return cudaErrorInvalidConfiguration;
    const int grid = decode_grid((tiles + kSmallWarps - 1) / kSmallWarps, (uint64_t)num_sms() * (uint64_t)bps);
    bool direct = false;
    return launch_counted(direct, err, det, grid, bare, st, [&](bool pdl) {
        return launch_kernel(kern, dim3((unsigned)grid), dim3(kSmallWarps * 32), 0, st, pdl, in,
                             words_for_bits(num_cw * n), n, r, num_cw, out, words_for_bits(num_cw * (n - r)), syn,
                             syn_type, err, det, direct);
    });
}

}  // namespace
}  // namespace hd

using namespace hd;

namespace {
bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
}  // namespace

extern "C" {

hd_status hd_short_params(uint32_t n, uint32_t *r, uint32_t *k)
{
    if (n < 3 || n > kShortMaxN) return HD_ERR_INVALID_N;
    const uint32_t rr = short_r(n);
    if (r) *r = rr;
    if (k) *k = n - rr;
    return HD_OK;
}

hd_status hd_segment_params(uint32_t packet_bytes, uint32_t t, uint32_t *n, uint32_t *k, uint32_t *r)
{
    if (packet_bytes == 0 || t == 0 || t > 8u * packet_bytes) return HD_ERR_INVALID_ARG;
    const uint64_t kk = (8ull * packet_bytes + t - 1) / t;  // data bits per segment
    uint32_t rr = 0;
    while ((1ull << rr) < kk + rr + 1) ++rr;
    const uint64_t nn = kk + rr;
    if (nn < 3 || nn > kShortMaxN) return HD_ERR_SIZE;
    if (n) *n = (uint32_t)nn;
    if (k) *k = (uint32_t)kk;
    if (r) *r = rr;
    return HD_OK;
}

}  // extern "C"

namespace {

hd_status check_short_args(const uint32_t *stream, uint64_t in_bits, uint32_t n, uint64_t num_codewords,
                           uint32_t *out_bits, void *syndromes, hd_syn_type syn_type)
{
    if (n < 3 || n > kShortMaxN) return HD_ERR_INVALID_N;
    if (syn_type != HD_SYN_NONE && syn_type != HD_SYN_U8 && syn_type != HD_SYN_U16) return HD_ERR_INVALID_ARG;
    if (syn_type == HD_SYN_U8 && n > 255) return HD_ERR_INVALID_ARG;
    if (num_codewords > (1ull << 40)) return HD_ERR_SIZE;
    if (in_bits != (uint64_t)n * num_codewords) return HD_ERR_SIZE;
    if (num_codewords != 0) {
        if (!stream || !out_bits) return HD_ERR_NULL;
        if (syn_type != HD_SYN_NONE && !syndromes) return HD_ERR_NULL;
        if (!aligned16(stream) || !aligned16(out_bits) || (syndromes && !aligned16(syndromes))) return HD_ERR_ALIGN;
    }
    return HD_OK;
}

// The decode itself, the counters' clear included, given the output-word table
// of n (unused for k < 64).
hd_status decode_short_with(const uint32_t *stream, uint64_t in_bits, uint32_t n, uint64_t num_codewords,
                            uint32_t *out_bits, void *syndromes, hd_syn_type syn_type,
                            unsigned long long *err_count, unsigned long long *detected_count, cudaStream_t st,
                            const void *table, uint32_t tab_len)
{
    if (num_codewords == 0) {
        if (!err_count && !detected_count) return HD_OK;
        return launch_zero_counts(err_count, detected_count, st) == cudaSuccess ? HD_OK : HD_ERR_CUDA;
    }
    const uint32_t r = short_r(n), k = n - r;
    const int syn = syndromes ? (int)syn_type : 0;
    // the tiled kernel from kLaneMaxN on, and below it (k >= 64) where a configuration is
    // pinned or the autotuner found one faster
    int vi = k >= kLongMinK ? chosen_short_variant(n) : -1;
    if (vi == kLanes && n >= kLaneMaxN) vi = 0;
    if (vi == kLanes || (vi < 0 && n < kLaneMaxN && (n < kLaneTileN || num_codewords * n < kLaneTileBits)))
        return launch_short_lanes(stream, n, num_codewords, out_bits, syndromes, syn, err_count, detected_count, st,
                                  false) == cudaSuccess
                   ? HD_OK
                   : HD_ERR_CUDA;
    if (vi < 0) vi = 0;  // the built-in configuration
    if (vi > 0 && kShortVariants[vi].stage * 8u < n + 256u) vi = 0;  // stage too small for a codeword
    return launch_short_tiles(vi, stream, n, num_codewords, out_bits, syndromes, syn, err_count, detected_count, st,
                              table, tab_len, false) == cudaSuccess
               ? HD_OK
               : HD_ERR_CUDA;
}

}  // namespace

struct hd_short_plan {
    int device = 0;
    uint32_t n = 0;
    void *table = nullptr;  // output-word table (k >= 64), owned by the plan
    uint32_t tab_len = 0;
};

extern "C" {

hd_status hd_decode_short(const uint32_t *stream, uint64_t in_bits, uint32_t n, uint64_t num_codewords,
                          uint32_t *out_bits, void *syndromes, hd_syn_type syn_type, unsigned long long *err_count,
                          unsigned long long *detected_count, void *cuda_stream)
{
    hd_status rc = check_short_args(stream, in_bits, n, num_codewords, out_bits, syndromes, syn_type);
    if (rc != HD_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const uint32_t k = n - short_r(n);
    TableEntry *e = nullptr;
    if (num_codewords != 0 && k >= kLongMinK) {
        const cudaError_t te = table_for(n, k, st, &e);
        if (te == cudaErrorStreamCaptureUnsupported) return HD_ERR_INVALID_ARG;  // build it outside the capture
        if (te != cudaSuccess) return HD_ERR_CUDA;
    }
    rc = decode_short_with(stream, in_bits, n, num_codewords, out_bits, syndromes, syn_type, err_count,
                           detected_count, st, e ? e->dev : nullptr, e ? e->len : 0);
    if (e && rc == HD_OK) table_used(e, st);
    return rc;
}

hd_status hd_short_plan_create(uint32_t n, hd_short_plan **plan)
{
    if (!plan) return HD_ERR_NULL;
    *plan = nullptr;
    if (n < 3 || n > kShortMaxN) return HD_ERR_INVALID_N;
    hd_short_plan *p = new (std::nothrow) hd_short_plan();
    if (!p) return HD_ERR_CAPACITY;
    p->n = n;
    if (cudaGetDevice(&p->device) != cudaSuccess) {
        delete p;
        return HD_ERR_CUDA;
    }
    const uint32_t k = n - short_r(n);
    if (k >= kLongMinK && build_short_table(n, k, &p->table, &p->tab_len) != cudaSuccess) {
        delete p;
        return HD_ERR_CUDA;
    }
    *plan = p;
    return HD_OK;
}

hd_status hd_decode_short_plan(const hd_short_plan *plan, const uint32_t *stream, uint64_t in_bits,
                               uint64_t num_codewords, uint32_t *out_bits, void *syndromes, hd_syn_type syn_type,
                               unsigned long long *err_count, unsigned long long *detected_count, void *cuda_stream)
{
    if (!plan) return HD_ERR_NULL;
    hd_status rc = check_short_args(stream, in_bits, plan->n, num_codewords, out_bits, syndromes, syn_type);
    if (rc != HD_OK) return rc;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return HD_ERR_CUDA;
    if (dev != plan->device) return HD_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    return decode_short_with(stream, in_bits, plan->n, num_codewords, out_bits, syndromes, syn_type, err_count,
                             detected_count, st, plan->table, plan->tab_len);
}

void hd_short_plan_destroy(hd_short_plan *plan)
{
    if (!plan) return;
    if (plan->table) {
        int cur = 0;
        cudaGetDevice(&cur);
        if (cur != plan->device) cudaSetDevice(plan->device);
        cudaFree(plan->table);  // waits for the work that may still read it
        if (cur != plan->device) cudaSetDevice(cur);
    }
    delete plan;
}

hd_status hd_encode_short(const uint32_t *data_bits, uint32_t n, uint64_t num_codewords, uint32_t *stream,
                          void *cuda_stream)
{
    if (n < 3 || n > kShortMaxN) return HD_ERR_INVALID_N;
    if (num_codewords > (1ull << 40)) return HD_ERR_SIZE;
    if (num_codewords == 0) return HD_OK;
    if (!data_bits || !stream) return HD_ERR_NULL;
    if (!aligned16(data_bits) || !aligned16(stream)) return HD_ERR_ALIGN;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const uint32_t r = short_r(n), k = n - r;
    return launch_encode_short(data_bits, n, k, num_codewords, stream, st) == cudaSuccess ? HD_OK : HD_ERR_CUDA;
}

hd_status hd_short_autotune(uint32_t n, uint64_t num_codewords, uint32_t reps, void *cuda_stream, int32_t *chosen)
{
    if (n < 3 || n > kShortMaxN) return HD_ERR_INVALID_N;
    const uint32_t r = short_r(n), k = n - r;
    if (num_codewords == 0 || num_codewords > (1ull << 32)) return HD_ERR_SIZE;
    if (reps == 0) reps = 5;
    if (k < kLongMinK) {  // one kernel only
        if (chosen) *chosen = -1;
        return HD_OK;
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const size_t in_b = words_for_bits(num_codewords * n) * 4 + 16, out_b = words_for_bits(num_codewords * k) * 4 + 16;
    void *din = nullptr, *dout = nullptr, *dsyn = nullptr, *dcnt = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    hd_status rc = HD_OK;
    int best = -1;
    float best_ms = 0.f;
    if (cudaMalloc(&din, in_b) != cudaSuccess || cudaMalloc(&dout, out_b) != cudaSuccess ||
        cudaMalloc(&dsyn, num_codewords * 2 + 16) != cudaSuccess || cudaMalloc(&dcnt, 16) != cudaSuccess ||
        cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
        rc = HD_ERR_CUDA;
    // all-zero segments are codewords: the timing sees the common no-error path
    if (rc == HD_OK && cudaMemsetAsync(din, 0, in_b, st) != cudaSuccess) rc = HD_ERR_CUDA;
    auto *cnt = static_cast<unsigned long long *>(dcnt);
    TableEntry *tab = nullptr;
    if (rc == HD_OK && table_for(n, k, st, &tab) != cudaSuccess) rc = HD_ERR_CUDA;
    for (int v = 0; rc == HD_OK && v < kNumShortVariants; ++v) {
        if (v > 0 && kShortVariants[v].stage * 8u < n + 256u) continue;
        auto go = [&]() {
            return launch_short_tiles(v, static_cast<const uint32_t *>(din), n, num_codewords,
                                      static_cast<uint32_t *>(dout), dsyn, HD_SYN_U16, cnt, cnt + 1, st, tab->dev,
                                      tab->len, true);
        };
        if (go() != cudaSuccess) {  // warm-up (also configures the kernel)
            rc = HD_ERR_CUDA;
            break;
        }
        cudaEventRecord(e0, st);
        for (uint32_t i = 0; i < reps; ++i) go();
        cudaEventRecord(e1, st);
        float ms = 0.f;
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
            rc = HD_ERR_CUDA;
            break;
        }
        if (best < 0 || ms < best_ms) {
            best = v;
            best_ms = ms;
        }
    }
    // below kLaneMaxN a tile configuration is kept only if it beats one codeword per lane
    if (rc == HD_OK && best >= 0 && n < kLaneMaxN) {
        auto go = [&]() {
            return launch_short_lanes(static_cast<const uint32_t *>(din), n, num_codewords, static_cast<uint32_t *>(dout),
                                      dsyn, HD_SYN_U16, cnt, cnt + 1, st, true);
        };
        float ms = 0.f;
        if (go() != cudaSuccess) rc = HD_ERR_CUDA;
        cudaEventRecord(e0, st);
        for (uint32_t i = 0; rc == HD_OK && i < reps; ++i) go();
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) rc = HD_ERR_CUDA;
        if (ms <= best_ms) best = kLanes;
    }
    if (tab) table_used(tab, st);
    if (din) cudaFree(din);
    if (dout) cudaFree(dout);
    if (dsyn) cudaFree(dsyn);
    if (dcnt) cudaFree(dcnt);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (rc != HD_OK) return rc;
    if (best >= 0) remember_short_variant(n, best);
    if (chosen) *chosen = best;
    return HD_OK;
}

hd_status hd_short_variant_count(uint32_t *count)
{
    if (!count) return HD_ERR_NULL;
    *count = (uint32_t)kLanes + 1u;
    return HD_OK;
}

hd_status hd_short_variant_select(int32_t ordinal)
{
    if (ordinal > kLanes) return HD_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return HD_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_short_mu);
    g_short_choice[dev] = ordinal < 0 ? 0 : ordinal + 1;
    return HD_OK;
}

}  // extern "C"
