// hd_lanes.cu -- decode of short streams, one codeword per lane (plain codes
// and SECDED, every n).
//
// A chunk of the streaming kernel is 8 to 32 codewords a lane one after the
// other, so a stream of few chunks keeps few warps busy for 4 to 6 us.  Here a
// warp takes 32 codewords at a time and a CTA holds no ring, so the whole
// stream is in flight at once.  A stream of at most kOneCtaTiles tiles is one
// CTA's work, which adds up its counts in shared memory and overwrites
// err_count / detected_count itself: one launch instead of the counters' clear
// and the decode.
#include <algorithm>
#include <cstdint>

#include "hd_device.cuh"
#include "hd_internal.h"
#include "hd_lane.cuh"

namespace hd {
namespace {

constexpr int kLaneWarps = 8;        // per CTA of a grid
constexpr int kDirectWarps = 16;     // the single CTA: at most 512 threads
constexpr uint64_t kOneCtaTiles = 2 * kDirectWarps;  // 1024 codewords: two rounds

template <int N_, bool XH, int WARPS, bool DIRECT>
__global__ void __launch_bounds__(WARPS * 32)
    k_decode_lanes(const uint32_t *__restrict__ in, uint64_t in_words, uint64_t num_cw, uint32_t *__restrict__ out,
                   uint64_t out_words, void *__restrict__ syn, int syn_type, unsigned long long *__restrict__ err,
                   unsigned long long *__restrict__ det)
{
    __shared__ uint32_t slots[WARPS][32 * kLaneDataSlot<N_>];
    __shared__ uint32_t counts[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    if (threadIdx.x < 2) counts[threadIdx.x] = 0u;
    __syncthreads();
    const uint64_t tiles = (num_cw + 31) / 32;
    uint32_t errs = 0, dets = 0;
    grid_dep_launch_dependents();
    grid_dep_wait();  // the kernels ahead (the counters' clear, and what produced the input) have finished
    for (uint64_t t = (uint64_t)blockIdx.x * warps + warp; t < tiles; t += (uint64_t)gridDim.x * warps)
        decode_lane_tile<N_, XH>(in, in_words, num_cw, t, out, out_words, syn, syn_type, slots[warp], lane, errs, dets);
    if (lane == 0) {
        if (errs) atomicAdd(&counts[0], errs);
        if (dets) atomicAdd(&counts[1], dets);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if constexpr (DIRECT) {
            if (err) *err = counts[0];
            if (det) *det = counts[1];
        } else {
            if (err && counts[0]) atomicAdd(err, (unsigned long long)counts[0]);
            if (det && counts[1]) atomicAdd(det, (unsigned long long)counts[1]);
        }
    }
}

// CTAs of the grid kernel that the device holds at once.
template <int N_, bool XH>
uint64_t lane_ctas()
{
    static BlocksPerSm blocks;
    const int bps =
        blocks.get(reinterpret_cast<const void *>(k_decode_lanes<N_, XH, kLaneWarps, false>), kLaneWarps * 32, 0);
    return (uint64_t)num_sms() * (uint64_t)std::max(bps, 1);
}

template <int N_, bool XH>
cudaError_t launch_lanes(const DecodeJob &j, bool direct, cudaStream_t st, bool pdl)
{
    const uint64_t tiles = (j.num_cw + 31) / 32;
    const uint64_t in_words = words_for_bits(j.num_cw * (N_ + (XH ? 1u : 0u)));
    const uint64_t out_words = words_for_bits(j.num_cw * Code<N_>::k);
    if (direct)
        return launch_kernel(k_decode_lanes<N_, XH, kDirectWarps, true>, dim3(1),
                             dim3(32u * (unsigned)std::min<uint64_t>(tiles, kDirectWarps)), 0, st, pdl, j.in, in_words,
                             j.num_cw, j.out, out_words, j.syn, j.syn_type, j.err, j.det);
    const int grid = decode_grid((tiles + kLaneWarps - 1) / kLaneWarps, lane_ctas<N_, XH>());
    return launch_kernel(k_decode_lanes<N_, XH, kLaneWarps, false>, dim3((unsigned)grid), dim3(kLaneWarps * 32), 0, st,
                         pdl, j.in, in_words, j.num_cw, j.out, out_words, j.syn, j.syn_type, j.err, j.det);
}

template <int N_, bool XH>
bool suffice(uint64_t num_cw)
{
    const uint64_t ctas = lane_ctas<N_, XH>();
    return (num_cw + 31) / 32 <= (uint64_t)decode_grid(ctas, ctas) * kLaneWarps;
}

// f<n, XH>(args...) for the n of a job.
#define HD_FOR_N(n, XH, f, other, ...)        \
    switch (n) {                              \
        case 3: return f<3, XH>(__VA_ARGS__);     \
        case 7: return f<7, XH>(__VA_ARGS__);     \
        case 15: return f<15, XH>(__VA_ARGS__);   \
        case 31: return f<31, XH>(__VA_ARGS__);   \
        case 63: return f<63, XH>(__VA_ARGS__);   \
        case 127: return f<127, XH>(__VA_ARGS__); \
        case 255: return f<255, XH>(__VA_ARGS__); \
        default: return other;                \
    }

template <bool XH>
cudaError_t dispatch(const DecodeJob &j, bool direct, cudaStream_t st, bool pdl)
{
    HD_FOR_N(j.n, XH, launch_lanes, cudaErrorInvalidValue, j, direct, st, pdl)
}

template <bool XH>
bool dispatch_suffice(uint32_t n, uint64_t num_cw)
{
    HD_FOR_N(n, XH, suffice, false, num_cw)
}

}  // namespace

bool lanes_one_cta(uint64_t num_cw) { return num_cw <= 32 * kOneCtaTiles; }

// One round of tiles on the CTAs a launch may have and the device holds at once
// (152 SMs: 311,296 codewords, fewer for the long codes' wider kernels).  On GB300
// the paths cross about there; u16 syndromes, lanes against chunks: n = 31 2.2
// against 4.1 us at 20,000 codewords, 3.0 against 4.1 at 100,000, 4.3 against 4.2 at
// 300,000; n = 255 3.1 against 3.9 at 20,000, 5.0 against 4.8 at 100,000; SECDED
// n = 63 2.3 against 5.0 at 20,000, 4.5 against 5.0 at 300,000.
bool lanes_suffice(uint32_t n, bool xh, uint64_t num_cw)
{
    return xh ? dispatch_suffice<true>(n, num_cw) : dispatch_suffice<false>(n, num_cw);
}

cudaError_t launch_decode_lanes(const DecodeJob &j, bool direct, cudaStream_t st, bool pdl)
{
    return j.xh ? dispatch<true>(j, direct, st, pdl) : dispatch<false>(j, direct, st, pdl);
}

}  // namespace hd
