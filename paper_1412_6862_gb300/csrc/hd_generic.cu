// hd_generic.cu -- warp-tile decoder for every supported n.
//
// One warp handles one warp tile of 32 consecutive codewords: n input words
// and k output words (n is odd, so 32 codewords always fill whole words).
// Lane L decodes codeword 32t + L in registers; the lanes then merge their
// data bits into the tile's output words through shared memory.  These
// kernels cover any n, any stream length and every ragged tail; the
// specialised streaming kernels of hd_decode.cu take the bulk of long streams.
#include <cstdint>

#include "hd_device.cuh"
#include "hd_generic.cuh"
#include "hd_internal.h"

namespace hd {
namespace {

constexpr int kGenericWarps = 8;

__global__ void __launch_bounds__(kGenericWarps * 32)
    k_decode_generic(const uint32_t *__restrict__ in, uint64_t in_words, uint32_t n, uint32_t m, uint64_t num_cw,
                     uint64_t tile_begin, uint64_t tile_end, uint32_t *__restrict__ out, uint64_t out_words,
                     void *__restrict__ syn, int syn_type, unsigned long long *__restrict__ err)
{
    __shared__ uint32_t sy[kGenericWarps][kWarpSlotWords];
    __shared__ uint32_t sd[kGenericWarps][kWarpSlotWords];
    const int wp = threadIdx.x >> 5;
    const unsigned long long cnt =
        generic_decode_tiles(in, in_words, n, m, num_cw, tile_begin + (uint64_t)blockIdx.x * kGenericWarps + wp,
                             tile_end, (uint64_t)gridDim.x * kGenericWarps, out, out_words, syn, syn_type, sy[wp],
                             sd[wp]);
    if (err != nullptr && (threadIdx.x & 31) == 0 && cnt != 0) atomicAdd(err, cnt);
}

int grid_for_tiles(uint64_t tiles)
{
    const uint64_t want = (tiles + kGenericWarps - 1) / kGenericWarps;
    const uint64_t cap = (uint64_t)num_sms() * 8;
    return decode_grid(want, cap);
}

}  // namespace

cudaError_t launch_decode_generic(const uint32_t *in, uint64_t in_words, uint32_t n, uint64_t num_cw,
                                  uint64_t tile_begin, uint64_t tile_end, uint32_t *out, uint64_t out_words,
                                  void *syn, int syn_type, unsigned long long *err, cudaStream_t st)
{
    if (tile_end <= tile_begin) return cudaSuccess;
    const uint32_t m = (uint32_t)code_m(n);
    const int grid = grid_for_tiles(tile_end - tile_begin);
    k_decode_generic<<<grid, kGenericWarps * 32, 0, st>>>(in, in_words, n, m, num_cw, tile_begin, tile_end, out,
                                                          out_words, syn, syn_type, err);
    count_launch();
    return cudaGetLastError();
}

}  // namespace hd
