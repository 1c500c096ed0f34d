// hd_secded.cu -- SECDED decoding (extended Hamming codes), an extension of the
// paper's single-error decoder that is not in the paper: a full-length code
// n = 2^m - 1 plus an overall parity bit at position 0, so a codeword has
// n + 1 = 2^m bits and 32 codewords fill n + 1 words.  The overall parity P
// of the n + 1 bits decides: P = 1, one error, flip position s (s = 0 is the
// parity bit itself); P = 0 with s != 0, two errors, detected and left as
// received.  The decode is the streaming kernel compiled with XH (see
// hd_stream_x.cu), or one codeword per lane for short streams (hd_lanes.cu).
#include <algorithm>
#include <cstdint>

#include "hd_internal.h"

namespace hd {
namespace {

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace
}  // namespace hd

using namespace hd;

extern "C" {

hd_status hd_decode_secded(const uint32_t *stream, uint64_t in_bits, uint32_t n, uint64_t num_codewords,
                           uint32_t *out_bits, void *syndromes, hd_syn_type syn_type, unsigned long long *err_count,
                           unsigned long long *detected_count, void *cuda_stream)
{
    const int m = code_m(n);
    if (m == 0) return HD_ERR_INVALID_N;
    if (syn_type != HD_SYN_NONE && syn_type != HD_SYN_U8 && syn_type != HD_SYN_U16) return HD_ERR_INVALID_ARG;
    if (syn_type == HD_SYN_U8 && m == 8) return HD_ERR_INVALID_ARG;  // s | P << 8 needs 9 bits
    if (num_codewords > (1ull << 40)) return HD_ERR_SIZE;
    if (in_bits != (uint64_t)(n + 1u) * num_codewords) return HD_ERR_SIZE;
    if (num_codewords != 0) {
        if (!stream || !out_bits) return HD_ERR_NULL;
        if (syn_type != HD_SYN_NONE && !syndromes) return HD_ERR_NULL;
        if (!aligned16(stream) || !aligned16(out_bits) || (syndromes && !aligned16(syndromes))) return HD_ERR_ALIGN;
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const bool counted = err_count != nullptr || detected_count != nullptr;
    const DecodeJob j{stream,   n,    num_codewords, out_bits, syndromes, syndromes ? (int)syn_type : 0,
                      err_count, detected_count, true};
    // one CTA's work overwrites the counts itself: no clear
    if (num_codewords != 0 && lanes_one_cta(num_codewords) && !secded_variant_pinned(n, j.syn_type))
        return launch_decode_lanes(j, true, st, true) == cudaSuccess ? HD_OK : HD_ERR_CUDA;
    if (counted && launch_zero_counts(err_count, detected_count, st, true) != cudaSuccess) return HD_ERR_CUDA;
    if (num_codewords == 0) return HD_OK;
    return launch_decode_secded(j, st, true) == cudaSuccess ? HD_OK : HD_ERR_CUDA;
}

hd_status hd_encode_secded(const uint32_t *data_bits, uint32_t n, uint64_t num_codewords, uint32_t *stream,
                           void *cuda_stream)
{
    const int m = code_m(n);
    if (m == 0) return HD_ERR_INVALID_N;
    if (num_codewords > (1ull << 40)) return HD_ERR_SIZE;
    if (num_codewords == 0) return HD_OK;
    if (!data_bits || !stream) return HD_ERR_NULL;
    if (!aligned16(data_bits) || !aligned16(stream)) return HD_ERR_ALIGN;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const uint32_t k = n - (uint32_t)m;
    return launch_encode_secded(data_bits, words_for_bits(num_codewords * k), n, num_codewords, stream, st) == cudaSuccess
               ? HD_OK
               : HD_ERR_CUDA;
}

}  // extern "C"
