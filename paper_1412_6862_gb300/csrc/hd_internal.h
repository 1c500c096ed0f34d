// hd_internal.h -- host-side declarations shared by the translation units of
// libhd.so.  Not installed; the public interface is include/hd.h.
#pragma once

#include <array>
#include <atomic>
#include <cstdint>
#include <utility>
#include <cuda_runtime.h>

#include "hd.h"

namespace hd {

// Kernels launched by this library (hd_launch_count()).
extern std::atomic<uint64_t> g_launches;
inline void count_launch(uint64_t c = 1) { g_launches.fetch_add(c, std::memory_order_relaxed); }

// m for n = 2^m - 1 (2 <= m <= 8), else 0.
inline int code_m(uint32_t n)
{
    for (int m = 2; m <= 8; ++m)
        if (n == (1u << m) - 1u) return m;
    return 0;
}

inline uint64_t words_for_bits(uint64_t bits) { return (bits + 31) >> 5; }

// Multiprocessor count of the current device (cached per device).
int num_sms();

// Upper bound on the CTAs of one decode launch (hd_set_max_ctas(); 0 = none).
extern std::atomic<uint32_t> g_max_ctas;

// Grid of a decode launch: `want` CTAs (enough for the work), at most `cap`
// (what the device holds at once) and at most the caller's limit; at least 1.
inline int decode_grid(uint64_t want, uint64_t cap)
{
    uint64_t g = want < cap ? want : cap;
    const uint32_t lim = g_max_ctas.load(std::memory_order_relaxed);
    if (lim != 0 && g > lim) g = lim;
    return (int)(g > 0 ? g : 1);
}

// One stream to decode: plain code of length n, or with xh its SECDED extension
// (codewords of n + 1 bits).  syn_type 0 stores no syndromes; err / det may be null.
struct DecodeJob {
    const uint32_t *in;
    uint32_t n;
    uint64_t num_cw;
    uint32_t *out;
    void *syn;
    int syn_type;
    unsigned long long *err, *det;
    bool xh;
};

// The one-codeword-per-lane decoder, for any stream length.  direct: the whole
// stream is one CTA's work (lanes_one_cta) and *err / *det are overwritten, so
// that nothing needs clearing ahead; else they are added to.
cudaError_t launch_decode_lanes(const DecodeJob &j, bool direct, cudaStream_t st, bool pdl);
bool lanes_one_cta(uint64_t num_cw);
// Whether a stream is short enough that one codeword per lane beats whole chunks.
bool lanes_suffice(uint32_t n, bool xh, uint64_t num_cw);

// The encoders (any supported n, any length): data_words / stream_words are the
// buffers' lengths; launched as programmatic dependents of the kernel ahead.
cudaError_t launch_encode(const uint32_t *data, uint64_t data_words, uint32_t n, uint64_t num_cw, uint32_t *stream,
                          uint64_t stream_words, cudaStream_t st);
cudaError_t launch_encode_secded(const uint32_t *data, uint64_t data_words, uint32_t n, uint64_t num_cw,
                                 uint32_t *stream, cudaStream_t st);

// Words of the fullest shared-memory bank when a warp's teams of 2^lg lanes read the same
// word of segments `bits` apart, per lg.
using BankWays = std::array<uint8_t, 6>;
const BankWays &bank_ways(uint32_t bits);

cudaError_t launch_encode_short(const uint32_t *data, uint32_t n, uint32_t k, uint64_t num_cw, uint32_t *stream,
                                cudaStream_t st);

// Resident CTAs per SM of a kernel with `smem` bytes of dynamic shared memory
// (opted in to on first use), cached per device; <= 0 on failure.
int stream_blocks_per_sm(const void *kernel, int threads, uint32_t smem);

// stream_blocks_per_sm() of one kernel, kept per device without a lock: one static
// instance per kernel (its threads and shared memory never change).
class BlocksPerSm {
    std::atomic<int> v_[64] = {};

public:
    int get(const void *kernel, int threads, uint32_t smem)
    {
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev < 0 || dev >= 64) return stream_blocks_per_sm(kernel, threads, smem);
        int v = v_[dev].load(std::memory_order_relaxed);
        if (v == 0) {
            v = stream_blocks_per_sm(kernel, threads, smem);
            if (v > 0) v_[dev].store(v, std::memory_order_relaxed);
        }
        return v;
    }
};

// Whether `st` records into a graph.
inline bool stream_capturing(cudaStream_t st)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return cs != cudaStreamCaptureStatusNone;
}

// Launch `kern` on `st`, as the programmatic dependent of the kernel ahead of
// it in the stream when pdl is set (it may then start before that kernel has
// finished, and must wait for it before touching what that kernel writes).
template <typename... KArgs, typename... Args>
cudaError_t launch_kernel_uncounted(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                    bool pdl, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = pdl ? &attr : nullptr;
    cfg.numAttrs = pdl ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// launch_kernel_uncounted, counted in hd_launch_count().
template <typename... KArgs, typename... Args>
cudaError_t launch_kernel(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                          Args &&...args)
{
    count_launch();
    return launch_kernel_uncounted(kern, grid, block, smem, st, pdl, std::forward<Args>(args)...);
}

// Clear one or two device counters (either may be NULL) with a one-thread
// kernel that lets the next kernel of the stream start at once (programmatic
// dependent launch): a launch with pdl = true below overlaps it and waits for
// it before touching global memory.  Inside a CUDA graph this costs far less
// than a memset node between two kernels.  chained: the clear is itself
// launched as the programmatic dependent of the kernel ahead of it (it waits
// for that kernel before writing), so that it and the decode behind it can
// start while that kernel drains; only for decodes that wait before their
// first global access.
cudaError_t launch_zero_counts(unsigned long long *a, unsigned long long *b, cudaStream_t st, bool chained = false);

// Decode a stream (num_cw > 0) on `st` in one launch: the streaming kernel with
// its ragged tail, or one codeword per lane.  The counters are added to.  pdl:
// launched as the programmatic dependent of the kernel ahead.
cudaError_t launch_decode(const DecodeJob &j, cudaStream_t st, bool pdl);
// Whether launch_decode takes a job one codeword per lane.
bool decodes_by_lanes(const DecodeJob &j);
cudaError_t launch_decode_secded(const DecodeJob &j, cudaStream_t st, bool pdl);

// Whether the caller pinned a configuration (hd_variant_select, not the
// autotuner's pick; hd_secded_variant_select): short streams take it too.
bool variant_pinned(uint32_t n, int syn);
bool secded_variant_pinned(uint32_t n, int syn);

// Decode table of n = 7 or 15 (data | s << k per codeword; with xh the SECDED
// table of n + 1 bits, data | s << k | P << (k + m)), filled on `st` on first
// use per device; nullptr for other n, or when the table is not filled yet and
// `st` is capturing.
const uint16_t *lut_ptr(uint32_t n, cudaStream_t st, bool xh = false);

// Device address of the status word that kernels latch HD_ERR_TIMEOUT into
// (per device; nullptr on failure), and its host-side read-and-clear.
uint32_t *status_ptr();
uint32_t read_clear_status_decode();

}  // namespace hd
