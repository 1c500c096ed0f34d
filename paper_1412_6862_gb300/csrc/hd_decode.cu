// hd_decode.cu -- registry of the compiled streaming-decoder configurations,
// per-device launch setup, the configuration choice (built-in defaults or the
// autotuner's measured pick) and the device status word.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <tuple>
#include <vector>

#include "hd_internal.h"
#include "hd_stream.cuh"

namespace hd {

void register_stream_a(std::vector<StreamVariant> &v);
void register_stream_b(std::vector<StreamVariant> &v);
void register_stream_c(std::vector<StreamVariant> &v);
void register_stream_secded(std::vector<StreamVariant> &v);
void register_stream_n3(std::vector<StreamVariant> &v);

namespace {

// Scratch input for the autotuner: word i = the high half of SplitMix64
// (Steele, Lea and Flood, 2014) at state seed * 2^32 + i.
__global__ void k_fill_random(uint32_t *p, uint64_t words, uint64_t seed)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t z = (seed << 32) + i + 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        p[i] = (uint32_t)((z ^ (z >> 31)) >> 32);
    }
}

__device__ uint32_t g_hd_status;

std::mutex g_mu;

const std::vector<StreamVariant> &variants()
{
    static const std::vector<StreamVariant> v = [] {
        std::vector<StreamVariant> a;
        register_stream_a(a);
        register_stream_b(a);
        register_stream_c(a);
        return a;
    }();
    return v;
}

const std::vector<StreamVariant> &secded_variants()
{
    static const std::vector<StreamVariant> v = [] {
        std::vector<StreamVariant> a;
        register_stream_secded(a);
        return a;
    }();
    return v;
}

int current_device()
{
    int d = 0;
    cudaGetDevice(&d);
    return d;
}

// (device, kernel) -> resident CTAs per SM (0 = not yet configured)
std::map<std::pair<int, const void *>, int> g_bps;
// (device, n, syn) -> chosen variant index (autotuner or explicit selection)
std::map<std::tuple<int, uint32_t, int>, int> g_choice;
// (device, n, syn) whose choice the caller pinned
std::set<std::tuple<int, uint32_t, int>> g_pinned;
// (device, n, syn) -> pinned SECDED configuration (index into secded_variants())
std::map<std::tuple<int, uint32_t, int>, int> g_secded_choice;

// Built-in choice per (n, syndrome type or -1 for any, G, T, S, inplace,
// decode table), measured on GB300; used until the autotuner or the caller
// picks another configuration.  The first entry of n that matches the
// syndrome type and is compiled for it wins.  At 2^24 codewords: n = 15 with u16
// syndromes 18.1 us in place against 18.9 for the 576-thread configuration with
// separate output buffers; n = 31 with u16 syndromes 26.4 us with 16 codewords per
// thread, 27.4 with 32; n = 63 with none / u8 / u16 syndromes 40.9 / 42.6 / 47.0 us
// with separate output buffers (one CTA per SM, its four warps' loads a whole chunk
// further ahead), 41.4 / 47.7 / 52.0 in place with three stages (two CTAs per SM);
// at 2^26 codewords with u8 syndromes 169 against 186.
struct DefaultCfg {
    uint32_t n;
    int syn, G, T, S, inplace, lut;
};
constexpr DefaultCfg kDefaults[] = {
    {7, -1, 32, 128, 4, 1, 1},  {15, 2, 32, 512, 2, 1, 1},   {15, -1, 32, 576, 2, 0, 1},
    {15, -1, 32, 512, 2, 1, 1}, {31, 2, 16, 256, 3, 1, 0},   {31, -1, 32, 128, 3, 1, 0}, {63, -1, 32, 128, 3, 0, 0},
    {127, -1, 8, 256, 3, 1, 0}, {255, -1, 8, 128, 2, 1, 0},
};

// SECDED: the built-in arithmetic configuration, the first compiled one of n unless
// listed here (2^24 codewords, u8 syndromes: n = 31 24.4 us with four stages of 128
// threads against 26.1 with two of 256, n = 63 45.4 against 46.6 for 64 threads).
constexpr DefaultCfg kSecdedDefaults[] = {
    {31, -1, 32, 128, 4, 1, 0},
    {63, -1, 32, 128, 3, 1, 0},
};

bool secded_default(const StreamVariant &x)
{
    for (const auto &d : kSecdedDefaults)
        if (d.n == x.n && (d.syn < 0 || d.syn == x.syn) && d.G == x.G && d.T == x.T && d.S == x.S &&
            d.inplace == x.inplace)
            return true;
    return false;
}

int find_variant(uint32_t n, int syn, int G, int T, int S, int inplace, int lut)
{
    const auto &v = variants();
    for (size_t i = 0; i < v.size(); ++i)
        if (v[i].n == n && v[i].syn == syn && v[i].G == G && v[i].T == T && v[i].S == S &&
            v[i].inplace == inplace && v[i].lut == lut)
            return (int)i;
    return -1;
}

int find_default_variant(uint32_t n, int syn)
{
    for (const auto &d : kDefaults)
        if (d.n == n && (d.syn < 0 || d.syn == syn)) {
            const int i = find_variant(n, syn, d.G, d.T, d.S, d.inplace, d.lut);
            if (i >= 0) return i;
        }
    const auto &v = variants();
    for (size_t i = 0; i < v.size(); ++i)
        if (v[i].n == n && v[i].syn == syn) return (int)i;
    return -1;
}

// The built-in configuration of (n, syn), looked up once.
int default_variant(uint32_t n, int syn)
{
    struct Table {
        int v[9][3];
        Table()
        {
            for (int m = 0; m <= 8; ++m)
                for (int t = 0; t < 3; ++t) v[m][t] = find_default_variant((1u << m) - 1u, t);
        }
    };
    static const Table table;
    const int m = code_m(n);
    return m != 0 && syn >= 0 && syn < 3 ? table.v[m][syn] : -1;
}

// Whether any configuration was ever chosen (tuned or pinned) in this process:
// until then every launch takes the built-in ones without a lock.
std::atomic<bool> g_any_choice{false};

int chosen_variant(uint32_t n, int syn)
{
    if (!g_any_choice.load(std::memory_order_acquire)) return default_variant(n, syn);
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_choice.find({current_device(), n, syn});
    if (it != g_choice.end()) return it->second;
    return default_variant(n, syn);
}

}  // namespace

int stream_blocks_per_sm(const void *kernel, int threads, uint32_t smem)
{
    const int dev = current_device();
    std::lock_guard<std::mutex> lk(g_mu);
    int &b = g_bps[{dev, kernel}];
    if (b == 0) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return -1;
        int v = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kernel, threads, smem) != cudaSuccess) return -1;
        b = v > 0 ? v : -1;
    }
    return b;
}

uint32_t *status_ptr()
{
    static std::atomic<uint32_t *> cached[64];
    const int dev = current_device();
    const bool in_range = dev >= 0 && dev < 64;
    if (in_range)
        if (uint32_t *p = cached[dev].load(std::memory_order_acquire)) return p;
    void *a = nullptr;
    if (cudaGetSymbolAddress(&a, g_hd_status) != cudaSuccess) return nullptr;
    if (in_range) cached[dev].store(static_cast<uint32_t *>(a), std::memory_order_release);
    return static_cast<uint32_t *>(a);
}

uint32_t read_clear_status_decode()
{
    uint32_t v = 0, zero = 0;
    cudaMemcpyFromSymbol(&v, g_hd_status, sizeof(v));
    cudaMemcpyToSymbol(g_hd_status, &zero, sizeof(zero));
    return v;
}

namespace {

// Whole chunks of configuration v, and the ragged tail in the same launch.
StreamArgs stream_args(const StreamVariant &v, const DecodeJob &j, uint32_t *status, const uint16_t *lut)
{
    const uint64_t nchunks = j.num_cw / v.chunk_cw;
    return StreamArgs{j.in,    j.out,    j.syn_type != 0 ? j.syn : nullptr,
                      j.err,   j.det,    status,
                      lut,     nchunks,  j.num_cw,
                      words_for_bits(j.num_cw * (j.n + (j.xh ? 1u : 0u))), words_for_bits(j.num_cw * (j.n - (uint32_t)code_m(j.n))),
                      nchunks * v.chunk_cw / 32, (j.num_cw + 31) / 32};
}

// n = 3 (a codeword is three copies of its bit) has one streaming configuration,
// outside the selectable ones.
const StreamVariant *variant_n3(int syn)
{
    static const std::vector<StreamVariant> v = [] {
        std::vector<StreamVariant> a;
        register_stream_n3(a);
        return a;
    }();
    for (const StreamVariant &x : v)
        if (x.syn == syn) return &x;
    return nullptr;
}

}  // namespace

bool variant_pinned(uint32_t n, int syn)
{
    if (!g_any_choice.load(std::memory_order_acquire)) return false;
    std::lock_guard<std::mutex> lk(g_mu);
    return g_pinned.count({current_device(), n, syn}) != 0;
}

bool secded_variant_pinned(uint32_t n, int syn)
{
    if (!g_any_choice.load(std::memory_order_acquire)) return false;
    std::lock_guard<std::mutex> lk(g_mu);
    return g_secded_choice.count({current_device(), n, syn}) != 0;
}

// The streaming configuration that decodes a plain-code job, or nullptr for one
// codeword per lane.
static const StreamVariant *stream_variant(const DecodeJob &j)
{
    if (!variant_pinned(j.n, j.syn_type) && lanes_suffice(j.n, j.xh, j.num_cw)) return nullptr;
    const StreamVariant *v = nullptr;
    if (j.n == 3) {
        v = variant_n3(j.syn_type);
    } else {
        const int idx = chosen_variant(j.n, j.syn_type);
        if (idx >= 0) v = &variants()[idx];
    }
    return v != nullptr && j.num_cw >= v->chunk_cw ? v : nullptr;  // at least one whole chunk
}

bool decodes_by_lanes(const DecodeJob &j) { return stream_variant(j) == nullptr; }

cudaError_t launch_decode(const DecodeJob &j, cudaStream_t st, bool pdl)
{
    const StreamVariant *v = stream_variant(j);
    const uint16_t *lut = v != nullptr && v->lut ? lut_ptr(j.n, st) : nullptr;
    // no table yet: first call inside a capture
    if (v == nullptr || (v->lut && lut == nullptr)) return launch_decode_lanes(j, false, st, pdl);
    uint32_t *status = status_ptr();
    if (status == nullptr) return cudaErrorInvalidSymbol;
    return v->launch(stream_args(*v, j, status, lut), st, pdl);
}

// SECDED: the streaming kernel with codewords of n + 1 bits.
cudaError_t launch_decode_secded(const DecodeJob &j, cudaStream_t st, bool pdl)
{
    int pinned = -1;
    if (g_any_choice.load(std::memory_order_acquire)) {
        std::lock_guard<std::mutex> lk(g_mu);
        auto it = g_secded_choice.find({current_device(), j.n, j.syn_type});
        if (it != g_secded_choice.end()) pinned = it->second;
    }
    if (pinned < 0 && lanes_suffice(j.n, j.xh, j.num_cw)) return launch_decode_lanes(j, false, st, pdl);
    // a pinned configuration (hd_secded_variant_select), else the table
    // configuration when its table is filled (not while `st` captures before
    // the first fill), else the arithmetic one
    const StreamVariant *v = nullptr, *vt = nullptr;
    for (const StreamVariant &x : secded_variants())
        if (x.n == j.n && x.syn == j.syn_type) {
            if (!x.lut) {
                if (v == nullptr || secded_default(x)) v = &x;
            } else if (vt == nullptr) {
                vt = &x;
            }
        }
    if (pinned >= 0) {
        const StreamVariant &x = secded_variants()[pinned];
        if (x.lut) vt = &x;
        else v = &x, vt = nullptr;
    }
    const uint16_t *lut = vt != nullptr ? lut_ptr(j.n, st, true) : nullptr;
    if (lut != nullptr) v = vt;
    if (v == nullptr || j.num_cw < v->chunk_cw) return launch_decode_lanes(j, false, st, pdl);
    uint32_t *status = status_ptr();
    if (status == nullptr) return cudaErrorInvalidSymbol;
    return v->launch(stream_args(*v, j, status, v->lut ? lut : nullptr), st, pdl);
}

// ---------------------------------------------------------------------------
// Variant queries, explicit selection and the autotuner (C ABI in hd.h)
// ---------------------------------------------------------------------------
static void fill_info(int idx, hd_variant_info *info)
{
    const StreamVariant &v = variants()[idx];
    std::memset(info, 0, sizeof(*info));
    info->index = (uint32_t)idx;
    info->n = v.n;
    info->syn_type = (uint32_t)v.syn;
    info->codewords_per_thread = (uint32_t)v.G;
    info->threads = (uint32_t)v.T;
    info->stages = (uint32_t)v.S;
    info->inplace = (uint32_t)v.inplace;
    info->smem_bytes = v.smem;
    info->chunk_codewords = v.chunk_cw;
    info->blocks_per_sm = stream_blocks_per_sm(v.kernel, v.T, v.smem);
    info->measured_us = -1.0f;
    info->table_lookup = (uint32_t)v.lut;
}

}  // namespace hd

using namespace hd;

extern "C" {

hd_status hd_variant_count(uint32_t n, hd_syn_type syn_type, uint32_t *count)
{
    if (!count) return HD_ERR_NULL;
    if (code_m(n) == 0) return HD_ERR_INVALID_N;
    uint32_t c = 0;
    for (const auto &v : variants())
        if (v.n == n && v.syn == (int)syn_type) ++c;
    *count = c;
    return HD_OK;
}

hd_status hd_variant_info_get(uint32_t n, hd_syn_type syn_type, uint32_t ordinal, hd_variant_info *info)
{
    if (!info) return HD_ERR_NULL;
    if (code_m(n) == 0) return HD_ERR_INVALID_N;
    uint32_t c = 0;
    const auto &v = variants();
    for (size_t i = 0; i < v.size(); ++i) {
        if (v[i].n == n && v[i].syn == (int)syn_type) {
            if (c == ordinal) {
                fill_info((int)i, info);
                info->index = ordinal;
                return HD_OK;
            }
            ++c;
        }
    }
    return HD_ERR_INVALID_ARG;
}

hd_status hd_variant_select(uint32_t n, hd_syn_type syn_type, int32_t ordinal)
{
    if (code_m(n) == 0) return HD_ERR_INVALID_N;
    const int dev = current_device();
    std::lock_guard<std::mutex> lk(g_mu);
    if (ordinal < 0) {
        g_choice.erase({dev, n, (int)syn_type});
        g_pinned.erase({dev, n, (int)syn_type});
        return HD_OK;
    }
    int32_t c = 0;
    const auto &v = variants();
    for (size_t i = 0; i < v.size(); ++i) {
        if (v[i].n == n && v[i].syn == (int)syn_type) {
            if (c == ordinal) {
                g_choice[{dev, n, (int)syn_type}] = (int)i;
                g_any_choice.store(true, std::memory_order_release);
                g_pinned.insert({dev, n, (int)syn_type});
                return HD_OK;
            }
            ++c;
        }
    }
    return HD_ERR_INVALID_ARG;
}

hd_status hd_variant_current(uint32_t n, hd_syn_type syn_type, hd_variant_info *info)
{
    if (!info) return HD_ERR_NULL;
    if (code_m(n) == 0) return HD_ERR_INVALID_N;
    const int idx = chosen_variant(n, (int)syn_type);
    if (idx < 0) return HD_ERR_INVALID_ARG;
    fill_info(idx, info);
    // report the ordinal within (n, syn) rather than the global index
    uint32_t c = 0;
    const auto &v = variants();
    for (int i = 0; i < idx; ++i)
        if (v[i].n == n && v[i].syn == (int)syn_type) ++c;
    info->index = c;
    return HD_OK;
}

hd_status hd_secded_variant_count(uint32_t n, hd_syn_type syn_type, uint32_t *count)
{
    if (!count) return HD_ERR_NULL;
    if (code_m(n) == 0) return HD_ERR_INVALID_N;
    uint32_t c = 0;
    for (const auto &v : secded_variants())
        if (v.n == n && v.syn == (int)syn_type) ++c;
    *count = c;
    return HD_OK;
}

hd_status hd_secded_variant_info_get(uint32_t n, hd_syn_type syn_type, uint32_t ordinal, hd_variant_info *info)
{
    if (!info) return HD_ERR_NULL;
    if (code_m(n) == 0) return HD_ERR_INVALID_N;
    uint32_t c = 0;
    for (const StreamVariant &v : secded_variants()) {
        if (v.n != n || v.syn != (int)syn_type) continue;
        if (c++ != ordinal) continue;
        std::memset(info, 0, sizeof(*info));
        info->index = ordinal;
        info->n = v.n;
        info->syn_type = (uint32_t)v.syn;
        info->codewords_per_thread = (uint32_t)v.G;
        info->threads = (uint32_t)v.T;
        info->stages = (uint32_t)v.S;
        info->inplace = (uint32_t)v.inplace;
        info->smem_bytes = v.smem;
        info->chunk_codewords = v.chunk_cw;
        info->blocks_per_sm = stream_blocks_per_sm(v.kernel, v.T, v.smem);
        info->measured_us = -1.0f;
        info->table_lookup = (uint32_t)v.lut;
        return HD_OK;
    }
    return HD_ERR_INVALID_ARG;
}

hd_status hd_secded_variant_select(uint32_t n, hd_syn_type syn_type, int32_t ordinal)
{
    if (code_m(n) == 0) return HD_ERR_INVALID_N;
    const int dev = current_device();
    std::lock_guard<std::mutex> lk(g_mu);
    if (ordinal < 0) {
        g_secded_choice.erase({dev, n, (int)syn_type});
        return HD_OK;
    }
    int32_t c = 0;
    const auto &v = secded_variants();
    for (size_t i = 0; i < v.size(); ++i) {
        if (v[i].n == n && v[i].syn == (int)syn_type) {
            if (c == ordinal) {
                g_secded_choice[{dev, n, (int)syn_type}] = (int)i;
                g_any_choice.store(true, std::memory_order_release);
                return HD_OK;
            }
            ++c;
        }
    }
    return HD_ERR_INVALID_ARG;
}

hd_status hd_autotune(uint32_t n, hd_syn_type syn_type, uint64_t num_codewords, uint32_t reps, void *cuda_stream,
                      hd_variant_info *chosen)
{
    const int m = code_m(n);
    if (m == 0) return HD_ERR_INVALID_N;
    if (syn_type != HD_SYN_NONE && syn_type != HD_SYN_U8 && syn_type != HD_SYN_U16) return HD_ERR_INVALID_ARG;
    if (num_codewords == 0 || num_codewords > (1ull << 32)) return HD_ERR_SIZE;
    if (reps == 0) reps = 5;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const uint32_t k = n - (uint32_t)m;
    const uint64_t in_words = words_for_bits(num_codewords * n) + 4;
    const size_t in_b = in_words * 4;
    const size_t out_b = words_for_bits(num_codewords * k) * 4 + 16;
    const size_t syn_b = num_codewords * 2 + 16;
    // Enough buffer sets that one round over them streams at least twice the
    // L2 (at most kMaxSets), so every timed launch reads its input from HBM
    // as a long stream would.
    constexpr int kMaxSets = 8;
    int l2 = 0;
    if (cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, current_device()) != cudaSuccess) l2 = 0;
    const size_t set_b = in_b + out_b + syn_b;
    const int nsets = (int)std::min<size_t>(kMaxSets, std::max<size_t>(1, (2 * (size_t)l2 + set_b - 1) / set_b));
    void *din[kMaxSets] = {}, *dout[kMaxSets] = {}, *dsyn[kMaxSets] = {};
    void *derr = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    hd_status rc = HD_OK;
    for (int i = 0; rc == HD_OK && i < nsets; ++i)
        if (cudaMalloc(&din[i], in_b) != cudaSuccess || cudaMalloc(&dout[i], out_b) != cudaSuccess ||
            cudaMalloc(&dsyn[i], syn_b) != cudaSuccess)
            rc = HD_ERR_CUDA;
    if (rc == HD_OK && (cudaMalloc(&derr, 8) != cudaSuccess || cudaEventCreate(&e0) != cudaSuccess ||
                        cudaEventCreate(&e1) != cudaSuccess))
        rc = HD_ERR_CUDA;
    uint32_t *status = status_ptr();
    if (rc == HD_OK && status == nullptr) rc = HD_ERR_CUDA;
    // random received words: table lookups then spread over the table as with
    // real data (a constant fill would make every lane read the same entry)
    for (int i = 0; rc == HD_OK && i < nsets; ++i) {
        k_fill_random<<<num_sms() * 4, 256, 0, st>>>(static_cast<uint32_t *>(din[i]), in_words, 0x5A17u + i);
        if (cudaGetLastError() != cudaSuccess) rc = HD_ERR_CUDA;
    }
    // candidates: one warm-up launch each
    struct Cand {
        int idx;
        uint64_t nchunks;
        const uint16_t *lut;
        std::vector<float> us;
    };
    std::vector<Cand> cands;
    const auto &vs = variants();
    auto *er = static_cast<unsigned long long *>(derr);
    // the whole chunks of buffer set i (no tail: the chunked prefix differs per configuration)
    auto set_args = [&](const StreamVariant &v, int i, const uint16_t *lut) {
        DecodeJob j{};
        j.in = static_cast<const uint32_t *>(din[i]);
        j.n = n;
        j.num_cw = num_codewords / v.chunk_cw * v.chunk_cw;
        j.out = static_cast<uint32_t *>(dout[i]);
        j.syn = dsyn[i];
        j.syn_type = (int)syn_type;
        j.err = er;
        return stream_args(v, j, status, lut);
    };
    for (size_t i = 0; rc == HD_OK && i < vs.size(); ++i) {
        const StreamVariant &v = vs[i];
        if (v.n != n || v.syn != (int)syn_type) continue;
        const uint64_t nchunks = num_codewords / v.chunk_cw;
        if (nchunks == 0) continue;
        if (stream_blocks_per_sm(v.kernel, v.T, v.smem) <= 0) continue;
        const uint16_t *lut = v.lut ? lut_ptr(n, st) : nullptr;
        if (v.lut && lut == nullptr) continue;
        if (v.launch(set_args(v, 0, lut), st, false) != cudaSuccess) {
            rc = HD_ERR_CUDA;
            break;
        }
        cands.push_back({(int)i, nchunks, lut, {}});
    }
    // rounds: every candidate once per round, over all buffer sets, so that
    // slow drifts of the clock affect all candidates alike; median per candidate
    for (uint32_t r = 0; rc == HD_OK && r < reps; ++r)
        for (Cand &c : cands) {
            const StreamVariant &v = vs[c.idx];
            cudaEventRecord(e0, st);
            for (int i = 0; i < nsets; ++i)
                v.launch(set_args(v, i, c.lut), st, false);
            cudaEventRecord(e1, st);
            if (cudaEventSynchronize(e1) != cudaSuccess) {
                rc = HD_ERR_CUDA;
                break;
            }
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            // normalise to the whole request (the chunked prefix differs per variant)
            c.us.push_back(ms * 1000.f / (float)nsets * (float)num_codewords / (float)(c.nchunks * v.chunk_cw));
        }
    int best = -1;
    float best_us = 0.f, default_us = -1.f;
    const int dflt = default_variant(n, (int)syn_type);
    for (Cand &c : cands) {
        if (c.us.empty()) continue;
        std::sort(c.us.begin(), c.us.end());
        const float us = c.us[c.us.size() / 2];
        if (c.idx == dflt) default_us = us;
        if (best < 0 || us < best_us) {
            best = c.idx;
            best_us = us;
        }
    }
    // the built-in choice stays unless another configuration beats it by more
    // than the run-to-run noise of these timings
    constexpr float kMargin = 1.02f;
    if (default_us > 0.f && default_us <= best_us * kMargin) {
        best = dflt;
        best_us = default_us;
    }
    for (int i = 0; i < nsets; ++i) {
        if (din[i]) cudaFree(din[i]);
        if (dout[i]) cudaFree(dout[i]);
        if (dsyn[i]) cudaFree(dsyn[i]);
    }
    if (derr) cudaFree(derr);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (rc != HD_OK) return rc;
    if (best < 0) return HD_ERR_SIZE;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        g_choice[{current_device(), n, (int)syn_type}] = best;
        g_any_choice.store(true, std::memory_order_release);
        g_pinned.erase({current_device(), n, (int)syn_type});
    }
    if (chosen) {
        hd_variant_current(n, syn_type, chosen);
        chosen->measured_us = best_us;
    }
    return HD_OK;
}

}  // extern "C"
