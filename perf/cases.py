"""The decoder's working set of calls, for timing: what a receiver (or the
transmitter that feeds it) has this library do, through its public entry
points, from one short packet to streams far larger than the GPU's L2.

A case names the entry point (``call``), the code and the size:

* ``decode``, ``decode_secded``, ``encode``, ``encode_secded`` and ``encode_short``:
  one stream of ``N`` codewords of length ``n`` in device memory;
* ``decode_short``: the same through a ``ShortPlan`` kept by the program;
* ``streams``: several streams side by side (``hd_decode_streams``), ``jobs`` = "n:N,n:N";
* ``plan`` / ``batch``: ``packets`` packets of mixed n and length drawn from ``table``
  (``synth.packet_table``), through a plan kept by the program or in one shot;
* ``host``: a stream in pinned host memory, decoded into pinned host memory.

``syn`` is 0 (no syndromes), 1 (u8) or 2 (u16).  Received streams are encoded
random messages with channel errors: one flipped bit in about 10 % of the
codewords (5 % for the long codes) and two in about one in a hundred.
"""
import math

import torch

from paper_1412_6862_gb300 import hd, synth

LENGTHS = (3, 7, 15, 31, 63, 127, 255)
PACKET_MAX_BITS = 4 * 1024 * 1024


def listed():
    return [
        # one short packet: a receiver that decodes each as it arrives
        {"name": "packet 63x500", "call": "decode", "n": 63, "N": 500, "syn": 1},
        # the (7,4) workload of 2^20 codewords: stays in L2
        {"name": "decode 7x2^20", "call": "decode", "n": 7, "N": 1 << 20, "syn": 1},
        # a capture of (31,26) codewords of no round length
        {"name": "decode 31 ragged", "call": "decode", "n": 31, "N": 20_000_003, "syn": 1},
        # the largest: about a gigabyte of (63,57)
        {"name": "decode 63x2^26", "call": "decode", "n": 63, "N": 1 << 26, "syn": 1},
        # long code, u16 syndromes kept for link statistics
        {"name": "decode 255 u16", "call": "decode", "n": 255, "N": 1 << 22, "syn": 2},
        # the benchmark's sweep: three streams in one call
        {"name": "sweep 15+31+63", "call": "streams", "jobs": "15:16777216,31:16777216,63:16777216", "syn": 1},
        # the batched workload: 10,000 packets of 64 bit .. 4 Mbit
        {"name": "plan 10000", "call": "plan", "packets": 10_000, "min_bits": 64, "max_bits": PACKET_MAX_BITS,
         "table": 20, "syn": 1},
        # host buffers in and out (link-bound)
        {"name": "host 63", "call": "host", "n": 63, "N": 1 << 22, "syn": 1},
        # the paper's packets: M = 1600 bytes in t = 4 segments, 40,000 packets
        {"name": "short 3212", "call": "decode_short", "n": 3212, "N": 160_000, "syn": 2},
        # (64,57) with double-error detection: a memory's or a link's word
        {"name": "secded 63", "call": "decode_secded", "n": 63, "N": 1 << 24, "syn": 1},
        # the transmitter of the sweep's longest code
        {"name": "encode 63x2^24", "call": "encode", "n": 63, "N": 1 << 24, "syn": 0},
        # the transmitter of the paper's packets: M = 800 bytes, t = 2, odd count
        {"name": "encode short 3212", "call": "encode_short", "n": 3212, "N": 40_001, "syn": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A call of the same kinds; its stream has 4 Kbit .. 1 Gbit."""
    call = rng.choice(["decode", "decode", "decode", "streams", "plan", "batch", "host", "decode_short",
                       "decode_short", "decode_secded", "encode", "encode_short", "encode_secded"])
    if call == "streams":
        jobs = []
        for _ in range(rng.randint(2, 6)):
            n = rng.choice(LENGTHS[1:])
            jobs.append("%d:%d" % (n, max(1, _log_int(rng, 1 << 12, 1 << 28) // n)))
        return {"call": call, "jobs": ",".join(jobs), "syn": rng.choice([0, 1, 2])}
    if call in ("plan", "batch"):
        return {"call": call, "packets": _log_int(rng, 8, 5000), "min_bits": 64,
                "max_bits": _log_int(rng, 1 << 12, PACKET_MAX_BITS), "table": rng.randrange(1 << 20),
                "syn": rng.choice([0, 1, 2])}
    bits = _log_int(rng, 1 << 12, 1 << (27 if call == "host" else 30))
    if call in ("decode_short", "encode_short"):
        n = _log_int(rng, 16, 32767)
        return {"call": call, "n": n, "N": max(1, bits // n),
                "syn": rng.choice([0, 2]) if call == "decode_short" else 0}
    n = rng.choice(LENGTHS)
    syn = 0
    if call == "decode_secded":
        syn = rng.choice([0, 2] if n == 255 else [0, 1, 2])
    elif call in ("decode", "host"):
        syn = rng.choice([0, 1, 2])
    return {"call": call, "n": n, "N": max(1, bits // n), "syn": syn}


# --------------------------------------------------------------------------
# the streams of a case and where they lie in its arenas
# --------------------------------------------------------------------------
def _is_short(case):
    return case["call"].endswith("_short")


def _is_secded(case):
    return case["call"].endswith("_secded")


def _is_encode(case):
    return case["call"].startswith("encode")


def _code(case, n):
    """(bits of a codeword, data bits) of length n under the case's code."""
    if _is_short(case):
        r, k = hd.hd_short_params(n)
        return n, k
    m, k = hd.code_params(n)
    return n + (1 if _is_secded(case) else 0), k


def _streams(case):
    """(n, N) of every stream."""
    if case["call"] == "streams":
        return [tuple(int(x) for x in j.split(":")) for j in case["jobs"].split(",")]
    if case["call"] in ("plan", "batch"):
        return [(p.n, p.num_codewords)
                for p in synth.packet_table(case["table"], case["packets"], case["min_bits"], case["max_bits"])]
    return [(case["n"], case["N"])]


class _Layout:
    """Word (and syndrome element) offsets of the streams, each on a 16-byte
    boundary, and the arenas' sizes."""

    def __init__(self, case):
        self.rows = []  # n, N, L, k, input word, data word, syndrome element
        iw = dw = sy = 0
        for n, N in _streams(case):
            L, k = _code(case, n)
            self.rows.append((n, N, L, k, iw, dw, sy))
            iw += (hd.words_for(N * L) + 3) // 4 * 4
            dw += (hd.words_for(N * k) + 3) // 4 * 4
            sy += (N + 15) // 16 * 16
        if len(self.rows) == 1:  # a single stream's buffers have their own sizes
            n, N, L, k = self.rows[0][:4]
            iw, dw, sy = hd.words_for(N * L), hd.words_for(N * k), N
        self.in_words, self.data_words, self.syn_elems = iw, dw, sy


def work(case):
    total = 0.0
    for n, N, L, k, *_ in _Layout(case).rows:
        total += N * (L + k) / 8.0 + N * case["syn"]
    return {"bytes": total, "flops": 0.0}


def _words(count, gen):
    return torch.randint(-(1 << 31), 1 << 31, (count,), dtype=torch.int32, device="cuda", generator=gen)


def _inject_errors(words, lay, gen):
    """Flip one bit in about p1 of the codewords and two in about p2 of them."""
    dev = "cuda"
    N = torch.tensor([r[1] for r in lay.rows], dtype=torch.int64, device=dev)
    L = torch.tensor([r[2] for r in lay.rows], dtype=torch.int64, device=dev)
    base = torch.tensor([r[4] * 32 for r in lay.rows], dtype=torch.int64, device=dev)
    ends = torch.cumsum(N, 0)
    total = sum(r[1] for r in lay.rows)
    p1, p2 = (0.05, 0.005) if max(r[0] for r in lay.rows) > 63 else (0.1, 0.01)
    singles = torch.randint(0, total, (max(1, int(p1 * total)),), device=dev, generator=gen)
    doubles = torch.randint(0, total, (int(p2 * total),), device=dev, generator=gen)
    cw = torch.cat([singles, doubles, doubles])
    row = torch.searchsorted(ends, cw, right=True)
    pos = (torch.rand(cw.shape, device=dev, generator=gen, dtype=torch.float64) * L[row]).to(torch.int64)
    bit = torch.unique(base[row] + (cw - (ends - N)[row]) * L[row] + pos)
    flips = torch.zeros_like(words)
    flips.index_add_(0, bit >> 5, torch.ones_like(bit).bitwise_left_shift_(bit & 31).to(torch.int32))
    words.bitwise_xor_(flips)


_ENCODE = {"plain": lambda d, n, N, s, st: hd.hd_encode(d, n, N, s, st),
           "short": lambda d, n, N, s, st: hd.hd_encode_short(d, n, N, s, st),
           "secded": lambda d, n, N, s, st: hd.hd_encode_secded(d, n, N, s, st)}


def _inputs(case, seed, lay):
    """The messages of an encode case, the received words of the others."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    data = _words(lay.data_words, gen)
    if _is_encode(case):
        return data
    words = torch.zeros(lay.in_words, dtype=torch.int32, device="cuda")
    encode = _ENCODE["short" if _is_short(case) else "secded" if _is_secded(case) else "plain"]
    st = torch.cuda.current_stream().cuda_stream
    for n, N, L, k, iw, dw, sy in lay.rows:
        hd.check(encode(data.data_ptr() + 4 * dw, n, N, words.data_ptr() + 4 * iw, st), "encode")
    _inject_errors(words, lay, gen)
    return words


class _State:
    pass


def prepare(case, seed):
    lay = _Layout(case)
    s = _State()
    s.case, s.lay = case, lay
    s.words = _inputs(case, seed, lay)
    syn_t = {0: None, 1: torch.uint8, 2: torch.int16}[case["syn"]]
    call = case["call"]
    if _is_encode(case):
        s.out = torch.empty(lay.in_words, dtype=torch.int32, device="cuda")
        return s
    if call == "host":
        s.words = s.words.cpu().pin_memory()
        s.out = torch.empty(lay.data_words, dtype=torch.int32, pin_memory=True)
        s.syn = None if syn_t is None else torch.empty(lay.syn_elems, dtype=syn_t, pin_memory=True)
        return s
    s.out = torch.zeros(lay.data_words, dtype=torch.int32, device="cuda")  # the gaps between packets stay 0
    s.syn = None if syn_t is None else torch.zeros(lay.syn_elems, dtype=syn_t, device="cuda")
    s.count = torch.zeros(2 if call in ("decode_short", "decode_secded") else len(lay.rows), dtype=torch.int64,
                          device="cuda")
    syn_b = 0 if s.syn is None else s.syn.data_ptr()
    if call == "streams":
        s.jobs = hd.stream_jobs([(s.words.data_ptr() + 4 * iw, n, N, s.out.data_ptr() + 4 * dw,
                                  syn_b + sy * case["syn"] if syn_b else None, case["syn"],
                                  s.count.data_ptr() + 8 * i)
                                 for i, (n, N, L, k, iw, dw, sy) in enumerate(lay.rows)])
    elif call in ("plan", "batch"):
        rows = [(s.words[iw:], s.out[dw:], None if s.syn is None else s.syn[sy:], N, n, case["syn"])
                for n, N, L, k, iw, dw, sy in lay.rows]
        if call == "plan":
            s.plan = hd.Plan(rows)
        else:
            s.table = hd.packet_table([(a.data_ptr(), b.data_ptr(), None if c is None else c.data_ptr(), N, n, st)
                                       for a, b, c, N, n, st in rows])
    elif call == "decode_short":
        s.plan = hd.ShortPlan(case["n"])
    return s


def run(s):
    case, call = s.case, s.case["call"]
    if call == "decode":
        hd.decode(s.words, case["n"], case["N"], case["syn"], out=s.out, syndromes=s.syn, err_count=s.count)
    elif call == "decode_short":
        s.plan.decode(s.words, case["N"], case["syn"], out=s.out, syndromes=s.syn, counts=s.count)
    elif call == "decode_secded":
        hd.decode_secded(s.words, case["n"], case["N"], case["syn"], out=s.out, syndromes=s.syn, counts=s.count)
    elif call == "streams":
        hd.check(hd.hd_decode_streams(s.jobs, len(s.lay.rows), torch.cuda.current_stream().cuda_stream), call)
    elif call == "plan":
        s.plan.launch(s.count)
    elif call == "batch":
        hd.check(hd.hd_decode_batch(s.table, len(s.lay.rows), s.count.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream), call)
    elif call == "host":
        out, syn, err = hd.decode_host(s.words, case["n"], case["N"], case["syn"], out=s.out, syndromes=s.syn)
        return {"out": out, "count": err} if syn is None else {"out": out, "syn": syn, "count": err}
    elif call == "encode":
        return {"stream": hd.encode(s.words, case["n"], case["N"], out=s.out)}
    elif call == "encode_short":
        return {"stream": hd.encode_short(s.words, case["n"], case["N"], out=s.out)}
    else:
        return {"stream": hd.encode_secded(s.words, case["n"], case["N"], out=s.out)}
    return {"out": s.out, "count": s.count} if s.syn is None else {"out": s.out, "syn": s.syn, "count": s.count}


# --------------------------------------------------------------------------
# the same results in plain torch, a bit a value (every output is a whole number)
# --------------------------------------------------------------------------
def _unpack(words, count):
    sh = torch.arange(32, dtype=torch.int32, device=words.device)
    return ((words[:, None] >> sh) & 1).to(torch.uint8).reshape(-1)[:count]


def _pack(bits):
    pad = -bits.numel() % 32
    if pad:
        bits = torch.cat([bits, bits.new_zeros(pad)])
    sh = torch.arange(32, dtype=torch.int64, device=bits.device)
    return (bits.reshape(-1, 32).to(torch.int64) << sh).sum(1).to(torch.int32)


def _syndrome(bits, pos):
    s = torch.zeros(bits.shape[0], dtype=torch.int64, device=bits.device)
    for j in range(int(pos[-1]).bit_length()):
        s |= (bits[:, ((pos >> j) & 1).bool()].sum(1) & 1).to(torch.int64) << j
    return s


def exact(case, seed):
    lay = _Layout(case)
    words, dev = _inputs(case, seed, lay), "cuda"
    secded, short, enc = _is_secded(case), _is_short(case), _is_encode(case)
    syn_t = {0: None, 1: torch.uint8, 2: torch.int16}[case["syn"]]
    out = torch.zeros(lay.in_words if enc else lay.data_words, dtype=torch.int32, device=dev)
    syn = None if syn_t is None else torch.zeros(lay.syn_elems, dtype=syn_t, device=dev)
    counts = []
    for n, N, L, k, iw, dw, sy in lay.rows:
        pos = torch.arange(0 if secded else 1, n + 1, device=dev)
        is_data = (pos & (pos - 1)) != 0
        src_b, dst_b, src_w, dst_w = (k, L, dw, iw) if enc else (L, k, iw, dw)
        step = max(32, (1 << 26) // max(L, 1) // 32 * 32)
        nonzero, detected = 0, 0
        for c0 in range(0, N, step):
            c = min(step, N - c0)
            w0 = src_w + c0 * src_b // 32
            bits = _unpack(words[w0:w0 + hd.words_for(c * src_b)], c * src_b).reshape(c, src_b)
            if enc:
                full = torch.zeros((c, L), dtype=torch.uint8, device=dev)
                full[:, is_data] = bits
                s = _syndrome(full, pos)
                for j in range(int(n).bit_length()):
                    full[:, (1 << j) - (0 if secded else 1)] = ((s >> j) & 1).to(torch.uint8)
                if secded:
                    full[:, 0] = (full.sum(1) & 1).to(torch.uint8)
                res = full
            else:
                s = _syndrome(bits, pos)
                value, flip = s, (s > 0) & (s <= n)
                odd = (bits.sum(1) & 1).to(torch.int64) if secded else None
                if secded:
                    value, flip = s | (odd << int(n).bit_length()), odd == 1
                    detected += int(((odd == 0) & (s != 0)).sum())
                elif short:
                    detected += int((s > n).sum())
                nonzero += int((value != 0).sum())
                rows = flip.nonzero().squeeze(1)
                bits[rows, s[rows] - (0 if secded else 1)] ^= 1
                res = bits[:, is_data]
                if syn is not None:
                    syn[sy + c0:sy + c0 + c] = value.to(syn_t)
            packed = _pack(res.reshape(-1))
            o = dst_w + c0 * dst_b // 32
            out[o:o + packed.numel()] = packed
        counts += [nonzero, detected] if secded or short else [nonzero]
    if enc:
        return {"stream": out}
    if case["call"] == "host":
        count = counts[0]
    else:
        count = torch.tensor(counts, dtype=torch.int64, device=dev)
    return {"out": out, "count": count} if syn is None else {"out": out, "syn": syn, "count": count}
