"""The work this library is given, as cases that a timing harness can run one pass at a time.

Every case goes through the public binding as a serving program would: the shape, the rule, the mask blob, the
scratch buffers and the outputs are made once and kept, and one pass is the calls a program makes for one layer of
one request batch.  Kinds:

  prefill  masks built from Q and K, then masked attention over the whole prompt(s)
  chunk    masked attention of the next rows of a prompt whose masks exist (chunked prefill)
  decode   one new token per sequence against a KV cache, keys chosen by the stored patterns
  capture  masks from the average map of several samples: maps of a batch, sums, average, rule, masked attention
  host     a prompt that lies in pinned host memory, results back to the host

Inputs carry the structure the method is made for (sink, local band, vertical stripes; see synth.make_sequence),
drawn per sequence and head from the seed.
"""
import math
import random

import torch

from paper_2506_11104_b200 import binding as dam
from paper_2506_11104_b200 import synth

DEVICE = "cuda:0"
DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}
BAND_HARMONICS = (0, 2, 3, 4, 6, 8, 12, 16, 24, 40)      # 0: no band; few harmonics: a wide band


def _case(name, kind, lengths, pcl, heads=32, kv_heads=8, dim=128, dtype="bf16", gather=True, tau=0.05, rows=0,
          samples=0):
    """`lengths`: tokens of every sequence (decode: the tokens its cache holds; capture: of the prompts that the masks
    are for); `rows`: rows a chunk adds to every sequence; `samples`: prompts of pcl tokens that a capture averages."""
    return {"name": name, "kind": kind, "lengths": " ".join(str(n) for n in lengths), "pcl": pcl, "heads": heads,
            "kv_heads": kv_heads, "dim": dim, "dtype": dtype, "gather": gather, "tau": tau, "rows": rows,
            "samples": samples}


def listed():
    return [
        # the smallest model anyone runs this on: two fp32 heads, a short prompt; launches and latency
        _case("prefill_tiny_fp32", "prefill", [512], 128, heads=2, kv_heads=2, dim=64, dtype="fp32", gather=False, tau=0.1),
        # a short chat prompt of an odd length, with the window the paper uses (512 tokens)
        _case("prefill_1k", "prefill", [1237], 512),
        # one layer of an ordinary long prompt
        _case("prefill_8k", "prefill", [8192], 1024),
        # one layer of the 32-layer stack at 32k tokens, the benchmark's default workload
        _case("prefill_32k", "prefill", [32768], 2048),
        # the longest context: stresses the work list and the mask emission
        _case("prefill_128k", "prefill", [131072], 4096),
        # requests of mixed and odd lengths packed into one batch
        _case("prefill_varlen", "prefill", [4096, 16384, 777, 32768, 9001, 65536], 1024),
        # head dimension 64, fewer heads, an odd length, plain tile lists (no gathered-column tiles: the rule's default)
        _case("prefill_16k_d64", "prefill", [16001], 1024, heads=16, kv_heads=4, dim=64, gather=False),
        # chunked prefill: the next 2048 rows of a prompt that has reached 24k tokens
        _case("chunk_2k_of_32k", "chunk", [24576 + 2048], 2048, rows=2048),
        # generation for a single user
        _case("decode_1x8k", "decode", [8000], 1024),
        # generation for a full batch
        _case("decode_64x32k", "decode", [32768] * 64, 2048),
        # masks from the average map of eight samples
        _case("capture_8x512", "capture", [4096], 512, samples=8),
        # a prompt handed over in host memory
        _case("host_8k", "host", [8192], 1024),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("prefill", "prefill", "prefill", "prefill", "fp32", "chunk", "decode", "decode", "capture", "host"))
    heads, kv_heads = rng.choice(((32, 8), (32, 8), (16, 4), (8, 8), (24, 8), (8, 1)))
    dim = rng.choice((128, 128, 64))
    gather = rng.random() < 0.6
    pcl = rng.choice((512, 1024, 2048, 4096))
    if kind == "prefill":
        total = _log_uniform(rng, 256, 98304 if gather else 57344)      # plain tile lists are longer
        n = rng.choice((1, 1, 2, 3, 5))
        cuts = sorted(rng.randrange(1, total) for _ in range(n - 1))
        lengths = [b - a for a, b in zip([0] + cuts, cuts + [total])]
        return _drawn("prefill", lengths, pcl, heads, kv_heads, dim, gather=gather)
    if kind == "fp32":
        return _drawn("prefill", [_log_uniform(rng, 200, 1500)], rng.choice((100, 128, 256)), rng.choice((2, 4)), 2, 64,
                      dtype="fp32", gather=False, tau=0.1)
    if kind == "chunk":
        rows = 256 * _log_uniform(rng, 1, 16)
        return _drawn("chunk", [256 * _log_uniform(rng, 4, 384) + rows], min(pcl, 1024), heads, kv_heads, dim,
                      gather=gather, rows=rows)
    if kind == "decode":
        n = _log_uniform(rng, 1, 64)
        return _drawn("decode", [_log_uniform(rng, 1500, 32768) for _ in range(n)], min(pcl, 2048), heads, kv_heads, dim,
                      gather=False)
    if kind == "capture":
        return _drawn("capture", [_log_uniform(rng, 1000, 8192)], rng.choice((256, 400, 512)), heads, kv_heads, dim,
                      gather=gather, samples=rng.randint(2, 8))
    return _drawn("host", [_log_uniform(rng, 2000, 8192)], min(pcl, 1024), heads, kv_heads, dim, gather=gather)


def _drawn(kind, lengths, *args, **kwargs):
    case = _case("", kind, lengths, *args, **kwargs)
    del case["name"]
    return case


def _lengths(case):
    return [int(n) for n in case["lengths"].split()]


def _cu(lengths):
    cu = [0]
    for n in lengths:
        cu.append(cu[-1] + n)
    return cu


def _plans(rng, heads, window):
    """What each head of one sequence attends to: a band, a sink, a few stripe columns (mostly few, sometimes many)."""
    plans = []
    for _ in range(heads):
        count = int(rng.random() ** 2 * 33)
        stripes = sorted(rng.randrange(1, max(2, window)) for _ in range(count))
        plans.append(synth.HeadPlan(sink=rng.random() < 0.85, band_m=rng.choice(BAND_HARMONICS), stripes=stripes))
    return plans


def _sequences(lengths, case, words):
    """Packed Q, K, V of the given lengths, every sequence and head with its own plan."""
    heads, kv, d, dtype = case["heads"], case["kv_heads"], case["dim"], DTYPES[case["dtype"]]
    amp = 8.0 if case["dtype"] == "fp32" else 10.0
    T = sum(lengths)
    Q = torch.empty(T, heads, d, dtype=dtype, device=DEVICE)
    K = torch.empty(T, kv, d, dtype=dtype, device=DEVICE)
    V = torch.empty(T, kv, d, dtype=dtype, device=DEVICE)
    at = 0
    for b, n in enumerate(lengths):
        window = min(n, case["pcl"])
        rng = random.Random("%s/%d" % (words, b))
        q, k, v = synth.make_sequence(n, heads, kv, d, window, _plans(rng, heads, window), amp, list(words) + [b], DEVICE)
        Q[at:at + n], K[at:at + n], V[at:at + n] = q, k, v
        at += n
    return Q, K, V


def _shape(lengths, case):
    return dam.make_shape(_cu(lengths), case["heads"], case["kv_heads"], case["dim"], DTYPES[case["dtype"]], DEVICE)


def _bytes_buffer(n):
    return torch.empty(max(256, n), dtype=torch.uint8, device=DEVICE)


def _buffers(s, shape, rule, like):
    """Mask blob, scratch buffers and outputs for `shape`, kept by the program."""
    mask, build, attn = dam.dam_mask_sizes(shape, rule)
    s["mask"], s["build_scratch"], s["attn_scratch"] = _bytes_buffer(mask), _bytes_buffer(build), _bytes_buffer(attn)
    s["O"] = torch.zeros_like(like)
    s["lse"] = torch.zeros(shape.c.num_q_heads, shape.c.total_tokens, dtype=torch.float32, device=DEVICE)


def prepare(case, seed):
    lengths, kind = _lengths(case), case["kind"]
    rule = dam.make_rule(case["pcl"], case["tau"], 0.8, gather_columns=case["gather"])
    s = {"kind": kind, "rule": rule}
    if kind == "decode":
        return _prepare_decode(s, case, seed, lengths)
    s["shape"] = shape = _shape(lengths, case)
    s["Q"], s["K"], s["V"] = Q, K, V = _sequences(lengths, case, [seed, 1])
    if kind == "host":
        s["Q"], s["K"], s["V"] = (x.cpu().pin_memory() for x in (Q, K, V))
        s["O"] = torch.zeros(Q.shape, dtype=Q.dtype).pin_memory()
        s["lse"] = torch.zeros(shape.c.num_q_heads, shape.c.total_tokens, dtype=torch.float32).pin_memory()
        s["workspace"] = _bytes_buffer(dam.dam_prefill_host(s["Q"], s["K"], s["V"], shape, rule, s["O"], s["lse"], None,
                                                            torch.device(DEVICE)))
        return s
    _buffers(s, shape, rule, Q)
    if kind == "chunk":
        # the blob was built when the prompt's window had been computed
        dam.dam_build_masks(Q, K, shape, rule, s["mask"], s["build_scratch"])
        s["ranges"] = [(n - case["rows"], n) for n in lengths]
    elif kind == "capture":
        pcl, heads = case["pcl"], case["heads"]
        sample_lengths = [pcl] * case["samples"]
        s["sample_Q"], s["sample_K"], _ = _sequences(sample_lengths, case, [seed, 2])
        s["sample_shape"] = _shape(sample_lengths, case)
        mask, build, _ = dam.dam_mask_sizes(s["sample_shape"], rule)
        s["sample_mask"], s["sample_scratch"] = _bytes_buffer(mask), _bytes_buffer(build)
        s["maps"] = torch.empty(case["samples"] * heads * pcl * pcl, dtype=torch.float32, device=DEVICE)
        s["A"] = torch.zeros(heads, pcl, pcl, dtype=torch.float32, device=DEVICE)
        s["C"] = torch.zeros(pcl, dtype=torch.int32, device=DEVICE)
    return s


def _prepare_decode(s, case, seed, lengths):
    """A KV cache filled up to each sequence's position; its first tokens are the window the masks were built from."""
    kv, d, dtype = case["kv_heads"], case["dim"], DTYPES[case["dtype"]]
    windows = [min(n, case["pcl"]) for n in lengths]
    Q, K, V = _sequences(windows, case, [seed, 1])
    s["shape"] = _shape(lengths, case)
    s["mask"], _ = dam.dam_build_masks(Q, K, _shape(windows, case), s["rule"])
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    T = sum(lengths)
    s["K"] = torch.randn(T, kv, d, generator=gen, dtype=dtype, device=DEVICE)
    s["V"] = torch.randn(T, kv, d, generator=gen, dtype=dtype, device=DEVICE)
    rng, at, source, positions = random.Random(seed), 0, 0, []
    for n, w in zip(lengths, windows):
        s["K"][at:at + w], s["V"][at:at + w] = K[source:source + w], V[source:source + w]
        positions.append(rng.randrange(n // 2, n))
        at, source = at + n, source + w
    s["Q"] = torch.randn(len(lengths), case["heads"], d, generator=gen, dtype=dtype, device=DEVICE)
    s["positions"] = torch.tensor(positions, dtype=torch.int32, device=DEVICE)
    s["O"] = torch.zeros_like(s["Q"])
    s["lse"] = torch.zeros(len(lengths), case["heads"], dtype=torch.float32, device=DEVICE)
    s["attn_scratch"] = _bytes_buffer(256)
    return s


def run(s):
    kind, shape, rule = s["kind"], s["shape"], s["rule"]
    if kind == "decode":
        dam.dam_decode_attention(s["Q"], s["K"], s["V"], s["mask"], shape, s["positions"], O=s["O"], lse=s["lse"],
                                 scratch=s["attn_scratch"])
        return {"O": s["O"], "lse": s["lse"]}
    if kind == "host":
        dam.dam_prefill_host(s["Q"], s["K"], s["V"], shape, rule, s["O"], s["lse"], s["workspace"], torch.device(DEVICE))
        return {"O": s["O"], "lse": s["lse"]}
    if kind == "chunk":
        dam.dam_sparse_attention_rows(s["Q"], s["K"], s["V"], s["mask"], shape, s["ranges"], s["O"], s["lse"],
                                      scratch=s["attn_scratch"])
        return {"O": s["O"], "lse": s["lse"]}
    if kind == "capture":
        A, C = s["A"].zero_(), s["C"].zero_()
        dam.dam_build_masks(s["sample_Q"], s["sample_K"], s["sample_shape"], rule, s["sample_mask"], s["sample_scratch"],
                            scores_dump=s["maps"])
        dam.dam_capture_accumulate(s["maps"], s["sample_shape"], rule.pcl_max, A, C)
        P = dam.dam_capture_average(A, C, rule.pcl_max, rule.eps, shape)
        dam.dam_build_masks_from_scores(P, shape, rule, s["mask"], s["build_scratch"])
    else:
        dam.dam_build_masks(s["Q"], s["K"], shape, rule, s["mask"], s["build_scratch"])
    dam.dam_sparse_attention(s["Q"], s["K"], s["V"], s["mask"], shape, True, 0.0, s["O"], s["lse"], s["attn_scratch"])
    out = {"O": s["O"], "lse": s["lse"]}
    if kind == "capture":
        out.update(A=A, C=C, P=P)
    return out


def _kept_per_row(case, window):
    """Keys a row of one head keeps, on average over these plans (dam_mask_stats: 0.11 - 0.26 of the window, 0.46 under
    the fp32 case's threshold and after averaging several samples); a decode step reads the union over the heads of a
    group, about twice that."""
    return (0.45 if case["kind"] == "capture" or case["dtype"] == "fp32" else 0.2) * window


def work(case):
    lengths, pcl, heads, kv, d = _lengths(case), case["pcl"], case["heads"], case["kv_heads"], case["dim"]
    item = 2 if case["dtype"] == "bf16" else 4
    kind = case["kind"]
    if kind == "decode":
        keys = sum(_kept_per_row(case, min(n, pcl)) for n in lengths)
        union = keys * (1.0 if heads == kv else 2.0)
        return {"bytes": union * kv * 2 * d * item + len(lengths) * heads * (2 * d * item + 4), "flops": keys * heads * 4 * d}
    attend = [(min(n, case["rows"]) if kind == "chunk" else n, min(n, pcl)) for n in lengths]
    rows = sum(n for n, _ in attend)
    flops = sum(n * _kept_per_row(case, L) for n, L in attend) * heads * 4 * d
    read = rows * (heads + 2 * kv) * d * item
    if kind == "chunk":                                     # the columns below the band come from the window
        read += sum(L for _, L in attend) * 2 * kv * d * item
    out = rows * heads * (d * item + 4)
    if kind == "capture":
        maps = heads * pcl * pcl * 4
        flops += case["samples"] * heads * pcl * pcl * d
        read += case["samples"] * pcl * (heads + kv) * d * item
        out += 2 * maps
    elif kind != "chunk":
        flops += sum(L * L for _, L in attend) * heads * d   # the window's map
    return {"bytes": read + out, "flops": flops}


def tolerance(case):
    # measured against float64 attention under the same masks: bf16 rel 2.0e-3 - 2.3e-3, max 1.0e-2 - 1.7e-2 (P and O are
    # rounded to bf16); fp32 rel 1.3e-6, max 1.2e-5.  The bf16 "max" leaves room for a cell of the window that sits on
    # the threshold to within the rounding of the softmax sums (one key of weight p* more or less in that row).
    if case["dtype"] == "fp32":
        return {"rel": 5e-6, "max": 5e-5}
    return {"rel": 8e-3, "max": 0.1}
