"""Timed cases of the library: decode attention, decode steps and cache builds, through ``binding``.

The shapes are those of the five workloads in ``synth.py`` (a single head; a 22-layer Llama-1.1B-shaped decoder
with 32 query / 4 KV heads and head_dim 64; ragged paged batches; a 32 / 8-head, head_dim 128 long-context sweep)
from one short sequence up to 32 sequences of 32 768 tokens.  Kinds of case:

  decode   one decode-attention call over a cache that is already there (one layer)
  step     one decode step of one layer (append the new token and attend), launched from Python
  layers   the decode steps of all layers of one token; ``graph`` = recorded once in a CUDA graph and replayed, as a
           serving loop does, otherwise launched call by call; ``host`` = activations in pinned host memory
  fill     bulk build of a cache from the keys and values of a prompt

Every step case takes the sequence lengths back to where they were first, as a program does that drops a rejected
token, so that a pass can be repeated: one small copy for all layers.
"""
import math

import numpy as np
import torch

from paper_2609_09208_b200 import binding as sa
from paper_2609_09208_b200 import synth

LAYERS = synth.LLAMA_1B_LAYERS
FP16 = sa.SA_KV_FP16


def _case(kind, code, *, dense=False, hadamard=False, outliers=True, d=64, q_heads=32, kv_heads=4, batch=1, tokens=1024,
          shortest=0, layers=1, graph=False, host=False, **more):
    """tokens: length of every sequence, or the longest of a ragged batch whose shortest is `shortest` (0: all equal).
    dense: the sub-byte container of the code (two PoT-4 codes per byte, bit planes for PoT-M1 / M2)."""
    return dict(more, kind=kind, code=code, dense=dense, hadamard=hadamard, outliers=outliers, d=d, q_heads=q_heads,
                kv_heads=kv_heads, batch=batch, tokens=tokens, shortest=shortest, layers=layers, graph=graph, host=host)


def listed():
    return [
        # the smallest call there is: one head over a short context (latency and launches)
        _case("decode", sa.SA_POT4, outliers=False, q_heads=1, kv_heads=1, tokens=1024, name="single_head_1k"),
        # a token of the 22-layer model at a chat-length context, called layer by layer from Python
        _case("layers", sa.SA_POTM1, tokens=4096, layers=LAYERS, name="llama_eager_4k"),
        # the same model at a long context in a serving loop: the benchmark's step
        _case("layers", sa.SA_POTM4, outliers=False, tokens=32768, layers=LAYERS, graph=True, name="llama_graph_32k"),
        # activations produced on the host: small batch, short context, 4-bit cache
        _case("layers", sa.SA_POT4, dense=True, tokens=2048, batch=4, layers=LAYERS, graph=True, host=True, name="llama_host_b4_2k"),
        # 4-bit rotated keys, a medium batch
        _case("decode", sa.SA_POT4, dense=True, hadamard=True, batch=8, tokens=32768, name="pot4_rotated_b8_32k"),
        # continuous batching: 16 sequences of mixed lengths take one step
        _case("step", sa.SA_POTM2, batch=16, tokens=16384, shortest=2048, name="ragged_b16"),
        # one very long document, head_dim 128, the dense 5-bit cache
        _case("decode", sa.SA_POTM1, dense=True, d=128, kv_heads=8, tokens=131072, name="long_d128_128k"),
        # head_dim 128, a large batch of ordinary contexts, 8-bit codes
        _case("decode", sa.SA_POTM4, d=128, kv_heads=8, batch=32, tokens=4096, name="d128_b32_4k"),
        # the largest: 32 sequences of 32k tokens
        _case("decode", sa.SA_POTM4, outliers=False, batch=32, tokens=32768, name="b32_32k"),
        # every query head with its own KV head, a length that fills no page
        _case("decode", sa.SA_POTM2, dense=True, d=128, q_heads=16, kv_heads=16, batch=3, tokens=5001, name="no_gqa_b3_5001"),
        # the unquantised cache
        _case("decode", FP16, batch=8, tokens=16383, name="fp16_b8_16383"),
        # prompts of four sequences into the cache
        _case("fill", sa.SA_POTM4, batch=4, tokens=8192, shortest=1000, name="fill_b4_8k"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "decode", "step", "layers", "layers", "fill"])
    code, dense = rng.choice([(sa.SA_POT4, False), (sa.SA_POT4, True), (sa.SA_POTM1, False), (sa.SA_POTM1, True),
                              (sa.SA_POTM2, False), (sa.SA_POTM2, True), (sa.SA_POTM4, False), (sa.SA_POTM4, False),
                              (sa.SA_INT8, False), (FP16, False)])
    hadamard = code != FP16 and rng.random() < 0.25
    d, q_heads, kv_heads = rng.choice([(64, 32, 4), (64, 32, 4), (128, 32, 8), (64, 8, 2), (64, 1, 1), (128, 16, 16), (64, 32, 2)])
    batch = rng.choice([1, 1, 2, 3, 4, 8, 13, 16, 32])
    layers = LAYERS if kind == "layers" else 1
    if kind == "layers":
        d, q_heads, kv_heads = 64, 32, 4
        batch = min(batch, 4)
    # at most the cached keys of the largest listed case, a quarter of them where the cache holds binary16
    most = 32 * 32768 * 4 * 64 // (batch * kv_heads * d * layers * (2 if code == FP16 else 1))
    if kind == "fill":
        most //= 4
    tokens = _log_int(rng, 200, max(400, min(most, 131072 if batch == 1 else 32768)))
    shortest = max(1, tokens // rng.choice([2, 8])) if kind == "fill" and batch > 1 else 0      # prompts differ in length
    graph = kind == "layers" and rng.random() < 0.6
    return _case(kind, code, dense=dense, hadamard=hadamard, outliers=rng.random() < 0.7, d=d, q_heads=q_heads, kv_heads=kv_heads,
                 batch=batch, tokens=tokens, shortest=shortest, layers=layers, graph=graph, host=graph and rng.random() < 0.3)


def _lens(case):
    """Cached tokens per sequence: all equal, or spread evenly from the shortest to the longest in a mixed order.  (A
    fixed function of the case: work() has to know them.)"""
    B, T, lo = case["batch"], case["tokens"], case["shortest"]
    if not lo or B == 1:
        return np.full(B, T, dtype=np.int64)
    steps = np.linspace(lo, T, B).astype(np.int64)
    return steps[(np.arange(B) * 7 + 3) % B] if B % 7 else steps[::-1].copy()


def _normal(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)


def _keys_values(case, gen, n):
    """n tokens of binary16 keys and values: Gaussians, the keys with per-channel log-normal outlier scales."""
    H, d = case["kv_heads"], case["d"]
    K = _normal(gen, n, H, d)
    if case["outliers"]:
        K *= torch.exp(_normal(gen, 1, H, d))
    return K.half(), _normal(gen, n, H, d).half()


def _launch(s, l):
    """The library call of layer l."""
    case, c = s["case"], s["caches"][l]
    cfg, O = s["cfg"], s["O"][l]
    if case["host"]:
        sa.decode_step_host(cfg, c.handle, s["Q"][l], s["K"][l], s["V"][l], O, s["staging"], c.workspace)
    elif case["kind"] in ("step", "layers"):
        sa.decode_step(cfg, c.handle, s["Q"][l], s["K"][l], s["V"][l], O, c.workspace)
    elif case["code"] == FP16:
        sa.decode_attention_fp16(cfg, c.handle, s["Q"][l], O, c.workspace)
    else:
        sa.decode_attention(cfg, c.handle, s["Q"][l], O, c.workspace)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    B, Hq, Hkv, d = case["batch"], case["q_heads"], case["kv_heads"], case["d"]
    cfg = sa.make_config(d, Hq, Hkv, case["code"], nibble=case["dense"], hadamard=case["hadamard"])
    lens = _lens(case)
    cu = np.concatenate([[0], np.cumsum(lens)])
    step = case["kind"] in ("step", "layers")
    room = 64 if step else 0
    n_pages = int(np.maximum((lens + room + 63) // 64, 1).sum())
    s = dict(case=case, cfg=cfg, cu=cu, caches=[], Q=[], K=[], V=[], O=[])
    s["lens0"] = torch.from_numpy(lens.astype(np.int32)).cuda().repeat(case["layers"], 1)
    s["lens"] = s["lens0"].clone()
    for l in range(case["layers"]):
        c = sa.PagedCache(cfg, lens, "cuda", extra_tokens=room, permutation=synth.page_permutation(n_pages, seed + l))
        c.seq_lens = s["lens"][l]                     # one tensor for the lengths of all layers
        c.handle = sa.make_cache(c.pages, c.page_table, c.seq_lens, c.n_pages)
        K, V = _keys_values(case, gen, int(cu[-1]))
        if case["kind"] == "fill":
            s["K"].append(K)
            s["V"].append(V)
        else:
            sa.fill_kv(cfg, c.handle, K, V, cu)
            s["Q"].append(_normal(gen, B, Hq, d).half())
            s["O"].append(torch.zeros((B, Hq, d), dtype=torch.float32, device="cuda"))
        if step:
            K, V = _keys_values(case, gen, B)
            s["K"].append(K)
            s["V"].append(V)
        s["caches"].append(c)
    if case["host"]:
        for name in "QKVO":
            s[name] = [x.cpu().pin_memory() for x in s[name]]
        s["staging"] = torch.empty(sa.staging_bytes(cfg, B), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    if case["graph"]:
        for l in range(case["layers"]):               # every kernel has been loaded before the recording
            _launch(s, l)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            s["lens"].copy_(s["lens0"])
            for l in range(case["layers"]):
                _launch(s, l)
        torch.cuda.synchronize()
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "fill":
        c = s["caches"][0]
        sa.fill_kv(s["cfg"], c.handle, s["K"][0], s["V"][0], s["cu"])
        return c.pages
    if case["kind"] == "decode":
        _launch(s, 0)
        return s["O"][0]
    if case["graph"]:
        s["graph"].replay()
    else:
        s["lens"].copy_(s["lens0"])
        for l in range(case["layers"]):
            _launch(s, l)
    return {"O": s["O"], "lens": s["lens"], "pages": [c.pages for c in s["caches"]]}


def _bytes_per_key(case):
    """Bytes of one cached token of one KV head: key codes, 4 bytes of scales, values."""
    d, code = case["d"], case["code"]
    if code == FP16:
        return 4 * d
    bits = 4 + code if case["dense"] else 8
    return d * bits // 8 + 4 + d


def work(case):
    """Each cached key read once (fill: each prompt token read and its record written once), the step's new tokens read
    and written, queries read, outputs written; 4 operations per query head, key and dimension."""
    n, B, L, d = int(_lens(case).sum()), case["batch"], case["layers"], case["d"]
    Hq, Hkv, rec = case["q_heads"], case["kv_heads"], _bytes_per_key(case)
    if case["kind"] == "fill":
        return {"bytes": n * Hkv * (4 * d + rec), "flops": 0}
    per_layer = n * Hkv * rec + B * Hq * d * (2 + 4)
    if case["kind"] != "decode":
        per_layer += B * Hkv * (4 * d + rec)
        n += B
    return {"bytes": L * per_layer, "flops": L * 4 * n * Hq * d}


def tolerance(case):
    if case["kind"] == "fill":
        return "exact"
    # binary16 cache: the weights enter the product rounded to 11 bits; otherwise 32-bit sums of weights of 21 bits
    return {"rel": 5e-4} if case["code"] == FP16 else {"rel": 1e-5}
