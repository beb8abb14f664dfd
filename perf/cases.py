"""The work this library is used for, as a list of cases that can be timed and compared.

A prompt's K/V cache is compressed once per layer after the prompt phase (the whole-step calls),
and every generated token then attends to the compressed cache of that layer (the decode call).
One pass of a case is one such call for one layer, through the Python binding, the way a serving
program makes it: the outputs are fresh tensors (they become the layer's cache), the scratch
workspace that the call returns is handed to the next call.

listed()   the cases; draw(rng): one more of the same ranges
prepare    inputs of a case from a seed, on the GPU (on the host where the call takes host buffers)
run        one pass, returns the whole outputs
work       bytes and operations that the step cannot do without
tolerance  how far another correct implementation may be off
"""
from __future__ import annotations

import math
import random

import torch

from paper_2404_14469_b200 import binding as sk
from paper_2404_14469_b200 import synth

PAGE = 256  # positions per page of the paged cases


def _compress(name, B, heads, L, W, pool, kernel, budget, spans, heavy=False, store="dense",
              lse=False, grouped=False):
    Hq, Hkv, d = heads
    return {"name": name, "kind": "compress", "B": B, "Hq": Hq, "Hkv": Hkv, "d": d, "L": L, "W": W,
            "pool": pool, "kernel": kernel, "budget": budget, "spans": spans, "heavy": heavy,
            "store": store, "lse": lse, "grouped": grouped}


def _ragged(name, B, heads, Lmin, Lmax, mix, W, pool, kernel, budget, store, lse=False):
    Hq, Hkv, d = heads
    return {"name": name, "kind": "ragged", "B": B, "Hq": Hq, "Hkv": Hkv, "d": d, "Lmin": Lmin,
            "Lmax": Lmax, "mix": mix, "W": W, "pool": pool, "kernel": kernel, "budget": budget,
            "store": store, "lse": lse}


def _decode(name, B, heads, rows):
    Hq, Hc, d = heads
    return {"name": name, "kind": "decode", "B": B, "Hq": Hq, "Hc": Hc, "d": d, "rows": rows}


def _host(name, B, heads, L, W, pool, kernel, budget, spans):
    c = _compress(name, B, heads, L, W, pool, kernel, budget, spans)
    c["kind"] = "host"
    return c


MHA, GQA, TINY = (32, 32, 128), (32, 8, 128), (4, 4, 64)


def listed():
    return [
        # the smallest configuration (workload 0): a toy model or a unit test, launch latency only
        _compress("tiny-mha-1k", 1, TINY, 1024, 32, "max", 7, 256, 3),
        # a short prompt at the needle-test settings (window 16, kernel 5, budget 1024), odd length
        _compress("short-gqa-3k", 1, GQA, 3001, 16, "max", 5, 1024, -1),
        # an ordinary prompt: LongBench inputs average about 13K tokens (window 32, max pool 7)
        _compress("longbench-gqa-13k", 1, GQA, 13013, 32, "max", 7, 2048, -1),
        # workload 1: a 7B MHA model at 16K tokens
        _compress("lwm7b-mha-16k", 1, MHA, 16384, 32, "max", 7, 4096, -1),
        # workload 2, the benchmark's default: a batch of four 32K prompts, GQA, average pooling
        _compress("mistral7b-gqa-32k", 4, GQA, 32768, 32, "avg", 5, 4096, -1),
        # workload 3: one 128K prompt, window 64, heavy-tailed key norms, clusters at both edges
        _compress("mixtral-gqa-128k", 1, GQA, 131072, 64, "max", 7, 8192, 16, heavy=True),
        # workload 4, the longest: 380K tokens, MHA, one needle
        _compress("mha-380k-needle", 1, MHA, 380000, 32, "max", 7, 4096, 1),
        # a serving batch: prompts of very different lengths in a paged cache, the shortest of
        # them within the budget (copied through)
        _ragged("ragged-paged-8", 8, GQA, 600, 24000, 8, 32, "max", 7, 1024, "paged"),
        # the cache kept at Hkv heads, read from the framework's [B, L, Hkv, d] order, with the
        # window rows' log-sum-exp handed over by the prompt phase's attention kernel
        _compress("grouped-lse-20k", 2, GQA, 20011, 32, "max", 7, 2048, -1, store="blhd", lse=True,
                  grouped=True),
        # a generated token on the expanded cache of workload 2
        _decode("decode-expanded-4k", 4, MHA, 4096),
        # a generated token of a larger batch on a cache kept at Hkv heads, odd row count
        _decode("decode-gqa-1k", 8, GQA, 1057),
        # K and V held in (pinned) host memory: copies in, the step, copies out
        _host("host-gqa-8k", 1, GQA, 8192, 32, "max", 7, 2048, -1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# window, pooling and kernel size of the configurations in use
SETTINGS = [(32, "max", 7), (32, "max", 7), (32, "avg", 5), (16, "max", 5), (64, "max", 13), (64, "max", 7)]


def draw(rng: random.Random):
    """Another case: kinds, models, lengths (over their logarithm), batch sizes and options."""
    W, pool, kernel = rng.choice(SETTINGS)
    heads = rng.choice([MHA, GQA, GQA, GQA, TINY, (8, 2, 64)])
    pick = rng.random()
    if pick < 0.2:
        B, rows = _log_int(rng, 1, 16), _log_int(rng, 200, 8300)
        heads = rng.choice([MHA, GQA, GQA, (8, 2, 64)])
        while B * heads[1] * rows > 600_000:
            B = max(1, B // 2)
            rows = max(200, rows * 3 // 4)
        c = _decode("", B, heads, rows)
    elif pick < 0.4:
        B, Lmax = rng.randint(2, 16), _log_int(rng, 1500, 30000)
        heads = rng.choice([GQA, GQA, MHA, (8, 2, 64)])
        while B * heads[1] * Lmax > 2_500_000:
            B = max(2, B // 2)
            Lmax = Lmax * 3 // 4
        budget = rng.choice([512, 1024, 2048])
        c = _ragged("", B, heads, max(W + 100, Lmax // 30), Lmax, rng.randint(0, 10**6), W, pool, kernel,
                    budget, rng.choice(["paged", "paged", "packed", "padded"]), rng.random() < 0.3)
    elif pick < 0.48:
        L = _log_int(rng, 2000, 16000)
        c = _host("", 1, heads, L, W, pool, kernel, min(rng.choice([512, 1024, 2048]), L // 2), -1)
    else:
        B, L = rng.choice([1, 1, 1, 2, 3, 4]), _log_int(rng, 1000, 380000)
        while B * heads[1] * L > 2_500_000:
            B = max(1, B // 2)
            L = L * 3 // 4
        budget = min(rng.choice([256, 1024, 1024, 2048, 4096, 4096]), max(L // 2, W + 1))
        c = _compress("", B, heads, L, W, pool, kernel, budget, -1, heavy=rng.random() < 0.2,
                      store="blhd" if rng.random() < 0.25 else "dense", lse=rng.random() < 0.2,
                      grouped=heads[0] != heads[1] and rng.random() < 0.25)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _workload(case, B, L):
    n = L - case["W"]
    spans = case.get("spans", -1)
    if spans < 0:  # 1 % of the prefix positions lie in planted spans of eight keys
        spans = max(3, round(0.01 * n / synth.CLUSTER_LEN))
    heavy = case.get("heavy", False)
    return synth.Workload(9, "perf", B, case["Hq"], case["Hkv"], case["d"], L, case["W"], case["kernel"],
                          case["pool"], (case["budget"],), 1, spans, 0.5 if heavy else 0.0, heavy)


def _lengths(case):
    """Prompt lengths of a ragged batch: spread over their logarithm, the longest one Lmax."""
    rng = random.Random(case["mix"])
    lens = [_log_int(rng, case["Lmin"], case["Lmax"]) for _ in range(case["B"] - 1)] + [case["Lmax"]]
    rng.shuffle(lens)
    return lens


def _window_lse(q, k):
    """What the prompt phase's attention kernel keeps: log-sum-exp of every window row, fp32."""
    B, Hq, W, d = q.shape
    Hkv, L = k.shape[1], k.shape[2]
    g = Hq // Hkv
    out = torch.empty(B, Hq, W, dtype=torch.float32, device=q.device)
    seen = (torch.arange(L, device=q.device)[None, :]
            <= (L - W + torch.arange(W, device=q.device))[:, None]).repeat(g, 1)
    for b in range(B):
        for c in range(Hkv):
            rows = q[b, c * g:(c + 1) * g].reshape(g * W, d).float()
            logits = rows @ k[b, c].float().t() / math.sqrt(d)
            logits.masked_fill_(~seen, float("-inf"))
            out[b, c * g:(c + 1) * g] = torch.logsumexp(logits, dim=-1).view(g, W)
    return out


def _pages(parts, lens, seed):
    """One pool [pages, Hkv, PAGE, d] and a block table for sequences in `parts` ([1, Hkv, L, d])."""
    dev = parts[0].device
    counts = [-(-x // PAGE) for x in lens]
    order = torch.randperm(sum(counts) + 8, generator=torch.Generator().manual_seed(seed)).to(dev)
    Hkv, d = parts[0].shape[1], parts[0].shape[3]
    pool = torch.zeros(sum(counts) + 8, Hkv, PAGE, d, dtype=torch.bfloat16, device=dev)
    table = torch.zeros(len(lens), max(counts), dtype=torch.int32, device=dev)
    at = 0
    for b, (x, cnt) in enumerate(zip(parts, counts)):
        mine = order[at:at + cnt]
        whole = torch.zeros(Hkv, cnt * PAGE, d, dtype=torch.bfloat16, device=dev)
        whole[:, :lens[b]] = x[0]
        pool[mine] = whole.view(Hkv, cnt, PAGE, d).permute(1, 0, 2, 3)
        table[b, :cnt] = mine.to(torch.int32)
        at += cnt
    return pool, table


def _prepare_ragged(case, seed):
    lens = _lengths(case)
    seqs = [synth.make_layer(_workload(case, 1, x), seed + 1_000_003 * (b + 1), device="cuda")
            for b, x in enumerate(lens)]
    s = {"lens": lens, "q": torch.cat([x["q_obs"] for x in seqs]),
         "lse": torch.cat([_window_lse(x["q_obs"], x["k"]) for x in seqs]) if case["lse"] else None}
    ks, vs = [x["k"] for x in seqs], [x["v"] for x in seqs]
    if case["store"] == "paged":
        s["k"], s["table"] = _pages(ks, lens, seed)
        s["v"], _ = _pages(vs, lens, seed)
    elif case["store"] == "packed":  # [total tokens, Hkv, d]
        s["k"], s["v"] = (torch.cat([x[0].permute(1, 0, 2) for x in part]).contiguous() for part in (ks, vs))
        s["cu"] = [sum(lens[:b]) for b in range(len(lens))]
    else:                            # [B, Hkv, Lmax, d]
        for name, part in (("k", ks), ("v", vs)):
            s[name] = torch.zeros(case["B"], case["Hkv"], max(lens), case["d"], dtype=torch.bfloat16,
                                  device="cuda")
            for b, x in enumerate(part):
                s[name][b, :, :lens[b]] = x[0]
    return s


def prepare(case, seed):
    seed = int(seed)
    kind = case["kind"]
    if kind == "decode":
        x = synth.make_random(case["B"], case["Hq"], case["Hc"], case["rows"], case["d"], 1, seed=seed,
                              device="cuda", q_scale=2.0)
        s = {"q": x["q_obs"][:, :, 0].contiguous(), "k": x["k"], "v": x["v"]}
    elif kind == "ragged":
        s = _prepare_ragged(case, seed)
    else:
        x = synth.make_layer(_workload(case, case["B"], case["L"]), seed, device="cuda")
        s = {"q": x["q_obs"], "k": x["k"], "v": x["v"]}
        s["lse"] = _window_lse(s["q"], s["k"]) if case["lse"] else None
        if case["store"] == "blhd":  # stored [B, L, Hkv, d], seen as [B, Hkv, L, d]
            for t in ("k", "v"):
                s[t] = s[t].permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    if kind != "decode":
        s["pool"] = sk.POOL_MAX if case["pool"] == "max" else sk.POOL_AVG
    if kind == "host":
        B, Hq, d, W, budget = case["B"], case["Hq"], case["d"], case["W"], case["budget"]
        for t in ("q", "k", "v"):
            s[t] = torch.empty(s[t].shape, dtype=s[t].dtype, pin_memory=True).copy_(s[t])
        s["out_k"] = torch.empty(B, Hq, budget, d, dtype=torch.bfloat16, pin_memory=True)
        s["out_v"] = torch.empty(B, Hq, budget, d, dtype=torch.bfloat16, pin_memory=True)
        s["out_idx"] = torch.empty(B, Hq, budget - W, dtype=torch.int32, pin_memory=True)
        need = sk.snapkv_host_staging_size(B, Hq, case["Hkv"], case["L"], d, W, case["kernel"], s["pool"],
                                           budget)
        s["staging"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    s["case"] = case
    s["ws"] = None  # the first call allocates it, later calls get it back
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "decode":
        out, lse, s["ws"] = sk.snapkv_decode_attention(s["q"], s["k"], s["v"], s["ws"])
        return out, lse
    kernel, pool, budget = case["kernel"], s["pool"], case["budget"]
    if kind == "host":
        sk.snapkv_compress_host(s["q"], s["k"], s["v"], kernel, pool, budget, s["out_k"], s["out_v"],
                                s["out_idx"], s["staging"])
        return s["out_k"], s["out_v"], s["out_idx"]
    if kind == "ragged":
        if case["store"] == "paged":
            ok, ov, oi, s["ws"] = sk.snapkv_compress_paged(
                s["q"], s["k"], s["v"], s["table"], case["Lmax"], kernel, pool, budget, seq_lens=s["lens"],
                lse_obs=s["lse"], workspace=s["ws"])
        else:
            ok, ov, oi, s["ws"] = sk.snapkv_compress_varlen(
                s["q"], s["k"], s["v"], s["lens"], kernel, pool, budget, cu_seqlens=s.get("cu"),
                lse_obs=s["lse"], workspace=s["ws"])
        return ok, ov, oi
    ok, ov, oi, s["ws"] = sk.snapkv_compress(s["q"], s["k"], s["v"], kernel, pool, budget, workspace=s["ws"],
                                             lse_obs=s["lse"], grouped=case["grouped"])
    return ok, ov, oi


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Bytes: every key and every window query read once, the value rows that at least are selected
    (one set per KV head) read once, the compressed rows and the positions written once.  Operations:
    the window's logits, or a decode step's two matrix-vector products."""
    B, Hq, d = case["B"], case["Hq"], case["d"]
    if case["kind"] == "decode":
        cache = 2 * B * case["Hc"] * case["rows"] * d * 2
        return {"bytes": cache + B * Hq * d * 2 + B * Hq * (d + 1) * 4, "flops": 4 * B * Hq * case["rows"] * d}
    Hkv, W, budget = case["Hkv"], case["W"], case["budget"]
    Ho = Hkv if case.get("grouped") else Hq
    lens = _lengths(case) if case["kind"] == "ragged" else [case["L"]] * B
    nbytes = flops = 0
    for L in lens:
        rows = min(budget, L)
        nbytes += Hq * W * d * 2 + (Hq * W * 4 if case["lse"] else 0)
        nbytes += (Hkv * L * d * 2) + Hkv * rows * d * 2
        nbytes += 2 * Ho * rows * d * 2 + Ho * (rows - W) * 4
        if L > budget:
            flops += 2 * Hq * W * L * d
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "decode":
        return {"rel": 1e-5}  # bf16 products summed in fp32
    # The kept rows are byte copies; votes are fp32 sums, so where two pooled votes at the cut
    # are equal to rounding another correct implementation may keep the other position, and the
    # ascending list between the two is then shifted by one.
    return {"rel": 0.02, "max": 0.9, "differ": 0.005}
