"""GPU parity for batches of prompts of different lengths (snapkv_compress_varlen): every
sequence must come out as the oracle's single-sequence step on that sequence alone, for a padded
[B, Hkv, Lmax, d] cache and for a packed [total_tokens, Hkv, d] cache."""
import numpy as np
import pytest
import torch

from oracle import snapkv_oracle as orc
from paper_2404_14469_b200 import binding as sk
from paper_2404_14469_b200 import synth

import parity
from test_gpu_parity import PT, _bits

pytestmark = pytest.mark.gpu


def _sequences(lens, Hq, Hkv, d, W, kernel, ptype, budget, seed):
    """One seeded single-sequence layer per length (clusters planted as in the workloads)."""
    out = []
    for i, L in enumerate(lens):
        w = synth.Workload(80 + seed, "t", 1, Hq, Hkv, d, L, W, kernel, ptype, (budget,), 1, 2)
        out.append(synth.make_layer(w, 100 * seed + i))
    return out


def _check_sequence(b, seq, L, W, kernel, ptype, budget, out_k, out_v, out_idx, lse=None):
    q, k, v = (_bits(seq[x]) for x in ("q_obs", "k", "v"))
    ref = orc.compress(q, k, v, kernel, PT[ptype], budget, lse=lse)
    Hq, Hkv = q.shape[1], k.shape[1]
    g = Hq // Hkv
    rows = min(budget, L)
    ksel = rows - W
    idx = out_idx[b].cpu().numpy()
    ok, ov = _bits(out_k[b]), _bits(out_v[b])
    for h in range(Hq):
        if budget >= L:   # copied through; nothing beyond its rows is touched
            assert np.array_equal(idx[h, :ksel], np.arange(ksel)) and np.all(idx[h, ksel:] == -1)
            assert not ok[h, rows:].any() and not ov[h, rows:].any()
        else:
            parity.check_indices(idx[h], ref["pooled"][0, h], ksel, ref["out_idx"][0, h])
        parity.check_rows(ok[h, :rows], ov[h, :rows], k[0, h // g], v[0, h // g],
                          idx[h, :ksel].astype(np.int64), W)


@pytest.mark.parametrize("lens,Hq,Hkv,d,W,kernel,ptype,budget", [
    ([1000, 333, 2048, 129], 4, 2, 128, 32, 5, "avg", 200),     # 129 < budget: copied through
    ([700, 64, 1500], 8, 1, 64, 32, 7, "max", 256),             # 64 = 2 W, shorter than a tile
    ([900, 50000], 2, 2, 64, 16, 7, "max", 512),                # a long row next to a short one
])
def test_padded_batch_matches_per_sequence_oracle(lens, Hq, Hkv, d, W, kernel, ptype, budget):
    seqs = _sequences(lens, Hq, Hkv, d, W, kernel, ptype, budget, seed=1)
    B, Lmax = len(lens), max(lens)
    k = torch.full((B, Hkv, Lmax, d), float("nan"), dtype=torch.bfloat16)   # padding must not be read
    v = torch.full((B, Hkv, Lmax, d), float("nan"), dtype=torch.bfloat16)
    for b, s in enumerate(seqs):
        k[b, :, :lens[b]] = s["k"][0]
        v[b, :, :lens[b]] = s["v"][0]
    q = torch.cat([s["q_obs"] for s in seqs])
    out_k, out_v, out_idx, ws = sk.snapkv_compress_varlen(q.cuda(), k.cuda(), v.cuda(), lens, kernel,
                                                          PT[ptype], budget)
    code, detail = sk.snapkv_device_status(ws)
    assert code == sk.OK, (code, detail)
    for b, s in enumerate(seqs):
        _check_sequence(b, s, lens[b], W, kernel, ptype, budget, out_k, out_v, out_idx)


def test_packed_cache_with_supplied_lse_matches_per_sequence_oracle():
    lens, Hq, Hkv, d, W, kernel, budget = [640, 1111, 200], 8, 2, 128, 32, 7, 300
    seqs = _sequences(lens, Hq, Hkv, d, W, kernel, "max", budget, seed=2)
    cu = [0, 640, 640 + 1111]
    k = torch.cat([s["k"][0].permute(1, 0, 2) for s in seqs]).contiguous()      # [T, Hkv, d]
    v = torch.cat([s["v"][0].permute(1, 0, 2) for s in seqs]).contiguous()
    q = torch.cat([s["q_obs"] for s in seqs])
    lses = [orc.lse_obs(_bits(s["q_obs"]), _bits(s["k"])).astype(np.float32) for s in seqs]
    lse = torch.from_numpy(np.concatenate(lses)).cuda()
    for use_lse in (False, True):
        out_k, out_v, out_idx, ws = sk.snapkv_compress_varlen(
            q.cuda(), k.cuda(), v.cuda(), lens, kernel, sk.POOL_MAX, budget, cu_seqlens=cu,
            lse_obs=lse if use_lse else None)
        code, detail = sk.snapkv_device_status(ws)
        assert code == sk.OK, (code, detail)
        for b, s in enumerate(seqs):
            _check_sequence(b, s, lens[b], W, kernel, "max", budget, out_k, out_v, out_idx,
                            lse=lses[b].astype(np.float64) if use_lse else None)


@pytest.mark.parametrize("use_lse", [False, True])
def test_status_block_is_clean_whichever_path_the_first_sequence_takes(use_lse):
    # first sequence shorter than the budget (copied through), second one compressed; the
    # workspace arrives full of 0xFF, as memory that was never cleared may
    lens, Hq, Hkv, d, W, kernel, budget = [129, 1000], 4, 2, 128, 32, 5, 200
    seqs = _sequences(lens, Hq, Hkv, d, W, kernel, "avg", budget, seed=3)
    B, Lmax = len(lens), max(lens)
    k = torch.zeros(B, Hkv, Lmax, d, dtype=torch.bfloat16)
    v = torch.zeros(B, Hkv, Lmax, d, dtype=torch.bfloat16)
    for b, s in enumerate(seqs):
        k[b, :, :lens[b]] = s["k"][0]
        v[b, :, :lens[b]] = s["v"][0]
    q = torch.cat([s["q_obs"] for s in seqs])
    lses = [orc.lse_obs(_bits(s["q_obs"]), _bits(s["k"])).astype(np.float32) for s in seqs]
    lse = torch.from_numpy(np.concatenate(lses)).cuda() if use_lse else None
    need = sk.snapkv_workspace_size(1, Hq, Hkv, Lmax, d, W, kernel, sk.POOL_AVG, budget)
    ws = torch.full((need,), 0xFF, dtype=torch.uint8, device="cuda")
    out_k, out_v, out_idx, ws2 = sk.snapkv_compress_varlen(q.cuda(), k.cuda(), v.cuda(), lens, kernel,
                                                           sk.POOL_AVG, budget, lse_obs=lse, workspace=ws)
    assert ws2 is ws
    assert sk.snapkv_device_status(ws) == (sk.OK, 0)
    for b, s in enumerate(seqs):
        _check_sequence(b, s, lens[b], W, kernel, "avg", budget, out_k, out_v, out_idx,
                        lse=lses[b].astype(np.float64) if use_lse else None)
    # the same for a plain call that only copies the cache through
    ws.fill_(0xFF)
    dev = {x: seqs[0][x].cuda() for x in ("q_obs", "k", "v")}
    sk.snapkv_compress(dev["q_obs"], dev["k"], dev["v"], kernel, sk.POOL_AVG, budget, workspace=ws)
    assert sk.snapkv_device_status(ws) == (sk.OK, 0)


@pytest.mark.parametrize("lens,Hq,Hkv,d,W,kernel,ptype,budget,use_lse", [
    ([300, 5000, 129, 2049, 700, 17], 8, 2, 128, 16, 5, "max", 200, False),   # copied through in between
    ([1500] * 3 + [40, 9000, 641], 4, 4, 64, 32, 7, "max", 256, True),
    ([2000, 300, 4097, 1025], 6, 2, 128, 24, 13, "avg", 128, False),          # window not a multiple of 16
    ([900, 33000, 4000], 8, 1, 128, 64, 7, "max", 512, False),                # clusters of select CTAs
    ([50000, 60000, 1000, 70000], 16, 8, 128, 32, 7, "max", 1024, False),     # more than one wave per sequence
    ([150 + 37 * i for i in range(70)], 2, 1, 64, 32, 5, "avg", 140, False),  # more sequences than a launch takes
    ([700, 1900, 800], 4, 2, 128, 32, 17, "max", 100, False),                 # radius 8: one sequence at a time
])
def test_ragged_batch_equals_the_calls_one_by_one(lens, Hq, Hkv, d, W, kernel, ptype, budget, use_lse):
    # bit for bit: every sequence of the batch is scored in the order of a call of its own.  Once
    # with the workspace the call picks and once with the least it must accept (groups of one).
    g = torch.Generator(device="cuda").manual_seed(len(lens) + W)
    seqs = [{x: torch.randn(*sh, generator=g, device="cuda").to(torch.bfloat16)
             for x, sh in (("q", (1, Hq, W, d)), ("k", (1, Hkv, L, d)), ("v", (1, Hkv, L, d)))} for L in lens]
    lses = [torch.randn(1, Hq, W, generator=g, device="cuda") + 7.0 for _ in lens] if use_lse else None
    k, v = (torch.cat([s[x][0].permute(1, 0, 2) for s in seqs]).contiguous() for x in "kv")   # [T, Hkv, d]
    q = torch.cat([s["q"] for s in seqs])
    cu = [sum(lens[:b]) for b in range(len(lens))]
    least = max([sk.snapkv_workspace_size(1, Hq, Hkv, L, d, W, kernel, PT[ptype], budget) for L in lens if L > budget])
    for ws in (None, torch.full((least,), 0xFF, dtype=torch.uint8, device="cuda")):
        out_k, out_v, out_idx, used = sk.snapkv_compress_varlen(
            q, k, v, lens, kernel, PT[ptype], budget, cu_seqlens=cu, workspace=ws,
            lse_obs=torch.cat(lses) if use_lse else None)
        assert (used is ws) == (ws is not None) and sk.snapkv_device_status(used) == (sk.OK, 0)
        for b, s in enumerate(seqs):
            rows = min(budget, lens[b])
            ok, ov, oi, _ = sk.snapkv_compress(s["q"], s["k"], s["v"], kernel, PT[ptype], budget,
                                               lse_obs=lses[b] if use_lse else None)
            assert torch.equal(out_idx[b, :, :rows - W], oi[0]) and bool((out_idx[b, :, rows - W:] == -1).all())
            for got, want in ((out_k, ok), (out_v, ov)):
                assert torch.equal(got[b, :, :rows], want[0]) and not bool(got[b, :, rows:].any())


def test_a_workspace_from_a_smaller_batch_does_not_cost_launches():
    Hq, Hkv, d, W, kernel, budget = 4, 2, 128, 32, 5, 200
    g = torch.Generator(device="cuda").manual_seed(9)
    k = torch.randn(16, Hkv, 1500, d, generator=g, device="cuda").to(torch.bfloat16)
    q = torch.randn(16, Hq, W, d, generator=g, device="cuda").to(torch.bfloat16)
    small, large = [900, 1500, 640], [300 + 80 * i for i in range(16)]

    def call(lens, ws):
        out = sk.snapkv_compress_varlen(q[:len(lens)], k[:len(lens)], k[:len(lens)], lens, kernel, sk.POOL_MAX, budget,
                                        workspace=ws)
        assert sk.snapkv_device_status(out[3]) == (sk.OK, 0)
        return out, sk.snapkv_last_launch_count()

    want, fewest = call(large, None)
    (_, _, _, ws), _ = call(small, None)
    got, launches = call(large, ws)                       # handed on, as a serving loop does
    assert launches == fewest and all(torch.equal(x, y) for x, y in zip(got[:3], want[:3]))
    again, launches = call(small, got[3])                 # and kept from then on
    assert again[3] is got[3] and launches == fewest
    # a workspace of the caller's own is used as it is: of the size the library names, one set of launches
    size = sk.snapkv_varlen_workspace_size(large, Hq, Hkv, d, W, kernel, sk.POOL_MAX, budget)
    for nbytes, sets in ((size, 1), (size - 256, 2)):
        own = torch.full((nbytes,), 0xFF, dtype=torch.uint8, device="cuda")
        got, launches = call(large, own)
        assert got[3] is own and all(torch.equal(x, y) for x, y in zip(got[:3], want[:3]))
        assert (launches - fewest) // 3 == sets - 1       # preparation, scores, selection per set; one gather


@pytest.mark.parametrize("lens,ptype,kernel,selects", [
    # rows of 4097 and more, and up to 4096 and 2048, in two launches side by side; the last ones all long or all in one
    ([700, 20000, 4128, 2081, 9000, 4129, 2080, 4127], "max", 7, 2),
    ([24000, 1400, 23000, 8000, 1500, 21000], "avg", 5, 2),
    ([12283, 900, 2990, 2867], "max", 5, 1),
    ([17000, 16416, 8225, 8224, 33000], "max", 13, 1),
])
def test_rows_of_a_ragged_batch_in_one_or_two_select_launches(lens, ptype, kernel, selects):
    Hq, Hkv, d, W, budget = 32, 8, 64, 32, 512
    g = torch.Generator(device="cuda").manual_seed(sum(lens))
    seqs = [{x: torch.randn(*sh, generator=g, device="cuda").to(torch.bfloat16)
             for x, sh in (("q", (1, Hq, W, d)), ("k", (1, Hkv, L, d)), ("v", (1, Hkv, L, d)))} for L in lens]
    k, v = (torch.cat([s[x][0].permute(1, 0, 2) for s in seqs]).contiguous() for x in "kv")
    q = torch.cat([s["q"] for s in seqs])
    cu = [sum(lens[:b]) for b in range(len(lens))]
    want = [sk.snapkv_compress(s["q"], s["k"], s["v"], kernel, PT[ptype], budget)[:3] for s in seqs]

    def call(ws):
        return sk.snapkv_compress_varlen(q, k, v, lens, kernel, PT[ptype], budget, cu_seqlens=cu, workspace=ws)

    got = call(None)
    assert sk.snapkv_last_launch_count() == 3 + selects  # preparation, scores, selection, gather
    runs = [got] + [call(got[3]) for _ in range(3)]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = call(got[3])
    for _ in range(3):
        for x in captured[:3]:
            x.zero_()
        graph.replay()
    runs.append(captured)
    for run in runs:
        for b in range(len(lens)):
            assert all(torch.equal(x[b], y[0]) for x, y in zip(run[:3], want[b]))


def test_two_select_launches_read_the_votes_of_their_own_call():
    # Calls on different inputs follow one another on one workspace without a synchronisation: the second
    # select launch of each reads votes while the first one runs, and must find this call's.
    lens, Hq, Hkv, d, W, budget = [700, 20000, 4128, 2081, 9000, 4129, 2080, 4127], 32, 8, 64, 32, 512
    inputs, want = [], []
    for i in range(4):
        g = torch.Generator(device="cuda").manual_seed(i)
        x = [torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
             for s in ((len(lens), Hq, W, d), (sum(lens), Hkv, d), (sum(lens), Hkv, d))]
        inputs.append(x)
        at = 0
        for b, L in enumerate(lens):
            one = [t[at:at + L].permute(1, 0, 2)[None].contiguous() for t in x[1:]]
            want.append(sk.snapkv_compress(x[0][b:b + 1].contiguous(), *one, 7, sk.POOL_MAX, budget)[2])
            at += L
    cu = [sum(lens[:b]) for b in range(len(lens))]
    ws, got = None, []
    for _ in range(5):
        for x in inputs:
            *out, ws = sk.snapkv_compress_varlen(*x, lens, 7, sk.POOL_MAX, budget, cu_seqlens=cu, workspace=ws)
            got.append(out[2])
            assert sk.snapkv_last_launch_count() == 5  # preparation, scores, two selections, gather
    for c, idx in enumerate(got):
        for b in range(len(lens)):
            assert torch.equal(idx[b], want[c % 4 * len(lens) + b][0])


def test_two_groups_of_sequences_with_two_select_launches_each():
    lens = [19000 + 37 * b if b % 4 == 0 else 300 + 29 * b for b in range(40)]
    Hq, Hkv, d, W, budget = 16, 4, 64, 32, 128
    g = torch.Generator(device="cuda").manual_seed(40)
    q, k, v = (torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
               for s in ((len(lens), Hq, W, d), (sum(lens), Hkv, d), (sum(lens), Hkv, d)))
    cu = [sum(lens[:b]) for b in range(len(lens))]
    ws = None
    for _ in range(2):  # the second time on a workspace that the first one left
        *out, ws = sk.snapkv_compress_varlen(q, k, v, lens, 7, sk.POOL_MAX, budget, cu_seqlens=cu, workspace=ws)
        assert sk.snapkv_last_launch_count() == 2 * 4 + 2  # two groups, and a gather for 32 and for 8 sequences
        for b, L in enumerate(lens):
            one = [t[cu[b]:cu[b] + L].permute(1, 0, 2)[None].contiguous() for t in (k, v)]
            want = sk.snapkv_compress(q[b:b + 1].contiguous(), *one, 7, sk.POOL_MAX, budget)[:3]
            assert all(torch.equal(x[b], y[0]) for x, y in zip(out, want))
