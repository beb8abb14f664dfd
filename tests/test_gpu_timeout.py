"""The time-out path of the scoring kernel, exercised on the GPU in the only safe form: a
wait on a flag that nothing ever sets, with a short limit.  Every wait in the kernel is
bounded; when one runs out the block records the wait's code, lets its copies and
tensor-core operations finish, frees its tensor memory and returns, and the host reads
SNAPKV_ERR_TIMEOUT from the workspace.  Nothing here faults or hangs the device."""
import time

import pytest
import torch

from oracle import snapkv_oracle as orc
from paper_2404_14469_b200 import binding as sk
from paper_2404_14469_b200 import synth

import parity

pytestmark = pytest.mark.gpu

TIMEOUT, WAIT_UNIT_STATS = 5, 7


@pytest.mark.parametrize("B,Hq,Hkv,L,d,W", [
    (1, 4, 2, 3000, 128, 32),       # a few blocks have work
    (2, 32, 8, 16384, 128, 32),     # every block of the grid has work and runs into the limit
])
def test_a_wait_that_nothing_satisfies_runs_out_and_the_context_survives(B, Hq, Hkv, L, d, W):
    data = synth.make_random(B, Hq, Hkv, L, d, W, seed=77)
    q, k = data["q_obs"].cuda(), data["k"].cuda()
    vote = torch.full((B, Hq, L - W), -1.0, dtype=torch.float32, device="cuda")
    prev = sk.snapkv_set_wait_limit_ns(20_000_000)          # 20 ms; waits on other blocks: 10 ms
    try:
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        _, ws = sk.snapkv_selftest_stalled_scores(q, k, vote)
        code, detail = sk.snapkv_device_status(ws)           # synchronises the stream
        took = time.perf_counter() - t0
    finally:
        sk.snapkv_set_wait_limit_ns(prev)
    assert (code, detail) == (TIMEOUT, WAIT_UNIT_STATS)
    assert sk.status_string(code) == "SNAPKV_ERR_TIMEOUT"
    assert 0.005 < took < 2.0                                # it did wait, and it did return
    assert bool((vote == -1.0).all())                        # no vote was written
    # the context is intact: the ordinary call on the same buffers is correct and clean
    vote2, ws2 = sk.snapkv_window_scores(q, k, vote, ws)
    assert sk.snapkv_device_status(ws2) == (sk.OK, 0)
    heads = [(0, 0), (B - 1, Hq - 1)]
    qb, kb = synth.bf16_bits(data["q_obs"]), synth.bf16_bits(data["k"])
    g = Hq // Hkv
    for b, h in heads:
        ref = orc.window_votes(orc.bf16_bits_to_f64(qb[b, h]), orc.bf16_bits_to_f64(kb[b, h // g]))
        parity.check_votes(vote2[b, h].cpu().numpy(), ref)


@pytest.mark.parametrize("lens,Hq,Hkv,L,d,W", [
    (None, 4, 2, 3000, 128, 32),               # one wave, a few tiles per block
    (None, 32, 8, 16384, 128, 32),             # every block of the grid has work
    (None, 8, 8, 40000, 64, 16),               # narrow units, 32 columns
    ([3000, 700, 16384, 129], 32, 8, 16384, 128, 32),   # ragged: the folding blocks wait for slots, the others for rows
    ([900, 5000], 4, 1, 5000, 64, 24),
])
def test_partials_that_are_never_published_run_out(lens, Hq, Hkv, L, d, W):
    # the waits on the main path: both sweeps run, the statistics are computed, no slot is written
    B = 2 if lens is None else len(lens)
    g = torch.Generator(device="cuda").manual_seed(78)
    q, k = (torch.randn(B, h, r, d, generator=g, device="cuda").to(torch.bfloat16) for h, r in ((Hq, W), (Hkv, L)))
    sizes = (Hq, Hkv, d, W, 1, sk.POOL_MAX, W + 1)
    need = (sk.snapkv_workspace_size(B, Hq, Hkv, L, *sizes[2:]) if lens is None
            else sk.snapkv_varlen_workspace_size(lens, *sizes))
    votes = -(-4 * Hq * sum((x - W) for x in (lens or [L] * B)) // 256) * 256
    ws = torch.full((need,), 0xFF, dtype=torch.uint8, device="cuda")
    call = lambda: (sk.snapkv_compress(q, k, k, 7, sk.POOL_MAX, 100) if lens is None
                    else sk.snapkv_compress_varlen(q, k, k, lens, 7, sk.POOL_MAX, 100))
    want = call()
    prev = sk.snapkv_set_wait_limit_ns(20_000_000)
    try:
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        sk.snapkv_selftest_withheld_partials(q, k, ws, lens)
        code, detail = sk.snapkv_device_status(ws)
        took = time.perf_counter() - t0
    finally:
        sk.snapkv_set_wait_limit_ns(prev)
    assert (code, detail) == (TIMEOUT, WAIT_UNIT_STATS)
    assert 0.005 < took < 2.0
    assert bool((ws[need - votes:] == 0xFF).all())           # no vote was written
    again = call()
    assert sk.snapkv_device_status(again[3]) == (sk.OK, 0)
    assert all(torch.equal(x, y) for x, y in zip(again[:3], want[:3]))
