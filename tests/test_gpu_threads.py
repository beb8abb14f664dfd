"""Calls from several threads.  A call's work is ordered by its stream; what the library shares
between threads is host state that the first call fills (driver entry points, device facts), and
each thread gets the device's context with its own first call."""
import threading

import pytest
import torch

from paper_2404_14469_b200 import binding as sk

pytestmark = pytest.mark.gpu


def _in_thread(f):
    got = []
    t = threading.Thread(target=lambda: got.append(f()))
    t.start()
    t.join()
    assert got, "the call raised"
    return got[0]


def test_a_threads_first_library_call_may_be_any():
    # each call is the first CUDA work of a thread of its own
    g = torch.Generator(device="cuda").manual_seed(4)
    q, k, v = (torch.randn(2, h, r, 128, generator=g, device="cuda").to(torch.bfloat16)
               for h, r in ((4, 16), (2, 700), (2, 700)))
    q1, lens = q[:, :, 0].contiguous(), [300, 700]
    calls = [lambda: sk.snapkv_decode_attention(q1, k, v),
             lambda: sk.snapkv_compress_varlen(q, k, v, lens, 5, sk.POOL_MAX, 128)[:3],
             lambda: sk.snapkv_compress(q, k, v, 5, sk.POOL_MAX, 128)[:3],
             lambda: (sk.snapkv_window_scores(q, k)[0],)]
    for call in calls:
        here = call()
        torch.cuda.synchronize()
        there = _in_thread(call)
        assert all(torch.equal(x, y) for x, y in zip(here[:2], there[:2]))
