"""Calls from several threads.  A call's work is ordered by its stream; what the library shares
between threads is host state that the first call fills (driver entry points, device facts), and
each thread gets the device's context with its own first call."""
import os
import subprocess
import sys
import threading

import pytest
import torch

from paper_2404_14469_b200 import binding as sk

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


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


# Eight threads of a fresh process whose first library calls overlap, all on the default stream (so
# that the device runs them one after the other): ragged batches first, which ask for a tensor map
# before anything else, then decode steps, which ask the device what clusters it holds.
FIRST_CALLS = """
import threading, torch
from paper_2404_14469_b200 import binding as sk
sk._load_native()
N, Hq, Hkv, d, W, lens = 8, 4, 2, 128, 16, [300, 700]
g = torch.Generator(device="cuda").manual_seed(5)
rand = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
ins = [(rand(2, Hq, W, d), rand(2, Hkv, 700, d), rand(2, Hkv, 700, d)) for _ in range(N)]
torch.cuda.synchronize()
gate, got, bad = threading.Barrier(N), [None] * N, []
def work(i):
    q, k, v = ins[i]
    try:
        gate.wait()
        a = sk.snapkv_compress_varlen(q, k, v, lens, 5, sk.POOL_MAX, 128)
        gate.wait()
        b = sk.snapkv_decode_attention(q[:, :, 0].contiguous(), a[0], a[1])
        got[i] = (a, b)
    except Exception as e:
        gate.abort()
        bad.append(repr(e))
threads = [threading.Thread(target=work, args=(i,)) for i in range(N)]
[t.start() for t in threads]
[t.join() for t in threads]
assert not bad, bad
for (q, k, v), (a, b) in zip(ins, got):
    assert sk.snapkv_device_status(a[3]) == (sk.OK, 0)
    a2 = sk.snapkv_compress_varlen(q, k, v, lens, 5, sk.POOL_MAX, 128)
    b2 = sk.snapkv_decode_attention(q[:, :, 0].contiguous(), a2[0], a2[1])
    assert all(torch.equal(x, y) for x, y in zip(a[:3] + b[:2], a2[:3] + b2[:2]))
print("same")
"""


def test_first_calls_of_several_threads_at_once():
    r = subprocess.run([sys.executable, "-c", FIRST_CALLS], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stdout + r.stderr


def _batches(n):
    g = torch.Generator(device="cuda").manual_seed(6)
    out = []
    for i in range(n):
        lens = [400 + 311 * i, 150, 2000 - 97 * i, 129]
        out.append((lens, [torch.randn(4, h, r, 128, generator=g, device="cuda").to(torch.bfloat16)
                           for h, r in ((4, 32), (2, 2400), (2, 2400))]))
    return out


@pytest.mark.parametrize("own_streams", [False, True])
def test_ragged_batches_of_several_threads(own_streams):
    # Each thread has its workspace.  On one stream their launches interleave as they come; on streams
    # of their own the calls are ordered by events, since two may not overlap on one device.
    batches, rounds = _batches(4), 3
    call = lambda lens, x, ws=None: sk.snapkv_compress_varlen(*x, lens, 5, sk.POOL_MAX, 200, workspace=ws)
    want = [call(lens, x) for lens, x in batches]
    torch.cuda.synchronize()
    got, bad, turn, last = [[] for _ in batches], [], threading.Lock(), [None]

    def work(i):
        try:
            lens, x = batches[i]
            ws = None
            stream = torch.cuda.Stream() if own_streams else torch.cuda.current_stream()
            with torch.cuda.stream(stream):
                for _ in range(rounds):
                    if own_streams:
                        with turn:
                            if last[0] is not None:
                                stream.wait_event(last[0])
                            got[i].append(call(lens, x, ws))
                            last[0] = stream.record_event()
                    else:
                        got[i].append(call(lens, x, ws))
                    ws = got[i][-1][3]
        except Exception as e:
            bad.append(repr(e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(batches))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not bad, bad
    for i, ref in enumerate(want):
        for out in got[i]:
            assert sk.snapkv_device_status(out[3]) == (sk.OK, 0)
            assert all(torch.equal(x, y) for x, y in zip(out[:3], ref[:3]))
