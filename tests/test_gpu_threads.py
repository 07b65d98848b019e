"""Calls from several host threads, each on a stream of its own."""
import os
import subprocess
import sys
import threading

import pytest
import torch

import sdq_synth
from tests.test_gpu_parity import sdq

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def in_threads(n, fn):
    """fn(i) on n threads at once, each with its own stream; the results in order"""
    start, out = threading.Barrier(n), [None] * n

    def body(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            start.wait()
            try:
                out[i] = fn(i)
            except Exception as e:
                out[i] = e
            torch.cuda.current_stream().synchronize()
    ts = [threading.Thread(target=body, args=(i,)) for i in range(n)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return out


@pytest.mark.parametrize("n", [6, 80])                  # (80: more than the packer has report words for)
def test_each_packing_call_gets_its_own_answer(n):
    """finite and non-finite matrices decomposed at once: an error where there is one and nowhere else, and the same bytes as alone"""
    m = sdq()
    cfg = m.Config()
    W = sdq_synth.make_weight(1024, 1024, 130).cuda()
    B = W.clone()
    B[700, 801] = float("nan")
    alone = m.sdq_decompose(W, cfg).buf
    torch.cuda.synchronize()
    got = in_threads(n, lambda i: m.sdq_decompose(B if i % 3 == 1 else W, cfg))
    for i, r in enumerate(got):
        if i % 3 == 1:
            assert isinstance(r, m.SdqError) and r.code == 6, i
        else:
            assert torch.equal(r.buf, alone), i


_FIRST = r"""
import sys
sys.path.insert(0, sys.argv[1])
import torch
import sdq_synth
from tests.test_gpu_parity import sdq
from tests.test_gpu_threads import in_threads
m = sdq()
cases = []
for M, N, K, block in ((300, 384, 2048, 32), (7, 4096, 1024, 64), (600, 2048, 1024, 64)):     # K over four pairs; grouped kernel; tasks of two units
    cfg = m.Config(1, m.GRAN_PAIR, block)
    cases.append((m.sdq_decompose(sdq_synth.make_weight(N, K, 131).cuda(), cfg), m.sdq_quantize_act(sdq_synth.make_act(M, K, 132).cuda(), cfg)))
torch.cuda.synchronize()
first = in_threads(12, lambda i: m.sdq_linear(cases[i % 3][1], cases[i % 3][0], f32=True))
for i, y in enumerate(first):
    assert torch.equal(y, m.sdq_linear(cases[i % 3][1], cases[i % 3][0], f32=True)), (i, y)
assert m.device_status() == 0
print("ok")
"""


def test_the_first_calls_of_a_process_from_several_threads():
    """whatever a first call looks up per device is there for the calls beside it: the same plan, so the same bits, as later on"""
    for _ in range(2):
        r = subprocess.run([sys.executable, "-c", _FIRST, ROOT], cwd=ROOT, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, timeout=300)
        assert r.returncode == 0 and r.stdout.decode().strip().endswith("ok"), r.stdout.decode()[-2000:]
