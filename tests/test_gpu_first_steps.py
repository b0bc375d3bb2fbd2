"""First steps: of handles in a CUDA context of the caller's own, and of several threads at once.  Each runs in a process of
its own, where nothing has prepared the kernels yet."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import threading
import torch
from paper_2511_22972_b200 import FlyVerify, VerifyBuffers, verify

def host_step(dtype, B, K, V):
    torch.manual_seed(V)
    logits = torch.randn(B, K + 1, V).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    draft = logits[:, :K].float().argmax(-1).to(torch.int32)
    draft[:, 1:2] = 0
    out = VerifyBuffers(B, K, "cpu")
    fv = FlyVerify(B, K, V, dtype)
    verify(fv, logits, draft, out, theta=1.0, W=0, host=True)
    fv.close()
    assert torch.equal(out.target_argmax.long(), logits.float().argmax(-1))
    return out.entropy
"""


def run(body):
    r = subprocess.run([sys.executable, "-c", PRELUDE + body], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-500:] + r.stderr[-1500:]


def test_a_handle_in_a_context_of_the_callers_own():
    # what a kernel needs before its first launch belongs to the context, not to the device or the process
    pytest.importorskip("cuda.bindings.driver")
    run("""
from cuda.bindings import driver as cu
shapes = [("bf16", 2, 3, 32000), ("f32", 2, 3, 32000), ("bf16", 470, 1, 2051), ("f32", 470, 1, 2051)]
torch.zeros(1, device="cuda")
first = [host_step(*s) for s in shapes]
err, ctx = cu.cuCtxCreate(0, 0)
assert err == cu.CUresult.CUDA_SUCCESS, err
second = [host_step(*s) for s in shapes]
cu.cuCtxPopCurrent()
assert cu.cuCtxDestroy(ctx)[0] == cu.CUresult.CUDA_SUCCESS
assert all(torch.equal(a, b) for a, b in zip(first, second))
""")


def test_first_steps_of_many_threads_at_once():
    run("""
torch.zeros(1, device="cuda")
failed, barrier = [], threading.Barrier(16)
def go(i):
    barrier.wait()
    try:
        host_step(("bf16", "f32")[i % 2], *((470, 1, 2051) if i % 4 < 2 else (2, 3, 32000)))
    except Exception as e:
        failed.append(str(e))
threads = [threading.Thread(target=go, args=(i,)) for i in range(16)]
[t.start() for t in threads]
[t.join() for t in threads]
assert not failed, failed
""")


def test_making_a_handle_does_not_wait_for_work_that_is_queued():
    # a server makes handles while the model runs; and the first step on a stream of its own finds the scratch clear
    run("""
logits = torch.randn(4, 4, 32000, device="cuda").to(torch.bfloat16)
draft = logits[:, :3].float().argmax(-1).to(torch.int32)
a = torch.randn(8192, 8192, device="cuda", dtype=torch.bfloat16)
FlyVerify(4, 3, 32000).close()
torch.mm(a, a)
side, out, out2 = torch.cuda.Stream(), VerifyBuffers(4, 3, "cuda"), VerifyBuffers(4, 3, "cuda")
torch.cuda.synchronize()
for mode in ("global", "thread_local", "relaxed"):
    for _ in range(60):
        torch.mm(a, a)                      # some 40 ms on the default stream
    queued = torch.cuda.Event()
    queued.record()
    fv = FlyVerify(4, 3, 32000)
    assert not queued.query(), "the handle was made only after the queue had run dry"
    for step in range(2):                   # neither waits for the default stream by itself
        verify(fv, logits, draft, out, theta=1.0, W=0, stream=side.cuda_stream)
    captured = FlyVerify(4, 3, 32000)       # ... nor can a first step that is captured
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        assert not queued.query()
        graph.capture_begin(capture_error_mode=mode)
        verify(captured, logits, draft, out2, theta=1.0, W=0, stream=side.cuda_stream)
        graph.capture_end()
        graph.replay()
    torch.cuda.synchronize()
    for o in (out, out2):
        assert torch.equal(o.target_argmax.long(), logits.float().argmax(-1)) and (o.row_flags == 0).all()
    captured.close()
    fv.close()
""")
