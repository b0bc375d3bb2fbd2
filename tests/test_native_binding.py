"""The native argument marshalling refuses what it cannot read with a Python exception, as the ctypes binding did: no C++
exception may leave it.  No call here reaches the library with a handle, so no GPU is needed; each runs in a process of
its own, because a failure ends it."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import torch
from paper_2511_22972_b200 import FlyVerify, VerifyBuffers, binding as B
class Handle:
    value = 0
class Fv:
    _h = Handle(); vocab = 8; weight_vd = False
    def _raise(self, status, what): raise B.FlyError(status, what)
i32 = dict(dtype=torch.int32)
fv, draft = Fv(), torch.zeros(1, 1, **i32)
"""


def run(body):
    r = subprocess.run([sys.executable, "-W", "ignore", "-c", PRELUDE + body], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout[-500:], r.stderr[-1500:])
    return r.stdout


CALLS = [
    "B.verify(fv, torch.nested.nested_tensor([torch.zeros(2, 8)]), draft, VerifyBuffers(1, 1, 'cpu'))",
    "B.verify(fv, torch.nested.nested_tensor([torch.zeros(2, 8)], layout=torch.jagged), draft, VerifyBuffers(1, 1, 'cpu'))",
    "B.verify(fv, torch.zeros(1, 2, 8).to_sparse(), draft, VerifyBuffers(1, 1, 'cpu'))",
    "B.verify(fv, torch.zeros(1, 2, 8), draft.to_sparse(), VerifyBuffers(1, 1, 'cpu'))",
    "B.verify_fused(fv, torch.nested.nested_tensor([torch.zeros(16), torch.zeros(16)]), torch.zeros(16, 8), draft, VerifyBuffers(1, 1, 'cpu'))",
    "FlyVerify.reduce_shard(fv, torch.nested.nested_tensor([torch.zeros(8)]), 0, torch.zeros(2, 4))",
    "B.pld_draft(torch.nested.nested_tensor([torch.zeros(8, **i32)]), torch.zeros(1, **i32), 4)",
    "B.pld_draft(torch.zeros(1, 8, **i32), torch.ones(1, **i32).to_sparse(), 4)",       # thrown while other threads may run
    "B.pld_draft(torch.zeros(1, 8, **i32), torch.zeros(1, **i32), -4)",
    "B.static_args(1, 1, draft.to_sparse(), draft, draft)",
    "torch.func.vmap(lambda x: B.verify(fv, x, draft, VerifyBuffers(1, 1, 'cpu')).accept_len)(torch.zeros(3, 1, 2, 8))",
]


def test_tensors_without_strides_or_data_raise():
    # one after the other in one process, so that each also shows that the one before it left the interpreter usable
    out = run("B.lib()\n" + "".join(f"try:\n    {c}\nexcept Exception as e:\n    print({i}, 'raised', type(e).__name__, flush=True)\n"
                                    for i, c in enumerate(CALLS)) + "print('alive', sum(range(4)))\n")
    lines = out.splitlines()
    assert [line.split()[:2] for line in lines] == [[str(i), "raised"] for i in range(len(CALLS))] + [["alive", "6"]], out


def test_numbers_are_taken_as_float_and_int_take_them():
    out = run("a = B.static_args(1, True, draft, draft, draft, theta='inf', W=torch.tensor(2), temperature=torch.tensor(0.5))\n"
              "print(a.theta, a.K, a.W, a.temperature)\n")
    assert out.split() == ["inf", "1", "2", "0.5"]


def test_arguments_can_be_filled_before_anything_has_loaded_the_library():
    out = run("print(FlyVerify.make_args(None, 2, 3, draft, draft, draft, theta=0.5).K)\n")
    assert out.split() == ["3"]
