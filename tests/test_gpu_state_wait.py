"""The logits path's bounded wait for a partial state: made to run out in 2 ms by a scan over slots that nothing fills.
Nothing faults or hangs; the failure is reported as one, not as a property of the logits."""
import ctypes as C
import subprocess

import pytest
import torch

from oracle import fly_oracle as O
from paper_2511_22972_b200 import FlyVerify, binding as Bd, build, synthetic as S
from tests._parity import assert_parity, draw, gpu_step, oracle_step

pytestmark = pytest.mark.gpu
DEV = "cuda"

# One sequence of K = 2: each row has two states.  Entropy 1 nat or so, greedy tokens 11, 12, 13; `missing` (1-based) names the
# row whose second state never comes.
HARNESS = r"""
#include "scan_kernel.cuh"
using namespace fly;
__global__ void fill(Partial* slots, int missing) {
  const int r = threadIdx.x;
  Partial a = {4.0f, 2.0f, -1.0f, 11 + r}, b = {1.0f, 1.5f, -0.5f, 500 + r};
  st_part(slots + 2 * r, tagged(a));
  st_part(slots + 2 * r + 1, r + 1 == missing ? make_int4(0, 0, 0, 0) : tagged(b));
}
extern "C" int scan(int missing, int shard, const int* draft, int* accept, int* tokens, float* entropy, unsigned* flags, int* status,
                    Partial* slots, Partial* row_out) {
  fill<<<1, 3>>>(slots, missing);
  ScanParams p = {};
  p.B = shard ? 3 : 1; p.K = shard ? 0 : 2; p.V = 1000; p.splits = 2; p.lanes_log2 = 1; p.row_pitch = 2; p.part_pitch = 1;
  p.scale = 1.4426950408889634f; p.partials = slots; p.row_out = shard ? row_out : nullptr; p.idx_offset = 7;
  p.draft = draft; p.theta_nats = 1e9f; p.accept_len = accept; p.out_tokens = tokens; p.entropy = entropy; p.row_flags = flags;
  p.status = status; p.wait_ns = 2000000;
  scan_sequences<true><<<p.B, kScanThreads>>>(p);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def scan(tmp_path_factory):
    d = tmp_path_factory.mktemp("scan")
    (d / "scan.cu").write_text(HARNESS)
    subprocess.run([build.nvcc_path(), *build.NVCC_FLAGS, "-I", build.CSRC, "-o", str(d / "scan.so"), str(d / "scan.cu")], check=True)
    fn = C.CDLL(str(d / "scan.so")).scan
    status = torch.zeros(1, dtype=torch.int32, device=DEV)

    def call(missing, shard=False):
        i32 = dict(dtype=torch.int32, device=DEV)
        draft = torch.tensor([11, 12], **i32)
        accept, tokens, flags = torch.zeros(1, **i32), torch.zeros(3, **i32), torch.zeros(3, **i32)
        entropy, slots, rows = torch.zeros(3, device=DEV), torch.zeros(6, 4, **i32), torch.zeros(3, 4, device=DEV)
        p = [C.c_void_p(t.data_ptr()) for t in (draft, accept, tokens, entropy, flags, status, slots, rows)]
        torch.cuda.synchronize()
        assert fn(missing, int(shard), *p) == 0
        assert (slots == 0).all()                         # empty again for the next launch, whatever happened
        return accept.item(), tokens.tolist(), flags.tolist(), rows
    return call, status


def test_a_state_that_never_comes_fails_its_row_and_every_later_step(scan):
    call, status = scan
    assert call(0)[:3] == (3, [11, 12, 13], [0, 0, 0]) and status.item() == 0
    accept, tokens, flags, _ = call(2)                    # row 2: a mismatch, and not "non-finite logits"
    assert flags[1] == 16 and all(f in (0, 16) for f in flags) and status.item() == 4
    assert accept in (1, 2)                               # (1 if row 1 read the record too)
    assert call(0)[0] == 1 and call(0)[2] == [16, 16, 16]  # the record is pending
    status.zero_()
    assert call(0)[:3] == (3, [11, 12, 13], [0, 0, 0])


def test_a_shard_hands_the_failure_on_to_the_merge(scan):
    call, status = scan
    good = call(0, shard=True)[3]
    assert good.view(torch.int32)[:, 3].tolist() == [18, 19, 20] and good[:, 0].tolist() == [4.0] * 3
    rows = call(3, shard=True)[3]
    assert status.item() == 4 and rows[2, 0].item() == float("inf") and rows[2, 1].isnan() and rows.view(torch.int32)[2, 3].item() == 0x7ffffffe
    status.zero_()
    # two "ranks": the failed states and good ones, in both orders; rows 1 and 2 are whole
    fv = FlyVerify(1, 2, 1000, "bf16")
    failed = good.clone()
    failed[2] = rows[2]
    for parts in ((good, failed), (failed, good)):
        out = Bd.VerifyBuffers(1, 2, DEV)
        draft = torch.tensor([[18, 19]], dtype=torch.int32, device=DEV)
        a = fv.make_args(1, 2, draft, out.accept_len, out.out_tokens, theta=1e9, W=1, state_out=out.state, row_flags=out.row_flags)
        fv.run_partials(a, torch.stack(parts), 2, 1000)
        torch.cuda.synchronize()
        assert out.row_flags.tolist() == [[0, 0, 16]] and out.out_tokens.tolist() == [[18, 19, 0]]
    fv.close()


def test_a_pending_record_marks_logits_steps_until_it_is_read():
    st = torch.cuda.current_stream().cuda_stream
    w = S.shrink(S.LLAMA3, B=4, K=3, V=32000)
    logits, draft = draw(w)
    fv = FlyVerify(w.B, w.K, w.V, w.dtype)
    ref = oracle_step(logits, draft, 1.0, 3)
    shard = torch.empty(w.rows, 4, device=DEV)
    for separate in (False, True):
        fv.set_scan_mode(separate)
        assert fv.device_status(st) == Bd.FLY_OK and fv.selftest_wait(st) == Bd.FLY_OK
        out = gpu_step(fv, logits, draft, 1.0, 3)
        assert (out.row_flags == 16).all() and (out.accept_len == 1).all()
        fv.reduce_shard(logits.view(-1, w.V), 0, shard, st)
        assert (shard.view(torch.int32)[:, 3] == 0x7ffffffe).all()
        assert fv.device_status(st) == Bd.FLY_ERR_TIMEOUT and fv.device_status(st) == Bd.FLY_OK
        assert_parity(gpu_step(fv, logits, draft, 1.0, 3), ref, "after a reported timeout")
    fv.close()
