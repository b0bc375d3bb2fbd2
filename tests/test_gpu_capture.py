"""Every entry point that enqueues work can be captured in a CUDA graph: the launches of a step, each a programmatic dependent
of the one before it, become a graph that is replayed over inputs that change in place and between plain calls."""
import numpy as np
import pytest
import torch

from oracle import fly_oracle as O
from oracle.pld_oracle import pld_draft as oracle_pld
from paper_2511_22972_b200 import FlyVerify, VerifyBuffers, binding as Bd, synthetic as S, verify, verify_fused
from tests._parity import assert_parity, draw, oracle_step
from tests.test_gpu_fused import fused_case

pytestmark = pytest.mark.gpu
DEV = "cuda"


def captured(step):
    """step(stream) three times in one graph, after one plain call; returns a replay that waits."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        step(stream.cuda_stream)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            for _ in range(3):
                out = step(stream.cuda_stream)

    def replay():
        with torch.cuda.stream(stream):
            g.replay()
        torch.cuda.synchronize()
        return out
    replay.plain = lambda: (step(stream.cuda_stream), torch.cuda.synchronize())
    return replay


@pytest.mark.parametrize("how", ["handle", "two kernels", "static", "shard"])
def test_captured_logits_steps(how):
    w = S.shrink(S.LLAMA3, B=5, K=6, V=50257)
    logits, draft = draw(w, step=1)
    fv, out = FlyVerify(w.B, w.K, w.V, "bf16"), VerifyBuffers(w.B, w.K, DEV)
    kw = dict(theta=1.0, W=2, state_out=out.state, rollback=out.rollback, target_argmax=out.target_argmax, entropy=out.entropy,
              row_flags=out.row_flags)
    if how == "static":
        a = Bd.static_args(w.B, w.K, draft, out.accept_len, out.out_tokens, logits=logits, **kw)
        step = lambda s: Bd.run_static(a, w.V, "bf16", 0, s)
    elif how == "shard":
        cut = 24000
        other = FlyVerify(w.B, w.K, w.V - cut, "bf16")
        fv = FlyVerify(w.B, w.K, cut, "bf16")
        parts, flat = torch.empty(2, w.rows, 4, device=DEV), logits.view(-1, w.V)
        a = fv.make_args(w.B, w.K, draft, out.accept_len, out.out_tokens, **kw)

        def step(s):
            fv.reduce_shard(flat[:, :cut], 0, parts[0], s)
            other.reduce_shard(flat[:, cut:], cut, parts[1], s)
            fv.run_partials(a, parts, 2, w.V, s)
    else:
        fv.set_scan_mode(how == "two kernels")
        step = lambda s: verify(fv, logits, draft, out, theta=1.0, W=2, stream=s)
    replay = captured(step)
    for i in range(2, 5):
        fresh, d = draw(w, step=i)
        logits.copy_(fresh)
        draft.copy_(d)
        torch.cuda.synchronize()
        ref = oracle_step(logits, draft, 1.0, 2)
        for run in (replay, replay.plain, replay):
            out.out_tokens.fill_(-9)
            out.entropy.fill_(-9)
            torch.cuda.synchronize()
            run()
            assert_parity(out, ref, f"{how} step {i}")
    fv.close()


@pytest.mark.parametrize("B,K", [(4, 8), (20, 14)])      # one launch and fold in the scan; two launches and a fold kernel
def test_captured_fused_steps(B, K):
    cases = [fused_case(B, K, 256, 1512, step=i) for i in range(3)]
    w, hidden, weight, draft = cases[0][0], cases[0][1].clone(), cases[0][2], cases[0][3].clone()
    fv, out = FlyVerify(B, K, w.V, "bf16", hidden=w.hidden), VerifyBuffers(B, K, DEV)
    replay = captured(lambda s: verify_fused(fv, hidden, weight, draft, out, theta=1.0, W=3, stream=s))
    for _, h, wt, d, logits in cases[1:]:
        hidden.copy_(h)
        weight.copy_(wt)
        draft.copy_(d)
        torch.cuda.synchronize()
        ref = O.verify_batch(logits.reshape(B, K + 1, w.V), draft.cpu().numpy(), 1.0, 3)
        for run in (replay, replay.plain, replay):
            out.out_tokens.fill_(-9)
            torch.cuda.synchronize()
            run()
            assert_parity(out, ref, f"{B}x{K}")
    assert fv.device_status() == Bd.FLY_OK
    fv.close()


def test_captured_drafting():
    g = torch.Generator().manual_seed(1)
    B, L = 6, 20000                               # a cluster of blocks per sequence
    tokens = torch.empty(B, L, dtype=torch.int32, device=DEV)
    lengths = torch.empty(B, dtype=torch.int32, device=DEV)
    tokens.zero_()
    lengths.fill_(L)
    replay = captured(lambda s: Bd.pld_draft(tokens, lengths, 8, 4, 1, stream=s))
    for _ in range(3):
        t = torch.randint(0, 30, (B, L), generator=g, dtype=torch.int32)
        n = torch.randint(1, L + 1, (B,), generator=g, dtype=torch.int32)
        tokens.copy_(t)
        lengths.copy_(n)
        torch.cuda.synchronize()
        draft, count, pos, ngram = replay()
        for b in range(B):
            prop, p, k = oracle_pld(t[b, :n[b]].tolist(), 8, 4, 1)
            assert (count[b].item(), pos[b].item(), ngram[b].item()) == (len(prop), p, k) and draft[b, :len(prop)].tolist() == prop
