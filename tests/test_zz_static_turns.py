"""The static entry point's calls take turns at the parts of its scratch: calls of many shapes in a row, on two streams one after the
other, between replays of a captured call and calls with inputs_ready, give what a handle gives."""
import pytest
import torch

from paper_2511_22972_b200 import FlyVerify, VerifyBuffers, binding as Bd, synthetic as S
from tests._parity import draw

pytestmark = pytest.mark.gpu
DEV = "cuda"
FIELDS = ("accept_len", "out_tokens", "target_argmax", "entropy", "row_flags", "rollback", "state")


def test_calls_take_turns():
    # the smallest and the largest number of sequences and rows, whole rows and pieces, element by element (V = 100)
    shapes = [(1, 1, 100, "bf16"), (4, 25, 128256, "bf16"), (1024, 1, 300, "f32"), (1, 8, 32000, "f32"), (256, 63, 257, "bf16"),
              (16, 8, 50257, "bf16"), (2, 15, 128256, "bf16")]
    steps = []
    for n, (B, K, V, dtype) in enumerate(shapes):
        w = S.shrink(S.LLAMA3, B=B, K=K, V=V, dtype=dtype)
        logits, draft = draw(w, step=n, guard=False)

        def args(out, ready, B=B, K=K, logits=logits, draft=draft):
            return Bd.static_args(B, K, draft, out.accept_len, out.out_tokens, logits=logits, theta=1.0, W=2, state_out=out.state,
                                  rollback=out.rollback, target_argmax=out.target_argmax, entropy=out.entropy, row_flags=out.row_flags,
                                  inputs_ready=ready)
        want, got = VerifyBuffers(B, K, DEV), VerifyBuffers(B, K, DEV)
        fv = FlyVerify(B, K, V, dtype)
        fv.run(args(want, False), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        fv.close()
        steps.append((args, want, got, V, dtype))

    def call(i, stream, ready=False):
        args, _, got, V, dtype = steps[i]
        got.entropy.fill_(-1.0)
        Bd.run_static(args(got, ready), V, dtype, 0, stream.cuda_stream)

    def check(i, what):
        torch.cuda.synchronize()
        _, want, got, V, dtype = steps[i]
        for f in FIELDS:
            a, b = getattr(got, f), getattr(want, f)
            ok = torch.equal(a, b) if f != "entropy" else torch.allclose(a, b, rtol=0, atol=1e-5, equal_nan=True)  # (pieces may differ)
            assert ok, (what, shapes[i], f)

    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    with torch.cuda.stream(streams[0]):
        call(1, streams[0])
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=streams[0]):
            call(1, streams[0])
    turn = 0
    for rounds in range(3):
        for i in range(len(steps)):
            stream, other = streams[turn % 2], streams[1 - turn % 2]
            turn += 1
            stream.wait_stream(other)
            with torch.cuda.stream(stream):
                call(i, stream)
                if i % 3 == 0:
                    graph.replay()
                call((i + 2) % len(steps), stream, ready=i % 2 == 0)
            check(i, "plain")
            check((i + 2) % len(steps), "after it")
            check(1, "captured") if i % 3 == 0 else None


def test_two_host_threads_on_one_stream():
    import threading
    shapes = [(4, 25, 32064, "bf16"), (300, 3, 1000, "f32")]
    stream, steps, failed = torch.cuda.Stream(), [], []
    for n, (B, K, V, dtype) in enumerate(shapes):
        w = S.shrink(S.LLAMA3, B=B, K=K, V=V, dtype=dtype)
        logits, draft = draw(w, step=n, guard=False)
        outs = [VerifyBuffers(B, K, DEV) for _ in range(400)]
        args = [Bd.static_args(B, K, draft, o.accept_len, o.out_tokens, logits=logits, theta=1.0, W=2, state_out=o.state,
                               rollback=o.rollback, target_argmax=o.target_argmax, entropy=o.entropy, row_flags=o.row_flags,
                               inputs_ready=i % 7 == 3) for i, o in enumerate(outs)]
        fv, want = FlyVerify(B, K, V, dtype), VerifyBuffers(B, K, DEV)
        fv.run(Bd.static_args(B, K, draft, want.accept_len, want.out_tokens, logits=logits, theta=1.0, W=2, state_out=want.state,
                              rollback=want.rollback, target_argmax=want.target_argmax, entropy=want.entropy,
                              row_flags=want.row_flags), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        fv.close()
        steps.append((args, outs, want, V, dtype))

    def work(args, V, dtype):
        try:
            for a in args:
                Bd.run_static(a, V, dtype, 0, stream.cuda_stream)
        except Exception as e:
            failed.append(e)
    threads = [threading.Thread(target=work, args=(args, V, dtype)) for args, _, _, V, dtype in steps]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed
    for (_, outs, want, _, _), shape in zip(steps, shapes):
        for i, got in enumerate(outs):
            for f in FIELDS:
                a, b = getattr(got, f), getattr(want, f)
                assert torch.equal(a, b) if f != "entropy" else torch.allclose(a, b, rtol=0, atol=1e-5), (shape, i, f)
