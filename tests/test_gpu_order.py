"""Plain stream order next to a kernel that lets its dependents start early: a step reads what the kernel just before it writes,
although its own blocks are resident by then and have asked for the first logits."""
import pytest
import torch

from paper_2511_22972_b200 import FlyVerify, VerifyBuffers, verify

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,K,V", [(1, 1, 128), (2, 1, 8192), (3, 2, 1003), (1, 7, 32000)])
def test_a_step_reads_what_the_kernel_before_it_writes(B, K, V):
    # the kernel before is a reduction whose states [rows, 4] are, as one row of numbers after the other, the step's logits
    rows = -(-B * (K + 1) * V // 4)
    g = torch.Generator(device=DEV)
    g.manual_seed(V)
    sources = [(3 * torch.randn(rows, 256, generator=g, device=DEV)).to(torch.bfloat16) for _ in range(2)]
    reducer, fv = FlyVerify(rows, 1, 256, "bf16"), FlyVerify(B, K, V, "f32")
    states = torch.zeros(rows, 4, device=DEV)
    logits = states.view(-1)[:B * (K + 1) * V].view(B, K + 1, V)
    draft = torch.randint(0, V, (B, K), generator=g, device=DEV, dtype=torch.int32)
    outs = [VerifyBuffers(B, K, DEV) for _ in sources]
    kept = lambda out: [t.clone() for t in (out.accept_len, out.out_tokens, out.target_argmax, out.entropy, out.row_flags)]

    def step(i, stream, apart=False):
        reducer.reduce_shard(sources[i], 0, states, stream)
        if apart:
            torch.cuda.synchronize()
        verify(fv, logits, draft, outs[i], theta=1.0, W=1, stream=stream)

    want = []
    for i in range(2):
        step(i, torch.cuda.current_stream().cuda_stream, apart=True)
        torch.cuda.synchronize()
        want.append(kept(outs[i]))
    assert not torch.equal(want[0][3], want[1][3])
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        with torch.cuda.graph(graph, stream=stream):
            for i in (0, 1, 1, 0, 1):
                step(i, stream.cuda_stream)
        for n in range(20):
            for out in outs:
                out.entropy.zero_()
            if n % 2:
                graph.replay()
            else:
                for i in (1, 0, 0, 1):
                    step(i, stream.cuda_stream)
            stream.synchronize()
            for i in range(2):
                assert all(torch.equal(a, b) for a, b in zip(kept(outs[i]), want[i])), (n, i)
