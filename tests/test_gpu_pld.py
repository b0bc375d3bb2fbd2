"""Prompt-lookup drafting on the GPU (through the C ABI) against the CPU oracle: bit-exact."""
import random

import pytest
import torch

from oracle.pld_oracle import pld_draft as oracle_pld
from paper_2511_22972_b200 import binding as Bd

pytestmark = pytest.mark.gpu
DEV = "cuda"


def run(seqs, K, mx, mn, pad_to=None):
    B = len(seqs)
    Lmax = pad_to or max(len(s) for s in seqs)
    tok = torch.full((B, Lmax), -7, dtype=torch.int32)
    for b, s in enumerate(seqs):
        tok[b, :len(s)] = torch.tensor(s, dtype=torch.int32)
    lengths = torch.tensor([len(s) for s in seqs], dtype=torch.int32)
    draft, count, pos, ng = Bd.pld_draft(tok.to(DEV), lengths.to(DEV), K, mx, mn,
                                         stream=torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for b, s in enumerate(seqs):
        prop, p, n = oracle_pld(s, K, mx, mn)
        assert count[b].item() == len(prop) and pos[b].item() == p and ng[b].item() == n, (b, s[:20])
        assert draft[b, :len(prop)].tolist() == prop and (draft[b, len(prop):] == -1).all()


def test_golden_cases_on_the_gpu():
    from tests.test_oracle_pld import golden_cases
    for toks, K, mx, mn, prop, pos, n in golden_cases():
        run([toks], K, mx, mn)


@pytest.mark.parametrize("alphabet", [2, 5, 1000, 128256])
def test_random_sequences(alphabet):
    rng = random.Random(alphabet)
    seqs = [[rng.randrange(alphabet) for _ in range(rng.choice([1, 2, 3, 17, 255, 256, 257, 1000, 4099]))] for _ in range(64)]
    for K, mx, mn in [(8, 3, 1), (25, 8, 1), (1, 1, 1), (15, 4, 2)]:
        run(seqs, K, mx, mn, pad_to=4100)


def test_long_context_with_a_planted_repeat():
    # a prompt-like sequence: 60k mostly unique tokens, the last 5 tokens copied from two earlier places
    rng = random.Random(9)
    base = [rng.randrange(10 ** 6) + 10 for _ in range(60000)]
    tail = base[40000:40005]
    base[1234:1239] = tail                       # an earlier copy: it must win over the one at 40000
    seq = base + tail
    run([seq, seq[:50000], base], 15, 5, 1)
    prop, p, n = oracle_pld(seq, 15, 5, 1)
    assert (p, n) == (1234, 5) and prop == seq[1239:1254]


def test_argument_errors():
    t = torch.zeros(1, 4, dtype=torch.int32, device=DEV)
    l = torch.ones(1, dtype=torch.int32, device=DEV)
    for K, mx, mn in [(0, 3, 1), (4, 9, 1), (4, 2, 3), (4, 3, 0)]:
        with pytest.raises(Bd.FlyError) as e:
            Bd.pld_draft(t, l, K, mx, mn)
        assert e.value.status == Bd.FLY_ERR_INVALID_ARG


def test_lengths_outside_the_row_propose_nothing_and_read_nothing_outside_it():
    # lengths is device data: a length larger than the row stride, or negative, must not steer a load past the row
    B, stride, K = 6, 64, 8
    rng = random.Random(3)
    tok = torch.tensor([[rng.randrange(4) for _ in range(stride)] for _ in range(B)], dtype=torch.int32)
    lengths = torch.tensor([stride, stride + 1, 10 ** 9, -1, -(10 ** 9), 40], dtype=torch.int32)
    draft, count, pos, ng = Bd.pld_draft(tok.to(DEV), lengths.to(DEV), K, 3, 1, stream=torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for b in (1, 2, 3, 4):
        assert count[b].item() == 0 and pos[b].item() == -1 and ng[b].item() == 0 and (draft[b] == -1).all()
    for b in (0, 5):
        prop, p, n = oracle_pld(tok[b, :lengths[b]].tolist(), K, 3, 1)
        assert count[b].item() == len(prop) and pos[b].item() == p and draft[b, :len(prop)].tolist() == prop


@pytest.mark.parametrize("L", [2, 3, 5, 4095, 4096, 4097, 8193, 32767, 32768, 33000])
@pytest.mark.parametrize("pad", [0, 1, 2, 3])
def test_matches_at_the_edges_of_segments_rounds_and_blocks(L, pad):
    # one 16-byte segment is 4 tokens, one block round 4096, one cluster round 32768; odd strides shift the segments
    n = min(3, L - 1)
    ends = sorted({e for e in (n, 4, 5, 4093, 4096, 4097, 4099, 8192, L // 2, L - 2, L - 1) if n <= e < L})
    seqs = []
    for e in ends:
        s = list(range(10, 10 + L))
        s[e - n:e] = s[L - n:]                        # the last n tokens also end just before position e
        seqs.append(s)
    stride = (L + 3) // 4 * 4 + pad
    for mx, mn in [(n, n), (5, 1)]:
        run(seqs, 8, mx, mn, pad_to=stride)


def test_contexts_written_by_the_kernel_before_in_the_stream():
    # the drafter is launched while the step before it still runs, and reads what that step writes: its out_tokens [B, K+1]
    from paper_2511_22972_b200 import FlyVerify, VerifyBuffers, verify
    B, K, V = 24, 31, 1000
    fv = FlyVerify(B, K, V, "f32")
    st = torch.cuda.current_stream().cuda_stream
    g = torch.Generator().manual_seed(5)
    steps = []
    for i in range(8):                            # tokens of a small alphabet, so that n-grams recur; every position is accepted
        y = torch.randint(0, 6, (B, K + 1), generator=g)
        logits = torch.zeros(B, K + 1, V)
        logits.scatter_(2, y[..., None], 30.0)
        steps.append((y, logits.to(DEV), y[:, :K].to(torch.int32).contiguous().to(DEV)))
    out, lengths, got = VerifyBuffers(B, K, DEV), torch.full((B,), K + 1, dtype=torch.int32, device=DEV), []
    torch.cuda.synchronize()
    for i in range(200):
        y, logits, draft = steps[i % len(steps)]
        verify(fv, logits, draft, out, theta=1.0, W=1, stream=st)
        got.append(Bd.pld_draft(out.out_tokens, lengths, 5, 4, 1, stream=st))
    torch.cuda.synchronize()
    want = [[oracle_pld(row.tolist(), 5, 4, 1) for row in y] for y, _, _ in steps]
    for i, (draft, count, pos, ng) in enumerate(got):
        for b, (prop, p, n) in enumerate(want[i % len(steps)]):
            assert (count[b].item(), pos[b].item(), ng[b].item()) == (len(prop), p, n) and draft[b, :len(prop)].tolist() == prop, (i, b)
    fv.close()


@pytest.mark.parametrize("width", [9, 4097, 8195, 32771, 70001])
def test_rows_at_every_alignment_and_lengths_around_a_round(width):
    # rows start 4, 8 and 12 bytes off a 16-byte boundary; contexts end just before, at and after what a block or a cluster of
    # blocks tests at a time; the repeat lies at the very start, across a boundary, or nowhere
    rng = random.Random(width)
    seqs = []
    for L in [1, 2, 3, 4, 5, 6, 7, 8, 9] + [width - d for d in (0, 1, 2, 3, 4, 5)] + [width // 2 + d for d in (0, 1, 2)]:
        L = max(1, min(L, width))
        s = [rng.randrange(10 ** 6) + 10 for _ in range(L)]
        n = min(rng.randrange(0, 6), L // 2)
        at = rng.choice([0, 1, 2, 3, max(0, L // 2 - n), max(0, L - 2 * n - 1), min(L, 4096) - n])
        if n > 0 and 0 <= at and at + n <= L - n:
            s[at:at + n] = s[L - n:]
        seqs.append(s)
    seqs.append([rng.randrange(3) for _ in range(width)])
    for K, mx, mn in [(15, 3, 1), (5, 8, 2)]:
        run(seqs, K, mx, mn, pad_to=width)


@pytest.mark.parametrize("slow,at", [((0,), 34000), ((0, 32768), 66000)])
def test_the_first_block_goes_on_when_others_end_first(slow, at):
    # The first block of a cluster is held up by look-backs one token short of a match, all over one or two of its rounds; the other
    # blocks have a match in a later round and end before it gets to its own, earlier one.
    query, L, B = [9] + [5] * 7, 100000, 64
    seqs = []
    for i in range(4):
        s = list(range(10, 10 + L))
        for lo in slow:
            s[lo:lo + 4096] = [5] * 4096
        for e in (at + 100 * i, *range(at + 3000, at + 3000 + 7 * 4096, 4096)):
            s[e:e + 8] = query
        s[L - 8 - i:] = query                     # (the last tokens at every alignment)
        seqs.append(s)
    want = [oracle_pld(s, 15, 8, 1) for s in seqs]
    assert [(p, n) for _, p, n in want] == [(at + 100 * i, 8) for i in range(4)]
    tok = torch.full((B, L + 1), -7, dtype=torch.int32)
    for b in range(B):
        tok[b, :len(seqs[b % 4])] = torch.tensor(seqs[b % 4], dtype=torch.int32)
    lengths = torch.tensor([len(seqs[b % 4]) for b in range(B)], dtype=torch.int32, device=DEV)
    tok, st = tok.to(DEV), torch.cuda.current_stream().cuda_stream
    got = [Bd.pld_draft(tok, lengths, 15, 8, 1, stream=st) for _ in range(20)]
    torch.cuda.synchronize()
    for draft, count, pos, ng in got:
        assert pos.tolist() == [want[b % 4][1] for b in range(B)] and ng.tolist() == [8] * B and count.tolist() == [15] * B
        assert draft.tolist() == [want[b % 4][0] for b in range(B)]


@pytest.mark.parametrize("L", [32800, 40000, 65560, 131072])
@pytest.mark.parametrize("pad", [0, 1, 2, 3])
def test_contexts_that_end_in_a_run_of_one_token(L, pad):
    # The tokens behind the last whole 16-byte segment are tested first and match the longest query; the earliest match lies in a
    # later round of the first block of the cluster, or in one of another block.
    seqs, cases = [], []
    for mx in (1, 3, 8):
        for at in (32770, 36850, 45000, 65540, 69620):
            if at + mx > L - 16:
                continue
            n = L - len(seqs) % 4                 # (the last tokens at every alignment)
            s = list(range(10, 10 + n))
            s[at:at + mx] = [7] * mx
            s[n - mx - 3:] = [7] * (mx + 3)
            seqs.append(s)
            cases.append((mx, at))
    for mx in (1, 3, 8):
        run([s for s, c in zip(seqs, cases) if c[0] == mx], 8, mx, 1, pad_to=(L + 3) // 4 * 4 + pad)
    assert all(oracle_pld(s, 8, mx, 1)[1:] == (at, mx) for s, (mx, at) in zip(seqs, cases))


def test_the_allocation_of_the_results_is_seen_by_modes_and_the_profiler():
    from torch.profiler import ProfilerActivity, profile
    from torch.utils._python_dispatch import TorchDispatchMode

    class Log(TorchDispatchMode):
        seen = []

        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            self.seen.append(str(func))
            return func(*args, **(kwargs or {}))
    tok = torch.randint(0, 9, (3, 100), dtype=torch.int32, device=DEV)
    lengths, st = torch.full((3,), 100, dtype=torch.int32, device=DEV), torch.cuda.current_stream().cuda_stream
    want = Bd.pld_draft(tok, lengths, 5, 3, 1, stream=st)
    with Log() as log:
        logged = Bd.pld_draft(tok, lengths, 5, 3, 1, stream=st)
    assert log.seen.count("aten.empty.memory_format") == 4, log.seen
    with profile(activities=[ProfilerActivity.CPU]) as prof:
        profiled = Bd.pld_draft(tok, lengths, 5, 3, 1, stream=st)
    assert sum(e.name == "aten::empty" for e in prof.events()) == 4
    for got in (logged, profiled):
        assert all(torch.equal(a, b) and a.stride() == b.stride() for a, b in zip(got, want))
