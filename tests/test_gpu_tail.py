"""The end of a logits step, by one warp or by the whole block, at the sizes where the one hands over to the other: as many rows and
parts as a warp has lanes, one more, and several short sequences that one block completes."""
import numpy as np
import pytest
import torch

from oracle import fly_oracle as O
from paper_2511_22972_b200 import FlyVerify, VerifyBuffers, binding as Bd, synthetic as S
from tests._parity import assert_parity, check, draw

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,K,V,pieces", [
    (3, 31, 2000, 1), (3, 32, 2000, 1), (40, 50, 600, 1),   # 32 rows are a warp's, 33 are not
    (3, 15, 4096, 2), (3, 16, 4096, 2),        # two lanes a row
    (3, 7, 8704, 4), (3, 7, 8704, 5),          # four
    (2, 1, 8704, 16), (2, 1, 8704, 17),        # sixteen
    (700, 1, 1003, 0), (650, 2, 1000, 0), (300, 7, 520, 0)])   # four or eight rows per block: one sequence or several, or parts of them
def test_warp_and_block_tails(B, K, V, pieces):
    w = S.shrink(S.SERVING, B=B, K=K, V=V)
    logits, draft = draw(w, step=K)
    if pieces:
        assert Bd.plan(148, w.rows, V, "bf16", forced_pieces=pieces).slots == pieces
    else:
        assert Bd.plan(148, w.rows, V, "bf16").units_per_block in (4 * (V // 8), 8 * (V // 8))
    fv = FlyVerify(B, K, V, "bf16")
    fv.set_splits(pieces)
    W = min(2, K)
    check(fv, logits, draft, 1.0, W, what="reject")
    rng = np.random.default_rng(B + K)
    state = np.stack([rng.integers(0, W + 1, B), rng.integers(1, K + 1, B), rng.integers(0, V, B)], axis=1).astype(np.int32)
    state[state[:, 0] == 0] = [0, 0, -1]
    state[0] = [K + 1, 1, 0]                   # no state that a step writes
    check(fv, logits, draft, 0.5, W, boundary="carry", state=state, what="carry")
    # the caller's tokens, some of them invalid
    target = logits.float().argmax(-1).to(torch.int32)
    pick = torch.from_numpy(rng.random(target.shape) < 0.3).to(DEV)
    target[pick] = torch.from_numpy(rng.integers(-1, V + 1, int(pick.sum()))).to(DEV, torch.int32)
    out = VerifyBuffers(B, K, DEV)
    stream = torch.cuda.current_stream().cuda_stream
    fv.run(fv.make_args(B, K, draft, out.accept_len, out.out_tokens, logits=logits, theta=1.0, W=W, state_out=out.state,
                        rollback=out.rollback, target_argmax=out.target_argmax, entropy=out.entropy, row_flags=out.row_flags,
                        target_tokens=target), stream)
    torch.cuda.synchronize()
    ref = O.verify_batch(logits.double().cpu().numpy(), draft.cpu().numpy(), 1.0, W, target_tokens=target.cpu().numpy())
    assert_parity(out, ref, "caller's tokens")
