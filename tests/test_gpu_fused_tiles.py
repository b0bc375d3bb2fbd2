"""The fused path's operand ring and vocabulary tiles where their shape changes: one and two slices of the hidden dimension per stage, an
odd number of slices, tiles of fewer than 256 entries (a weight stored [V, D], few positions) with halves that are no multiple of 16,
ragged last tiles, and the lines at which either is chosen."""
import pytest
import torch

from oracle import fly_oracle as O
from paper_2511_22972_b200 import FlyVerify, VerifyBuffers, binding as Bd, verify_fused
from tests._parity import assert_parity
from tests.test_gpu_fused import DEV, fused_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,K,D,V", [
    (1, 1, 64, 8), (2, 3, 64, 640), (4, 8, 136, 1000), (4, 8, 200, 4096),         # one slice, three, a ragged fourth; tiles of 128
    (3, 4, 128, 9472), (3, 4, 128, 9480),                                         # 37 tiles of 256, 38
    (2, 3, 3072, 9984), (2, 3, 3008, 9984),                                       # 48 slices, 47
    (4, 3, 72, 19000), (4, 3, 64, 20480), (8, 1, 64, 30304), (8, 1, 64, 30312),   # two rounds; 119 tiles of 148 are more than 80 %
    (9, 7, 320, 20008), (5, 12, 320, 20008), (16, 8, 192, 20008), (29, 4, 192, 20008)])   # 72 positions, 65, 144, 145
@pytest.mark.parametrize("vocab_major", [True, False])
def test_ring_and_tiles(B, K, D, V, vocab_major):
    w, hidden, weight, draft, logits = fused_case(B, K, D, V)
    fv, out = FlyVerify(B, K, V, "bf16", hidden=D), VerifyBuffers(B, K, DEV)
    fv.set_weight_layout(vocab_major)
    if vocab_major:
        weight = weight.t().contiguous()
    ref = O.verify_batch(logits.reshape(B, K + 1, V), draft.cpu().numpy(), 1.0, 1)
    stream = torch.cuda.current_stream().cuda_stream
    for again in range(2):
        verify_fused(fv, hidden, weight, draft, out, theta=1.0, W=1, stream=stream)
        assert fv.device_status(stream) == Bd.FLY_OK
        assert_parity(out, ref, f"{B}x{K} D={D} V={V} {'VD' if vocab_major else 'DV'}")
    # fewer positions on the same handle: another tile, another map of the same weight
    if B > 1:
        n = (K + 1) * (B // 2)
        part = VerifyBuffers(B // 2, K, DEV)
        verify_fused(fv, hidden[:n].contiguous(), weight, draft[:B // 2].contiguous(), part, theta=1.0, W=1, stream=stream)
        assert fv.device_status(stream) == Bd.FLY_OK
        ref = O.verify_batch(logits[:n].reshape(B // 2, K + 1, V), draft[:B // 2].cpu().numpy(), 1.0, 1)
        assert_parity(part, ref, "half of the batch")
    fv.close()
