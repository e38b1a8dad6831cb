"""Zeros of a decoder: the same bits whichever kernel makes them."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("d,b,K", [(300, 0, 1), (1 << 10, 0, 1), ((1 << 13) - 5, 0, 3), (1 << 15, 0, 1), (1 << 16, 0, 1), (1 << 17, 0, 3),
                                   (3 << 18, 18, 1), (1 << 20, 0, 1), (1 << 24, 0, 1), (1 << 25, 0, 1), (1 << 26, 0, 1)])
def test_a_decoded_zero_is_positive(d, b, K):
    """A sum starts from +0, so no flip leaves -0 behind: a server's only worker, and the downlink's decoder."""
    import paper_2405_11095_b200 as F
    dp, P = F.padded_dim(d, b), F.planes(K)
    bits = torch.full((P, dp // 32), -1, dtype=torch.int32, device=DEV)      # all ones: each transform is zero but for its first entry
    ws = torch.empty(max(16, F.workspace_bytes(F.OP_DOWNLINK_DECODE, d, block_log2=b, K=K)), dtype=torch.uint8, device=DEV)
    out, acc = torch.full((d,), 7.0, device=DEV), torch.full((dp,), 7.0, device=DEV)
    F.downlink_decode(bits, d, out, 0.5, 3, 1, K=K, block_log2=b, ws=ws)
    outs = [out]
    if K == 1:
        F.server_aggregate(bits, d, acc, 0.5, 3, 1, block_log2=b, ws=ws)
        outs.append(acc)
    torch.cuda.synchronize()
    for x in outs:
        zero = x == 0
        assert int(zero.sum()) == x.numel() - len(range(0, x.numel(), F.transform_len(d, b))) and not bool(torch.signbit(x[zero]).any())
