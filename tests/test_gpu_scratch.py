"""Averages of more workers than the scratch holds: the same sums, whatever a launch takes at a time."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("d,b,M", [((1 << 16) - 1, 0, 8), ((1 << 19) - 5, 0, 8), ((1 << 20) + 1, 0, 7), (3 << 18, 18, 9), ((1 << 22) - 9, 22, 8),
                                   ((1 << 25) - 3, 0, 6), ((1 << 26) - 3, 0, 3)])
def test_scratch_for_fewer_workers(d, b, M):
    import paper_2405_11095_b200 as F
    dp = F.padded_dim(d, b)
    bits = torch.randint(-2**31, 2**31 - 1, (M, dp // 32), generator=torch.Generator(device=DEV).manual_seed(M), device=DEV, dtype=torch.int32)
    need = F.workspace_bytes(F.OP_AGGREGATE, d, block_log2=b)
    ws = torch.empty(M * need, dtype=torch.uint8, device=DEV)
    outs = []
    for have in (M, 1, 2, 3, 5):
        acc = torch.full((dp,), 7.0, device=DEV)
        F.server_aggregate(bits, d, acc, 0.5, 3, 1, worker_id0=2, block_log2=b, ws=ws[: min(have, M) * need])
        outs.append(acc)
    torch.cuda.synchronize()
    assert all(torch.equal(outs[0], x) for x in outs[1:])
    assert F.async_timeouts() == 0
