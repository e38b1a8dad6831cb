"""Two workers in blocks of 2^22, on either side of the line between the two cuts."""
import pytest
import torch

import oracle
from parity import assert_l2_close, to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("blocks", [1, 2, 3, 8])
def test_average_of_two_workers(blocks):
    import paper_2405_11095_b200 as F
    b, d, seed, step = 22, (blocks << 22) - 5, 7, blocks
    dp = F.padded_dim(d, b)
    bits = torch.randint(-2**31, 2**31 - 1, (2, dp // 32), generator=torch.Generator(device=DEV).manual_seed(blocks), device=DEV, dtype=torch.int32)
    acc = torch.full((dp,), 7.0, device=DEV)
    ws = torch.empty(2 * F.workspace_bytes(F.OP_AGGREGATE, d, block_log2=b), dtype=torch.uint8, device=DEV)
    with F.PassTrace() as tr:
        F.server_aggregate(bits, d, acc, 0.5, seed, step, worker_id0=3, block_log2=b, ws=ws)
    torch.cuda.synchronize()
    assert any(x.startswith("row12" if blocks > 2 else "row14") for x in tr.labels), tr.labels
    assert_l2_close(acc.cpu().numpy(), oracle.aggregate(to_np_words(bits), d, seed, step, 0.5, 3, b))
