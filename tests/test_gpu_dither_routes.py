"""K dithers on either side of the lines between their two kernels: the same counts for the blocks that both calls have."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("b,few,more,Ks", [
    (14, 74, 75, (2, 7, 8, 15, 23, 24)),       # two blocks to a tile; one
    (13, 74, 75, (3, 8, 16, 17, 23)),
    (10, 512, 513, (3, 7, 8)),                 # overlapped launch; the ordinary one
    (12, 128, 1025, (7, 8, 15)),
    (10, 8191, 8192, (23, 24, 27, 28)),        # dithers shared among warps; in registers up to 28 of them
])
def test_counts_do_not_depend_on_the_route(b, few, more, Ks):
    import paper_2405_11095_b200 as F
    d = more << b
    g = torch.randn(d, generator=torch.Generator(device=DEV).manual_seed(b + more), device=DEV)
    for K in Ks:
        P = F.planes(K)
        planes = []
        for n in (few, more):
            down = torch.full((P, (n << b) // 32), -1, dtype=torch.int32, device=DEV)
            F.downlink_encode(g[: n << b], n << b, down, 0.75, 3, 1, K=K, block_log2=b)
            planes.append(down[:, : (few << b) // 32])
        torch.cuda.synchronize()
        assert torch.equal(*planes), K
