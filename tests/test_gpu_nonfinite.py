"""Transforms with entries that are not finite: which way their signs fall, and that they stay within their transform."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def F():
    import paper_2405_11095_b200 as f
    return f


def counts(words, P):
    """Planes [P, d'/32] -> count of every coordinate."""
    w = words.cpu().numpy().view(np.uint32).reshape(P, -1, 1)
    bit = (w >> np.arange(32, dtype=np.uint32)) & 1
    return (bit << np.arange(P, dtype=np.uint32)[:, None, None]).sum(axis=0).reshape(-1)


@pytest.mark.parametrize("b,nan_counts", [(5, False), (8, False), (9, False), (10, True), (13, True)])
@pytest.mark.parametrize("K", [1, 3, 8, 255])
def test_signs_of_what_is_not_a_number(F, b, nan_counts, K):
    """A block with a NaN has nothing but NaN before the sign: in transforms shorter than 2^10 no dithered value of it counts as
    non-negative, in longer ones every one does.  An infinity leaves infinities of either sign, whose counts are 0 or K.  The finite
    block beside them is encoded as if it were alone."""
    n, seed, step = 1 << b, 3, 1
    d = 3 * n
    g = torch.randn(d, generator=torch.Generator().manual_seed(b))
    alone = g.clone()
    g[n + 7] = float("nan")
    g[2 * n + 5] = float("inf")
    P, dp = F.planes(K), F.padded_dim(d, b)
    down, ref = (torch.zeros(P, dp // 32, dtype=torch.int32, device=DEV) for _ in range(2))
    F.downlink_encode(g.to(DEV), d, down, 0.5, seed, step, K=K, block_log2=b)
    F.downlink_encode(alone.to(DEV), d, ref, 0.5, seed, step, K=K, block_log2=b)
    torch.cuda.synchronize()
    c, r = counts(down, P), counts(ref, P)
    assert (c[:n] == r[:n]).all()
    assert (c[n:2 * n] == (K if nan_counts else 0)).all()
    assert set(np.unique(c[2 * n:])) == {0, K}
