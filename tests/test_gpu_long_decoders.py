"""Decoders with two strided passes, sign, flip and scale included, at every cut that they have."""
import numpy as np
import pytest
import torch

import oracle
from parity import to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("L,K", [(26, 1), (27, 1), (28, 1), (29, 1), (30, 1), (31, 1), (26, 3), (28, 3), (30, 3)])
def test_entries_of_a_long_decoder(L, K):
    """64 x 4 entries, spread over the top and the low bits of the index, against the matrix definition; and the whole vector's norm,
    which the transform keeps.  Each entry is an exact integer times a factor rounded a few times: 2^-24 each, far below 1e-6."""
    import paper_2405_11095_b200 as F
    n, d, seed, step, lam, split = 1 << L, (1 << L) - 7, 5, L, 0.5, L // 2
    P = F.planes(K)
    g = torch.Generator(device=DEV).manual_seed(L + K)
    bits = torch.empty(P, n // 32, dtype=torch.int32, device=DEV)
    for p in range(P):
        torch.randint(-2**31, 2**31 - 1, (n // 32,), generator=g, device=DEV, dtype=torch.int32, out=bits[p])
    minimum = F.workspace_bytes(F.OP_DOWNLINK_DECODE, d, K=K)
    rng = np.random.default_rng(L)
    hi = np.sort(rng.choice(1 << (L - split), 64, replace=False))
    lo = np.sort(rng.choice(1 << split, 4, replace=False))
    hi[0], lo[0] = 0, 0
    hi[-1], lo[-1] = (1 << (L - split)) - 1, (1 << split) - 8
    ref = oracle.decode_grid(to_np_words(bits), n, seed, step, oracle.SERVER_ID, lam, split, hi, lo, K=K)
    at = torch.from_numpy(((hi[:, None] << split) + lo[None, :]).reshape(-1)).to(DEV)
    for factor in (1.0, 1.5):                               # the first pass in fp32 and (one plane) in fp16
        ws = torch.empty(int(minimum * factor), dtype=torch.uint8, device=DEV)
        out = torch.full((d,), 7.0, device=DEV)
        F.downlink_decode(bits, d, out, lam, seed, step, K=K, ws=ws)
        torch.cuda.synchronize()
        got = out[at].double().cpu().numpy().reshape(64, 4)
        assert np.abs(got - ref).max() <= 1e-6 * np.abs(ref).max(), factor
        if K == 1:                                          # every value is +-1 before the transform, lam^2 n after it (but for the 7 cut off)
            assert abs(float((out.double() ** 2).sum()) / (lam * lam * n) - 1) <= 1e-5
        del ws, out
    assert F.async_timeouts() == 0
