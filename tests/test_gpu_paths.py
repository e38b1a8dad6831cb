"""The branches of the launch plans at the sizes where they change: each against the oracle, or bit for bit against the
calls that a combined entry point stands for."""
import numpy as np
import pytest
import torch

import oracle
from parity import assert_bits_match, assert_l2_close, to_np_words

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def F():
    import paper_2405_11095_b200 as f
    return f


def gradients(d, M, dtype, pad=8, seed=0):
    """[M, stride] with worker n scaled by 1 + n; the rows start `pad`-aligned."""
    g = torch.Generator(device=DEV).manual_seed(d % 99991 + 31 * M + seed)
    x = torch.randn(M, (d + pad - 1) // pad * pad, generator=g, device=DEV)
    return (x * (1 + torch.arange(M, device=DEV)[:, None])).to(dtype)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d,M,b", [
    (1000, 3, 6),                      # below 2^10: norm pass, then the encoder
    (5 * 1024 + 1, 2, 10),             # one warp per block
    (3 * 2048, 33, 11),
    (7 * 4096 - 5, 2, 12),
    (2 * (1 << 15) + 77, 2, 15),       # largest block of one thread block
    (3 * (1 << 16) + 9, 3, 16),        # strided passes that carry the sums: up to 2^22 (eight stages)
    (2 * (1 << 17) - 3, 2, 17),
    ((1 << 18) + 4099, 2, 18),
    (2 * (1 << 20), 2, 20),
    ((1 << 22) + 12345, 2, 22),
    ((1 << 23) - 1, 2, 23),
])
def test_encode_measured_blocks_equals_amplitudes_then_encode(F, d, M, b, dtype):
    """The same amplitudes as fosgd_amplitudes (their sums are taken in another order: fp32 within at most 512 terms of
    one sign, so 512 * 2^-24 / 2 relative at the worst and ~1e-6 in practice on the root), the same packed words
    for the amplitudes that it wrote, and those words against the oracle."""
    seed, step = 91, 6
    dp = F.padded_dim(d, b)
    grads = gradients(d, M, dtype)
    grads[M - 1, : min(d, 1 << b)] = 0                                    # a block of zeros
    stride = grads.shape[1]
    nb = dp >> b
    ws = torch.empty(max(16, F.workspace_bytes(F.OP_ENCODE, d, block_log2=b) * M), dtype=torch.uint8, device=DEV)
    amp_ws = torch.empty(F.workspace_bytes(F.OP_BLOCK_AMPLITUDES, d, M=M, block_log2=b), dtype=torch.uint8, device=DEV)
    lam1, lam2 = torch.full((2, M, nb), 7.0, device=DEV)
    lam_s1, lam_s2 = torch.full((2, nb), 7.0, device=DEV)
    bits1, bits2 = torch.zeros(2, M, dp // 32, dtype=torch.int32, device=DEV)
    F.encode_measured_blocks(grads, d, bits1, lam1, lam_s1, seed, step, alpha=2.0, alpha_s=3.0, worker_id0=4, block_log2=b,
                             ws=ws, amp_ws=amp_ws, worker_stride=stride)
    F.amplitudes(grads, d, lam2, lam_s2, alpha=2.0, alpha_s=3.0, block_log2=b, per_block=True, ws=amp_ws, worker_stride=stride)
    F.encode_dev(grads, d, bits2, lam1, seed, step, worker_id0=4, block_log2=b, per_block=True, ws=ws, worker_stride=stride)
    torch.cuda.synchronize()
    assert torch.allclose(lam1, lam2, rtol=2e-6, atol=0) and torch.allclose(lam_s1, lam_s2, rtol=2e-6, atol=0)
    x = torch.zeros(M, dp, dtype=torch.float64, device=DEV)
    x[:, :d] = grads[:, :d].double()
    n_eff = float(1 << b)
    ref = (2.0 * np.sqrt(np.log(n_eff) / n_eff) * x.view(M, nb, -1).norm(dim=2)).clamp_min(1e-30)
    assert torch.allclose(lam1.double(), ref, rtol=2e-6, atol=0)
    assert torch.equal(bits1, bits2)
    n = 0
    table = lam1[n].double().cpu().numpy()
    words, margin = oracle.encode(grads[n, :d].double().cpu().numpy(), seed, step, 4 + n, table, block_log2=b, want_margin=True)
    assert_bits_match(to_np_words(bits1[n])[None], words, margin, np.repeat(table, 1 << b))
