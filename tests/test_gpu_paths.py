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
    ((9 << 16) + 31, 2, 16),           # a cluster of thread blocks holds the block
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


def assert_bits_near_ties(words, ref, margin, lam, K):
    """As assert_bits_match, with a count that holds for any K and short vectors: a bit may differ only where the oracle's
    pre-sign value lies within 1e-5 lam of a tie.  A dither is uniform over 2 lam, so each of the K comparisons of a
    coordinate falls into that band with probability at most 1e-5; six sigma above the mean."""
    diff = np.zeros(ref.shape[-1], np.uint32)
    for p in range(ref.shape[0]):
        diff |= words.reshape(ref.shape)[p] ^ ref[p]
    bad = oracle.unpack(diff).astype(bool)
    assert (margin[bad] <= 1e-5 * lam).all(), margin[bad].max() / lam
    mean = 1e-5 * K * bad.size
    assert bad.sum() <= mean + 6 * np.sqrt(mean) + 1


@pytest.mark.parametrize("d,b,Ks", [
    (300, 0, (1, 2, 255)),                # one warp
    (5000, 0, (7, 8, 9, 24, 255)),        # one tile: its groups of dithers shared among blocks; threshold form from 8 on
    (70_000, 0, (3, 23, 24)),             # strided pass before it, sixteen tiles
    ((1 << 23) - 31, 10, (7, 24)),        # tiles enough to fill the chip by themselves: fewer than 24 dithers, and more
    ((1 << 25) - 3, 0, (3, 9)),           # tiles of 2^15: pairs of halves
    ((1 << 26) + 5, 0, (3,)),             # several planes through two strided passes
])
def test_dithers_and_planes_of_the_downlink(F, d, b, Ks):
    """fosgd_downlink_encode and fosgd_downlink_decode for K around each switch of the kernels."""
    seed, step = 17, 3
    dp, n_eff = F.padded_dim(d, b), F.transform_len(d, b)
    gbar = torch.zeros(dp, device=DEV)
    gbar[:d] = gradients(d, 1, torch.float32)[0, :d]
    gh = gbar.cpu().double().numpy()
    lam_s = oracle.lam_server(oracle.lam(float(np.linalg.norm(gh)), 2.0, n_eff), 2.0, n_eff)
    amp = torch.tensor([lam_s], device=DEV)
    for K in Ks:
        P = F.planes(K)
        ws = torch.empty(max(16, F.workspace_bytes(F.OP_DOWNLINK_DECODE, d, block_log2=b, K=K) * 3 // 2), dtype=torch.uint8, device=DEV)
        down = torch.full((P, dp // 32), -1, dtype=torch.int32, device=DEV)
        out = torch.full((d,), 7.0, device=DEV)
        F.downlink_encode(gbar, d, down, amp, seed, step, K=K, block_log2=b, ws=ws)
        F.downlink_decode(down, d, out, lam_s, seed, step, K=K, block_log2=b, ws=ws)
        torch.cuda.synchronize()
        lam32 = float(amp.item())
        if dp * K <= 1 << 28:
            ref, margin = oracle.downlink_encode(gh[:d] if b == 0 else gh, seed, step, lam32, K=K, block_log2=b, want_margin=True)
            assert_bits_near_ties(to_np_words(down), ref, margin, lam32, K)
        ref = oracle.downlink_decode(to_np_words(down), dp, seed, step, lam_s, K=K, block_log2=b)
        assert_l2_close(out.cpu().numpy(), ref[:d])


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("L", [10, 14, 15, 16, 18, 20, 21, 22, 23, 25])
def test_encoder_on_ragged_lengths(F, L, dtype):
    """Each cut of the encoder on a length that is odd and ends inside a row, for two workers: zero bits of the flattened
    vector differ from the oracle's but at ties."""
    d, seed, step = (1 << L) * 5 // 8 + 33, 23, L
    grads = gradients(d, 2, dtype)
    ws = torch.empty(max(16, 2 * F.workspace_bytes(F.OP_ENCODE, d)), dtype=torch.uint8, device=DEV)
    bits = torch.zeros(2, (1 << L) // 32, dtype=torch.int32, device=DEV)
    x = grads[1, :d].cpu().double().numpy()
    lam = oracle.lam(float(np.linalg.norm(x)), 2.0, 1 << L)
    F.encode(grads, d, bits, lam, seed, step, ws=ws, worker_stride=grads.shape[1])
    torch.cuda.synchronize()
    ref, margin = oracle.encode(x, seed, step, 1, lam, want_margin=True)
    assert_bits_near_ties(to_np_words(bits[1]), ref, margin, lam, 1)


@pytest.mark.parametrize("d,M", [(1000, 148), (1000, 149), (1 << 16, 18), ((1 << 16) - 5, 19), (10_000, 148), (10_000, 149)])
def test_encoder_of_as_many_blocks_as_processors(F, d, M):
    """Dither words made before or after the wait for the kernel in front (up to a block per processor, 148 of them): the
    first and last worker against the oracle, and the same words from single-worker calls."""
    seed, step = 29, d
    grads = gradients(d, M, torch.float32)
    dp = F.padded_dim(d)
    ws = torch.empty(max(16, M * F.workspace_bytes(F.OP_ENCODE, d)), dtype=torch.uint8, device=DEV)
    bits, one = torch.zeros(2, M, dp // 32, dtype=torch.int32, device=DEV)
    x = grads[:, :d].cpu().double().numpy()
    lam = oracle.lam(float(np.linalg.norm(x[M - 1])), 2.0, dp)
    F.encode(grads, d, bits, lam, seed, step, ws=ws, worker_stride=grads.shape[1])
    for n in (0, 1, M - 1):
        F.encode(grads[n], d, one[n], lam, seed, step, worker_id0=n, ws=ws, worker_stride=grads.shape[1])
    torch.cuda.synchronize()
    for n in (0, 1, M - 1):
        assert torch.equal(bits[n], one[n])
        ref, margin = oracle.encode(x[n], seed, step, n, lam, want_margin=True)
        assert_bits_near_ties(to_np_words(bits[n]), ref, margin, lam, 1)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d,M", [(1 << 19, 3), ((1 << 19) + 1, 1), ((9 << 16) - 2345, 2), ((7 << 16) + 1, 2), ((7 << 16) - 3, 2)])
def test_encoder_of_blocks_of_2p16(F, d, M, dtype):
    """The one-kernel form (from eight blocks on) and the two-kernel form against the oracle, and batches against single
    workers word for word."""
    seed, step, b = 31, 2, 16
    grads = gradients(d, M, dtype)
    dp, stride = F.padded_dim(d, b), grads.shape[1]
    ws = torch.empty(M * F.workspace_bytes(F.OP_ENCODE, d, block_log2=b), dtype=torch.uint8, device=DEV)
    bits, one = torch.zeros(2, M, dp // 32, dtype=torch.int32, device=DEV)
    x = grads[:, :d].double().cpu().numpy()
    lam = oracle.lam(float(np.linalg.norm(x[M - 1])) / 3, 2.0, 1 << b)
    with F.PassTrace() as tr:
        F.encode(grads, d, bits, lam, seed, step, worker_id0=3, block_log2=b, ws=ws, worker_stride=stride)
    torch.cuda.synchronize()
    assert any(lab.startswith("cluster") for lab in tr.labels) == (dp >= 1 << 19), tr.labels
    for n in range(M):
        F.encode(grads[n], d, one[n], lam, seed, step, worker_id0=3 + n, block_log2=b, ws=ws, worker_stride=stride)
    torch.cuda.synchronize()
    assert torch.equal(bits, one)
    ref, margin = oracle.encode(x[M - 1], seed, step, 2 + M, lam, block_log2=b, want_margin=True)
    assert_bits_near_ties(to_np_words(bits[M - 1]), ref, margin, lam, 1)


@pytest.mark.parametrize("d,b,M", [
    (700, 0, 9), (9000, 0, 2), (9000, 0, 33),        # one tile: up to eight blocks of a cluster share the workers
    (40_000, 0, 5), (40_000, 0, 1), (40_000, 0, 16), (40_000, 0, 17),     # top stages as counts of bits, up to 2^20 in all
    (100_000, 16, 3), (1 << 17, 0, 8), (200_000, 18, 2), ((1 << 18) - 1, 0, 4),
    (300_000, 0, 7), (300_000, 14, 3),
    (1 << 20, 0, 3), (1 << 20, 0, 128),              # ten strided stages; 64 tiles for the tensor-core pass, workers split
    (3 << 20, 20, 11), ((1 << 21) - 9, 0, 64),       # items that do not divide among the blocks
    ((1 << 25) - 5, 0, 2), ((1 << 25) - 5, 0, 5),    # pairs of halves, without and with the tensor-core pass
])
def test_workers_shared_among_blocks(F, d, b, M):
    """The averaged decoder against the oracle, with one amplitude and with one per worker and block."""
    seed, step = 3, 8
    dp = F.padded_dim(d, b)
    g = torch.Generator(device=DEV).manual_seed(d + M)
    bits = torch.randint(-2**31, 2**31, (M, dp // 32), generator=g, device=DEV, dtype=torch.int64).to(torch.int32)
    words = to_np_words(bits)
    ws = torch.empty(max(16, M * F.workspace_bytes(F.OP_AGGREGATE, d, M=M, block_log2=b)), dtype=torch.uint8, device=DEV)
    acc = torch.empty(dp, device=DEV)
    F.server_aggregate(bits, d, acc, 0.25, seed, step, worker_id0=1, block_log2=b, ws=ws)
    torch.cuda.synchronize()
    if M * dp <= 1 << 27:
        assert_l2_close(acc.cpu().numpy(), oracle.aggregate(words, d, seed, step, 0.25, 1, b))
    if b:
        lam = torch.rand(M, dp >> b, generator=g, device=DEV) + 0.5
        accw = torch.empty(dp, device=DEV)
        one = torch.empty(dp, device=DEV)
        F.server_aggregate_dev(bits, d, accw, lam, seed, step, worker_id0=1, block_log2=b, per_block=True, ws=ws)
        F.server_aggregate_dev(bits[:1], d, one, lam[:1].contiguous(), seed, step, worker_id0=1, block_log2=b, per_block=True, ws=ws)
        torch.cuda.synchronize()
        table = lam.cpu().double().numpy()
        assert_l2_close(accw.cpu().numpy(), oracle.aggregate(words, d, seed, step, table, 1, b))
        assert_l2_close(one.cpu().numpy(), oracle.aggregate(words[:1], d, seed, step, table[:1], 1, b))
    assert F.async_timeouts() == 0


@pytest.mark.parametrize("L,K", [(26, 1), (27, 1), (28, 1), (29, 1), (30, 1), (28, 3), (30, 3)])
def test_decoder_cuts_of_long_transforms(F, L, K):
    """Magnitudes of every decoded coordinate of 2^26 .. 2^30 against a transform in fp64, and one entry, with its sign and
    scale, against the oracle."""
    n, d, seed, step, lam = 1 << L, (1 << L) - 7, 5, L, 0.5
    P = F.planes(K)
    g = torch.Generator(device=DEV).manual_seed(L + K)
    bits = torch.randint(-2**31, 2**31, (P, n // 32), generator=g, device=DEV, dtype=torch.int64).to(torch.int32)
    if P > 1:        # counts of 0 .. K
        assert K == 3
    ws = torch.empty(F.workspace_bytes(F.OP_DOWNLINK_DECODE, d, K=K) * 3 // 2, dtype=torch.uint8, device=DEV)
    out = torch.empty(d, device=DEV)
    F.downlink_decode(bits, d, out, lam, seed, step, K=K, ws=ws)
    del ws
    y = torch.full((n,), -float(K), dtype=torch.float64, device=DEV)
    for p in range(P):
        for k in range(32):
            y.view(-1, 32)[:, k] += ((bits[p] >> k) & 1).double() * (2 << p)
    half = 1
    while half < n:
        v = y.view(-1, 2, half)
        a = v[:, 0].clone()
        v[:, 0] += v[:, 1]
        torch.sub(a, v[:, 1], out=v[:, 1])
        half *= 2
        del a
    y = y[:d].abs_()
    mag = out.abs().double()
    scale = float(mag.norm() / y.norm())
    assert float((mag - scale * y).norm()) <= 1e-5 * float(mag.norm())
    if L <= 28:
        k = 12_345_678
        ref = oracle.decode_entry(to_np_words(bits), n, seed, step, oracle.SERVER_ID, lam, k, K=K)
        assert abs(float(out[k]) - ref) <= 1e-5 * abs(ref) + 1e-6 * float(mag.mean())
