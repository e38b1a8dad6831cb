"""Amplitudes measured on the device, over the range of exponents that gradients can have: every kernel that takes sums of
squares, against a norm in fp64.

The squares of entries near 1e-24 vanish in fp32 and those near 1e20 overflow, while both norms are ordinary fp32 numbers.  Sums
in fp64 leave the amplitude with the rounding of its conversion to fp32, 2^-24 relative; the tolerance is twice that."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"
RTOL = 2.0 ** -23
SCALES = (1e-24, 1.0, 1e20)


@pytest.fixture(scope="module")
def F():
    import paper_2405_11095_b200 as f
    return f


def scaled(M, d, dtype, scale_of):
    """[M, stride] normal entries, coordinate i of worker n times scale_of(n, i)."""
    g = torch.Generator(device=DEV).manual_seed(d + M)
    x = torch.randn(M, (d + 7) // 8 * 8, generator=g, device=DEV)
    i = torch.arange(x.shape[1], device=DEV)
    s = torch.tensor(SCALES, device=DEV)
    return (x * s[torch.stack([scale_of(n, i) % len(SCALES) for n in range(M)])]).to(dtype)


def norms(grads, d, dp, b):
    """[M, d' >> b] norms in fp64."""
    x = torch.zeros(grads.shape[0], dp, dtype=torch.float64, device=DEV)
    x[:, :d] = grads[:, :d].double()
    return x.view(grads.shape[0], dp >> b, -1).norm(dim=2)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d,M,b", [
    (3 * 512 - 7, 2, 9), (9 * 1024 + 1, 2, 10), (5 * (1 << 13) - 3, 3, 13), (3 * (1 << 15) + 77, 2, 15),
    ((1 << 24) + 5, 1, 10), ((1 << 24) + 5, 1, 15),   # long inputs: by segments, where shorter ones go by tiles
    (3 * (1 << 16) + 9, 2, 16),                    # the strided pass carries the sums: four stages, ..
    ((9 << 16) + 31, 2, 16),                       # a cluster of thread blocks holds the block
    (3 * (1 << 17) - 3, 2, 17), (3 << 20, 2, 20), ((1 << 22) + 12345, 2, 22), ((1 << 23) - 1, 2, 23),   # .. up to eight; none
])
def test_block_amplitudes_at_the_ends_of_the_range(F, d, M, b, dtype):
    dp, n = F.padded_dim(d, b), float(1 << b)
    nb = dp >> b
    grads = scaled(M, d, dtype, lambda w, i: (i >> b) + w)
    stride = grads.shape[1]
    need = F.workspace_bytes(F.OP_ENCODE, d, block_log2=b)
    amp_ws = torch.empty(F.workspace_bytes(F.OP_BLOCK_AMPLITUDES, d, M=M, block_log2=b), dtype=torch.uint8, device=DEV)
    ref = (2.0 * np.sqrt(np.log(n) / n) * norms(grads, d, dp, b)).clamp_min(1e-30)
    ref_s = 3.0 * np.sqrt(np.log(n)) * ref.max(dim=0).values
    got = {}
    for name, workers in (("all", M), ("one", 1)):          # scratch for all workers, and for one
        ws = torch.empty(max(16, need * workers), dtype=torch.uint8, device=DEV)
        lam, lam_s = torch.full((M, nb), 7.0, device=DEV), torch.full((nb,), 7.0, device=DEV)
        bits, again = torch.zeros(2, M, dp // 32, dtype=torch.int32, device=DEV)
        F.encode_measured_blocks(grads, d, bits, lam, lam_s, 5, 1, alpha=2.0, alpha_s=3.0, block_log2=b, ws=ws, amp_ws=amp_ws,
                                 worker_stride=stride)
        F.encode_dev(grads, d, again, lam, 5, 1, block_log2=b, per_block=True, ws=ws, worker_stride=stride)
        torch.cuda.synchronize()
        assert torch.equal(bits, again)
        got[name] = lam, lam_s
    lam, lam_s = torch.full((M, nb), 7.0, device=DEV), torch.full((nb,), 7.0, device=DEV)
    F.amplitudes(grads, d, lam, lam_s, alpha=2.0, alpha_s=3.0, block_log2=b, per_block=True, ws=amp_ws, worker_stride=stride)
    torch.cuda.synchronize()
    got["amplitudes"] = lam, lam_s
    for name, (lam, lam_s) in got.items():
        assert torch.allclose(lam.double(), ref, rtol=RTOL, atol=0), (name, ((lam.double() - ref) / ref).abs().max())
        # (the server's amplitude is made from the rounded ones, and rounded itself)
        assert torch.allclose(lam_s.double(), ref_s, rtol=2 * RTOL, atol=0), name


@pytest.mark.parametrize("scale", range(len(SCALES)))
@pytest.mark.parametrize("L", [12, 16, 17, 20, 22, 24, 25])
def test_one_amplitude_at_the_ends_of_the_range(F, L, scale):
    """Global mode: one amplitude for all workers (2^17 .. 2^24: the strided pass carries the sums where scratch allows)."""
    d, M, n = (1 << L) - 3, 2, float(1 << L)
    grads = scaled(M, d, torch.float32, lambda w, i: torch.full_like(i, scale))
    stride = grads.shape[1]
    B = max(float(grads[w, :d].double().norm()) for w in range(M))
    ref = 2.0 * B * np.sqrt(np.log(n) / n)
    amp_ws = torch.empty(F.workspace_bytes(F.OP_AMPLITUDES, d, M=M), dtype=torch.uint8, device=DEV)
    for workers in (M, 1):
        ws = torch.empty(max(16, workers * F.workspace_bytes(F.OP_ENCODE, d)), dtype=torch.uint8, device=DEV)
        lam, lam_s = torch.full((2, 1), 7.0, device=DEV)
        bits, again = torch.zeros(2, M, (1 << L) // 32, dtype=torch.int32, device=DEV)
        F.encode_measured(grads, d, bits, lam, lam_s, 5, 1, alpha=2.0, alpha_s=2.0, ws=ws, amp_ws=amp_ws, worker_stride=stride)
        F.encode_dev(grads, d, again, lam, 5, 1, ws=ws, worker_stride=stride)
        torch.cuda.synchronize()
        assert torch.equal(bits, again)
        assert abs(float(lam) - ref) <= RTOL * ref, (workers, float(lam), ref)
        ref_s = 2.0 * ref * np.sqrt(np.log(n))
        assert abs(float(lam_s) - ref_s) <= RTOL * ref_s


@pytest.mark.parametrize("d,b,M", [
    ((5 << 17) + 1, 17, 3), ((3 << 18) - 1, 18, 2), ((3 << 20) - 5, 20, 2), ((3 << 22) - 7, 22, 1), ((1 << 23) - 3, 0, 2), ((3 << 23) + 1, 23, 1),
    ((3 << 24) - 9, 24, 1),
    ((1 << 20) + 1, 20, 1), (4 << 16, 16, 2),           # up to 256 sums; no kernel that carries them
])
def test_one_amplitude_of_a_long_vector(F, d, b, M):
    """More sums per worker than the scratch of the norms holds (256): they wait in the output and are added up there, and
    the packed words come out whole."""
    dp, n = F.padded_dim(d, b), float(F.transform_len(d, b))
    grads = scaled(M, d, torch.float32, lambda w, i: torch.full_like(i, 1) + (i == 12345).long())     # one entry of 1e20
    stride = grads.shape[1]
    ref = 2.0 * max(float(grads[w, :d].double().norm()) for w in range(M)) * np.sqrt(np.log(n) / n)
    amp_ws = torch.empty(F.workspace_bytes(F.OP_AMPLITUDES, d, M=M), dtype=torch.uint8, device=DEV)
    ws = torch.empty(M * F.workspace_bytes(F.OP_ENCODE, d, block_log2=b), dtype=torch.uint8, device=DEV)
    lam, lam_s = torch.full((2, 1), 7.0, device=DEV)
    bits, again = torch.zeros(2, M, dp // 32, dtype=torch.int32, device=DEV)
    F.encode_measured(grads, d, bits, lam, lam_s, 5, 1, alpha=2.0, alpha_s=2.0, block_log2=b, ws=ws, amp_ws=amp_ws, worker_stride=stride)
    F.encode_dev(grads, d, again, lam, 5, 1, block_log2=b, ws=ws, worker_stride=stride)
    torch.cuda.synchronize()
    assert torch.equal(bits, again)
    assert abs(float(lam) - ref) <= RTOL * ref
