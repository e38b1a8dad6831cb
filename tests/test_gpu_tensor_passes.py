"""The tensor-core passes of the one-plane decoders at every length they have: bit for bit what the plain ALUs give (all
values are exact integers until the final scale), and really the kernels that ran."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def F():
    import paper_2405_11095_b200 as f
    return f


def planes(M, dp, seed):
    """Random packed planes, with long runs of equal signs at both ends of the rows: the extreme values of the small factors."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    bits = torch.randint(-2**31, 2**31, (M, dp // 32), generator=g, device=DEV, dtype=torch.int64).to(torch.int32)
    bits[0, : dp // 64] = -1
    bits[-1, dp // 64:] = 0
    return bits


def with_mask(F, mask, run):
    """run() under a mask of tensor-core passes -> its outputs and the kernels that ran."""
    prev = F.set_tensor_core_pass(mask)
    try:
        with F.PassTrace() as tr:
            out = run()
        torch.cuda.synchronize()
        return out, tr.labels
    finally:
        F.set_tensor_core_pass(prev)


def ran(labels):
    """(strided, contiguous): did the tensor-core passes run?"""
    return any(x.startswith("tc10") for x in labels), any(x.startswith("tcrow") for x in labels)


@pytest.mark.parametrize("M", [1, 2, 5])
@pytest.mark.parametrize("L,blocks", [(16, 1), (16, 3), (17, 1), (18, 1), (18, 5), (19, 1), (20, 1), (21, 3), (22, 1), (23, 1), (24, 1), (25, 1)])
def test_any_size(F, L, blocks, M):
    """FOSGD_TC_ANY_SIZE lifts the thresholds of the chosen passes at every length they have."""
    b = 0 if blocks == 1 else L
    d, seed, step = (blocks << L) - 9, 11, L
    dp = F.padded_dim(d, b)
    bits = planes(M, dp, L + M)
    ws = torch.empty(M * F.workspace_bytes(F.OP_AGGREGATE, d, M=M, block_log2=b), dtype=torch.uint8, device=DEV)

    def run():
        acc = torch.full((dp,), 7.0, device=DEV)
        F.server_aggregate(bits, d, acc, 0.25, seed, step, worker_id0=1, block_log2=b, ws=ws)
        return acc

    plain, labels = with_mask(F, 0, run)
    assert ran(labels) == (False, False), labels
    S, C, A = F.TC_STRIDED, F.TC_CONTIGUOUS, F.TC_ANY_SIZE
    for mask, strided, contiguous in ((S | A, L >= 20, False), (C | A, False, L <= 24 or M >= 5),
                                      (S | C | A, L >= 20, L < 20 or L == 24 or (L == 25 and M >= 5))):
        acc, labels = with_mask(F, mask, run)
        assert ran(labels) == (strided, contiguous), (mask, labels)
        assert torch.equal(acc, plain), mask
    assert F.async_timeouts() == 0


DEFAULT = 3     # both passes, with their thresholds


@pytest.mark.parametrize("d,b,M", [
    ((9 << 16) - 1, 16, 15), ((5 << 17) + 9, 17, 7), ((1 << 18) - 1, 0, 9), (3 << 18, 18, 6), ((1 << 19) + 7, 19, 5), (1 << 20, 0, 128),
    (3 << 20, 20, 11), ((1 << 21) - 9, 0, 64), ((1 << 22) + 5, 22, 5), ((1 << 23) - 77, 0, 5), ((1 << 24) - 1, 0, 3), ((1 << 24) + 3, 24, 6),
    ((1 << 25) - 5, 0, 5), ((1 << 25) - 5, 0, 8), ((1 << 25) + 12345, 25, 6),
])
def test_contiguous_pass_of_every_length(F, d, b, M):
    """The averaged decoder by default, against the plain ALUs: the plain average, the average in two calls with an addition in between, scratch for
    five workers at a time, and (in blocks) an amplitude per worker and block, alone and by chunks."""
    seed, step = 13, M
    dp = F.padded_dim(d, b)
    bits = planes(M, dp, d % 1009 + M)
    need = F.workspace_bytes(F.OP_AGGREGATE, d, M=M, block_log2=b)
    ws = torch.empty(M * need, dtype=torch.uint8, device=DEV)
    few = ws[: min(M, 5) * need]
    lam = torch.rand(M, dp >> b, generator=torch.Generator(device=DEV).manual_seed(M), device=DEV) + 0.5 if b else None

    def run():
        outs = [torch.full((dp,), 7.0, device=DEV) for _ in range(5 if b else 3)]
        F.server_aggregate(bits, d, outs[0], 0.25, seed, step, worker_id0=1, block_log2=b, ws=ws)
        k = max(M - 5, M // 2)
        F.server_aggregate(bits[:k], d, outs[1], 0.25, seed, step, N_total=M, worker_id0=1, flags=F.AGG_BEGIN, block_log2=b, ws=ws)
        F.server_aggregate(bits[k:], d, outs[1], 0.25, seed, step, N_total=M, worker_id0=1 + k, flags=F.AGG_END, block_log2=b, ws=ws)
        F.server_aggregate(bits, d, outs[2], 0.25, seed, step, worker_id0=1, block_log2=b, ws=few)
        if b:
            F.server_aggregate_dev(bits, d, outs[3], lam, seed, step, worker_id0=1, block_log2=b, per_block=True, ws=ws)
            F.server_aggregate_dev(bits, d, outs[4], lam, seed, step, worker_id0=1, block_log2=b, per_block=True, ws=few)
        return outs

    plain, labels = with_mask(F, 0, run)
    assert ran(labels) == (False, False), labels
    outs, labels = with_mask(F, DEFAULT, run)
    T = 15 if (b or (dp - 1).bit_length()) == 25 else 14
    assert any(x.startswith(f"tcrow{T}") for x in labels), labels
    for k, (x, y) in enumerate(zip(outs, plain)):
        # (a weight rounds each worker's term, and the sum over the workers is rounded in the order of the blocks that share them)
        assert torch.equal(x, y) if k < 3 else float((x - y).norm()) <= 1e-6 * float(y.norm()), k
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
    assert F.async_timeouts() == 0
