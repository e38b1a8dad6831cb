"""The calls that programs built on this package make, as cases to time.

A case names a role of the protocol and its sizes.  The roles are the programs that exist in practice:

  round_trip  all workers of an iteration simulated as a batch on one GPU (distributed.round_trip):
              encode M gradients, decode + average + re-encode, decode the downlink
  worker      one training process: encodes its own gradient, applies the downlink to its parameters
  server      the aggregating process: packed uplink planes in, average and downlink planes out
  loop        one iteration of closed_loop.run after the gradients: amplitudes measured on the device, encode,
              aggregate, fused update

Amplitudes are passed by value ("value"), measured on the device by every pass, one for all workers
("device"), or measured per worker and block of the blocked mode ("block").
"""
import math

import torch

import paper_2405_11095_b200 as F
from paper_2405_11095_b200 import distributed, synthetic

#: log10 range of the per-tensor standard deviations of the layered gradients (as in the two layered workloads)
STD_LOG10 = {"fp32": (-4.0, -1.0), "bf16": (-5.0, -2.0)}
DTYPES = {"fp32": torch.float32, "bf16": torch.bfloat16}
MOST_COORDINATES = 1 << 29     # M d' of a drawn case: the largest batch among the listed ones


def _case(role, d, M=1, K=1, block=0, dtype="fp32", values="layered", amps="value", **more):
    return dict(role=role, d=d, M=M, K=K, block=block, dtype=dtype, values=values, amps=amps, **more)


def listed():
    return [
        # the closed-loop least-squares run at its default sizes: eight workers, 255 dithers on the downlink
        _case("loop", 8192, 8, K=255, values="normal", amps="device", name="loop_8k"),
        # the four batch workloads of the benchmark that fit a launch or two: the smallest is all latency
        _case("round_trip", 1 << 16, 4, values="normal", name="batch_64k"),
        _case("round_trip", 1 << 20, 16, values="student_t", name="batch_1m"),
        _case("round_trip", 1 << 24, 32, values="sparse", name="batch_16m"),
        _case("round_trip", 25_557_032, 8, name="batch_resnet50"),
        # the same model in blocks, with several dithers on the downlink
        _case("round_trip", 25_557_032, 8, K=3, block=20, name="batch_resnet50_blocks"),
        # one amplitude per worker and block, measured on the device (gradients whose scale differs by block)
        _case("round_trip", (1 << 23) + 77_777, 16, block=16, amps="block", name="batch_block_amps"),
        # a bf16 gradient of 1.3 billion parameters, one transform over all of it and in blocks
        _case("round_trip", 1_315_819_520, 2, dtype="bf16", name="batch_decoder_1p3b"),
        _case("round_trip", 1_315_819_520, 2, block=20, dtype="bf16", name="batch_decoder_blocks"),
        # one process of data-parallel training: its own gradient up, the average down
        _case("worker", 25_557_032, name="worker_resnet50"),
        _case("worker", 5_000_011, K=15, dtype="bf16", name="worker_bf16_odd"),
        # a server with many workers of a small odd-sized model
        _case("server", 300_007, 64, K=3, name="server_300k"),
    ]


def draw(rng):
    role = rng.choice(("round_trip", "round_trip", "worker", "server", "loop"))
    top = {"loop": 20, "server": 27}.get(role, 30.3)
    d = int(2 ** rng.uniform(9, top))
    shape = rng.random()
    if shape < 0.25:
        d = 1 << round(math.log2(d))
    elif shape < 0.75:
        d |= 1
    block = rng.choice((0, 0, 0, rng.randint(10, 20)))
    dp = F.padded_dim(d, block)
    M = 1 if role == "worker" else max(1, min(64, int(2 ** rng.uniform(0, 6.5)), MOST_COORDINATES // dp))
    dtype = "fp32" if role == "loop" else rng.choice(("fp32", "fp32", "bf16"))
    if role == "loop":
        amps = rng.choice(("device", "block")) if block else "device"
    elif role == "round_trip":
        amps = rng.choice(("value", "value", "device", "block" if block else "device"))
    else:
        amps = "value"
    K = rng.choice((1, 1, 3, 7, 15) if dp > 1 << 18 else (1, 3, 15, 255))
    if dp > 1 << 27:
        K = 1
    values = rng.choice(("normal", "student_t", "sparse", "layered")) if d < 1 << 25 else "layered"
    return _case(role, d, M, K=K, block=block, dtype=dtype, values=values, amps=amps)


def _row_stride(case):
    """Elements between the rows of a gradient matrix whose rows start 16-byte aligned."""
    per = 4 if case["dtype"] == "fp32" else 8
    return -(-case["d"] // per) * per


def _gradients(case, seed):
    d, M, dtype = case["d"], case["M"], DTYPES[case["dtype"]]
    w = synthetic.Workload("case", d, M, dtype, case["values"], seed=seed, std_log10=STD_LOG10[case["dtype"]])
    g = torch.zeros(M, _row_stride(case), dtype=dtype, device="cuda")
    for n in range(M):
        synthetic.worker_gradient(w, n, "cuda", out=g[n, :d])
    return g


def _random_planes(shape, seed):
    """Packed planes as they arrive from the network: the dithered signs are close to fair coins."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(-(1 << 31), 1 << 31, shape, generator=gen, device="cuda", dtype=torch.int32)


def prepare(case, seed):
    d, M, K, b, role = (case[k] for k in ("d", "M", "K", "block", "role"))
    dp, n_eff, P = F.padded_dim(d, b), F.transform_len(d, b), F.planes(K)
    s = dict(case=dict(case), seed=seed, step=0)
    per_worker = F.workspace_bytes(F.OP_AGGREGATE, d, block_log2=b, K=K)
    # scratch for all workers of a launch; a transform with two strided passes takes 1.5 times the minimum
    s["ws"] = torch.empty(max(16, M * per_worker * 3 // 2 if n_eff > 1 << 25 else M * per_worker),
                          dtype=torch.uint8, device="cuda")
    if role == "server":
        s["bits"] = _random_planes((M, dp // 32), seed)
        B = 1.0
    else:
        s["grads"] = _gradients(case, seed)
        s["bits"] = torch.zeros(M, dp // 32, dtype=torch.int32, device="cuda")
        B = max(float(g[:d].float().norm()) for g in s["grads"])
    s["lam"] = F.lambda_(B, 2.0, n_eff)
    s["lam_s"] = F.lambda_server(s["lam"], 2.0, n_eff)
    if role == "worker":
        s["down"] = _random_planes((P, dp // 32), seed + 1)
        s["x"] = torch.randn(d, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")
        return s
    s["acc"] = torch.zeros(dp, device="cuda")
    s["down"] = torch.zeros(P, dp // 32, dtype=torch.int32, device="cuda")
    if role == "round_trip":
        s["buf"] = distributed.RoundTripBuffers(s["bits"], s["acc"], s["down"], torch.zeros(d, device="cuda"), s["ws"])
    if case["amps"] != "value":
        per_block = case["amps"] == "block"
        nb = dp >> b if per_block else 1
        op = F.OP_BLOCK_AMPLITUDES if per_block else F.OP_AMPLITUDES
        lam = torch.zeros(M * nb if per_block else 1, device="cuda")
        ws = torch.empty(F.workspace_bytes(op, d, M=M, block_log2=b), dtype=torch.uint8, device="cuda")
        s["amps"] = distributed.DeviceAmplitudes(lam, torch.zeros(nb, device="cuda"), ws, per_block)
    if role == "loop":
        s["x"] = torch.zeros(d, device="cuda")
    return s


def run(s):
    case, seed, step = s["case"], s["seed"], s["step"]
    d, K, b, role, ws = case["d"], case["K"], case["block"], case["role"], s["ws"]
    s["step"] += 1                       # an iteration of the program: new flips and dithers
    stride = _row_stride(case)
    if role == "round_trip":
        out = distributed.round_trip(F, s["grads"], d, s["buf"], s["lam"], s["lam_s"], seed, step, K=K, block_log2=b,
                                     worker_stride=stride, amps=s.get("amps"))
        return [s["bits"], s["acc"], s["down"], out]
    if role == "worker":
        F.encode(s["grads"], d, s["bits"], s["lam"], seed, step, block_log2=b, ws=ws, worker_stride=stride)
        F.downlink_apply(s["down"], d, s["x"], s["lam_s"], seed, step, 1e-3, K=K, block_log2=b, ws=ws)
        return [s["bits"], s["x"]]
    if role == "server":
        F.server_aggregate(s["bits"], d, s["acc"], s["lam"], seed, step, lam_s=s["lam_s"], K=K, down_bits=s["down"],
                           block_log2=b, ws=ws)
        return [s["acc"], s["down"]]
    a = s["amps"]
    F.amplitudes(s["grads"], d, a.lam, a.lam_s, alpha=a.alpha, alpha_s=a.alpha_s, block_log2=b,
                 per_block=a.per_block, ws=a.ws, worker_stride=stride)
    F.encode_dev(s["grads"], d, s["bits"], a.lam, seed, step, block_log2=b, per_block=a.per_block, ws=ws,
                 worker_stride=stride)
    F.server_aggregate_dev(s["bits"], d, s["acc"], a.lam, seed, step, lam_s=a.lam_s, K=K, down_bits=s["down"],
                           block_log2=b, per_block=a.per_block, ws=ws)
    F.downlink_apply(s["down"], d, s["x"], a.lam_s, seed, step, 1e-3, K=K, block_log2=b, per_block=a.per_block, ws=ws)
    return [s["bits"], s["acc"], s["down"], s["x"]]


def work(case):
    """Bytes: gradients, packed planes, average and decoded vector, each once per call that takes or gives it.  Flops:
    the additions of the transforms, and one addition and one comparison per dither."""
    d, M, K, role = case["d"], case["M"], case["K"], case["role"]
    dp, P, L = F.padded_dim(d, case["block"]), F.planes(K), math.log2(F.transform_len(d, case["block"]))
    grad = d * (4 if case["dtype"] == "fp32" else 2)
    up = M * (grad + dp / 8), M * dp * (L + 2)
    average = M * dp / 8 + dp * 4 + P * dp / 8, M * dp * (L + 1) + dp * (L + 2 * K)
    down = P * dp / 8 + d * 4, dp * (L + 1)
    update = down[0] + d * 4, down[1] + d
    parts = {"round_trip": (up, average, down), "worker": (up, update), "server": (average,),
             "loop": (up, average, update)}[role]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    """Measured against the same chain in fp64 (the oracle; 2^16 .. 2^24 coordinates, both types, K = 1 .. 255), times four.

    Values: 2.5e-8 .. 4e-8 (largest difference 6e-8 .. 9e-8), the rounding of one fp32 product or update: everything
    before it is sums of small integers.  Packed signs: up to 1e-6 of the words hold a coordinate whose dithered
    value is within rounding of zero, none at all in batches below 2^18 coordinates.  Where a pass feeds
    its own signs into its server step, one such sign moves every entry of the average, and with it further signs of the
    downlink: 2.4e-4 of the words, 5.5e-3 of the decoded vector (largest difference 3e-2) at 2^24; a count of K
    dithers has K chances to change."""
    chained = case["role"] in ("round_trip", "loop")
    if chained and case["M"] * F.padded_dim(case["d"], case["block"]) > 1 << 18:
        return {"rel": 2.2e-2, "max": 0.15, "differ": min(1e-2, 1e-3 * case["K"])}
    return {"rel": 2e-7, "max": 5e-7, "differ": 0.0 if chained else 1e-5}
