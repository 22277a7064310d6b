"""The work that programs built on this library have it do, as measurable cases.

One case is one pass through the public entry points (``paper_2411_07942_b200.binding``) at one shape:

  step       N devices' partial sums quantised in one launch, then decompressed and summed (the single-GPU
             simulation of one synchronisation, what the benchmark times)
  rank       what one device of a tensor-parallel group computes: its own shard quantised, the N payloads reduced
  exchange   the fused exchange with this GPU's receive buffer as the destination: N pushes, then the reduction
             that waits for the arrival words
  calibrate  a resumed calibration job: running ranges restored, n_seq more sequences of every device folded,
             the feature set chosen, the ranges read back for the checkpoint
  layer      the producing linear layer fused with the quantiser

Sizes are the repository's workloads (Llama-2-13B- and Gemma-2-27B-shaped synchronisations, the large sweep,
the calibration pass, the fused layer of the benchmark) and the ranges between and below them.
"""
import math

import numpy as np
import torch

from paper_2411_07942_b200 import binding

CAL_ROWS = 256      # tokens of the calibration sequence that fixes a case's steps and feature set
GAMMA = 0.01        # the paper's moving-average constant


def _case(name, op, N=1, T=1, E=5120, k=-1, bits=4, out="bf16", bias=False, pad=0, n_seq=0, S=0, K=0):
    """k = -1: the paper's E/64 selected features.  pad: elements between the rows of the BF16 inputs."""
    c = {"op": op, "N": N, "T": T, "E": E, "k": k, "bits": bits, "out": out, "bias": bias, "pad": pad,
         "n_seq": n_seq, "S": S, "K": K}
    return {"name": name, **c} if name else c


def listed():
    return [
        # one generated token of a Gemma-2-27B-shaped model over 8 devices: nothing but latency
        _case("token", "step", N=8, T=1, E=4608),
        # the decode configuration: a batch of 64 sequences
        _case("decode", "step", N=8, T=64, E=4608),
        # the headline prefill configuration (Llama-2-13B-shaped, 4 devices)
        _case("prefill", "step", N=4, T=2048, E=5120),
        # a rank of the paper's 8-device group whose next layer wants the sum with its bias in FP32; odd token count
        _case("rank_fp32_bias", "rank", N=8, T=2047, E=5120, out="fp32", bias=True),
        # the end of the large sweep
        _case("large", "step", N=16, T=8192, E=8192),
        # lower and higher precision than Int4 (the paper's comparison over code widths)
        _case("three_bit", "step", N=4, T=2048, E=5120, bits=3),
        _case("eight_bit", "step", N=8, T=1000, E=4608, bits=8),
        # one per cent of the features kept in BF16 instead of E/64: a count that is no multiple of anything
        _case("one_percent", "step", N=4, T=2048, E=5120, k=51),
        # the fused exchange at a medium prompt
        _case("exchange", "exchange", N=4, T=512, E=5120),
        # a chunk of the calibration pass: 8 devices, 8 sequences of 2048 tokens each
        _case("calibrate", "calibrate", N=8, E=4608, n_seq=8, S=2048),
        # the feed-forward down projection of the headline configuration and a small decode batch of the
        # attention output projection, each with its compression
        _case("layer_prefill", "layer", T=2048, E=5120, K=3456),
        _case("layer_decode", "layer", T=64, E=5120, K=1280),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choices(["step", "rank", "exchange", "calibrate", "layer"], [40, 20, 10, 10, 20])[0]
    if rng.random() < 0.5:
        E = rng.choice([1024, 2048, 4096, 4608, 5120, 6144, 8192])
    else:  # any model width: a multiple of 64, its E/64 mostly no multiple of 8
        E = 64 * rng.randint(8, 128)
    if op == "layer":  # the fused layer takes widths whose selected count is a multiple of 8
        E = 512 * max(1, round(E / 512))
        K = 8 * _log_int(rng, 64, 1024)
        most = max(1, min(8192, int(2048 * 3456 * 5120 * 4 / (K * E))))
        return _case(None, op, T=_log_int(rng, 1, most), E=E, K=K)
    N = rng.choice([2, 4, 4, 8, 8, 16, rng.randint(2, 16)])
    if op == "calibrate":
        S = _log_int(rng, 16, 4096)
        n_seq = max(1, min(_log_int(rng, 1, 128), int(8 * 8 * 2048 * 4608 / (N * S * E))))
        return _case(None, op, N=N, E=E, n_seq=n_seq, S=S)
    if rng.random() < 0.1:  # small widths of no particular form
        E = rng.randint(65, 1024)
    k = rng.choices([-1, E // 100, 0], [65, 20, 15])[0]
    bits = 4 if rng.random() < 0.75 else rng.choice([2, 3, 5, 6, 7, 8])
    kk = E // 64 if k < 0 else k
    plain = bits == 4 and E % 8 == 0 and kk % 8 == 0
    # the largest sizes belong to the paper's own width and rule, the variants stay at the prefill sizes
    most = (16 * 8192 * 8192 if op == "step" else 8 * 8192 * 8192) if plain else 4 * 2048 * 5120
    T = _log_int(rng, 1, max(1, min(8192, most // (N * E))))
    return _case(None, op, N=N, T=T, E=E, k=k, bits=bits, out=rng.choice(["bf16", "bf16", "fp32"]),
                 bias=op != "step" and rng.random() < 0.5, pad=rng.choice([0, 0, 0, 64]))


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + stream) & 0x7FFFFFFFFFFF)
    return g


def _scales(case, seed):
    """Per-feature scale: log-normal, one per cent of the columns 20 to 200 times larger (shared by all devices)."""
    g, E = _gen(seed, 0), case["E"]
    s = torch.exp(0.7 * torch.randn(E, generator=g, device="cuda"))
    n = max(1, E // 100)
    cols = torch.randperm(E, generator=g, device="cuda")[:n]
    s[cols] *= torch.exp(torch.empty(n, device="cuda").uniform_(math.log(20.0), math.log(200.0), generator=g))
    return s


def _partial_sums(rows, E, scale, g, pad=0):
    """[rows, E] BF16, in a buffer whose rows are E + pad apart."""
    buf = torch.empty((rows, E + pad), dtype=torch.bfloat16, device="cuda")
    step = max(1, (1 << 26) // E)
    for r in range(0, rows, step):
        n = min(step, rows - r)
        buf[r:r + n, :E] = torch.randn((n, E), generator=g, device="cuda").mul_(scale)
    return buf[:, :E]


def _inputs(case, seed):
    """The device tensors a program has before the call."""
    d = {}
    N, T, E = case["N"], case["T"], case["E"]
    scale = _scales(case, seed)
    if case["op"] == "calibrate":
        d["seqs"] = [_partial_sums(case["n_seq"] * case["S"], E, scale, _gen(seed, 100 + i)) for i in range(N)]
        g = _gen(seed, 1)
        z = 3.5 + torch.rand((2, N, E), generator=g, device="cuda")
        d["m"], d["M"] = (-z[0] * scale).cpu().numpy(), (z[1] * scale).cpu().numpy()
        return d
    d["cal"] = [_partial_sums(CAL_ROWS, E, scale, _gen(seed, 200 + i)) for i in range(N)]
    if case["op"] == "layer":
        # x and W of unit variance over K: outputs of the same family of scales
        g, K = _gen(seed, 2), case["K"]
        d["x"] = torch.randn((T, K), generator=g, device="cuda").to(torch.bfloat16)
        w = torch.randn((E, K), generator=g, device="cuda") * (scale / math.sqrt(K))[:, None]
        d["w"] = w.to(torch.bfloat16)
        return d
    d["y"] = [_partial_sums(T, E, scale, _gen(seed, 100 + i), case["pad"]) for i in range(N)]
    if case["bias"]:
        d["bias"] = torch.randn(E, generator=_gen(seed, 3), device="cuda")
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    N, T, E, op = case["N"], case["T"], case["E"], case["op"]
    stream = torch.cuda.current_stream().cuda_stream
    tpq = binding.Tpq(N, E, bits=case["bits"], gamma=GAMMA)
    s = {"op": op, "tpq": tpq, "T": T, "N": N, "stream": stream, "inputs": d}
    if op == "calibrate":
        s.update(n_seq=case["n_seq"], S=case["S"], m=d["m"], M=d["M"], counts=np.full(N, 4, np.int64),
                 seq_ptrs=[y.data_ptr() for y in d["seqs"]])
        return s
    for i, y in enumerate(d["cal"]):
        tpq.calibrate_ranges(i, y.data_ptr(), 1, CAL_ROWS, stream=stream)
    tpq.select_features(case["k"])
    P = tpq.payload_bytes(T)
    s["P"] = P
    if op == "layer":
        s["K"] = case["K"]
        s["w_slots"] = torch.empty_like(d["w"])
        tpq.permute_weight(d["w"].data_ptr(), case["K"], s["w_slots"].data_ptr(), stream=stream)
        s["payload"] = torch.empty(P, dtype=torch.uint8, device="cuda")
        s["code_bytes"] = P - 2 * T * tpq.num_selected()
        del d["w"]
        return s
    s["stride"] = E + case["pad"]
    s["payloads"] = [torch.empty(P, dtype=torch.uint8, device="cuda") for _ in range(N)]
    s["out"] = torch.empty((T, E), dtype=torch.float32 if case["out"] == "fp32" else torch.bfloat16, device="cuda")
    s["dtype"] = binding.TPQ_OUT_FP32 if case["out"] == "fp32" else binding.TPQ_OUT_BF16
    s["bias_ptr"] = d["bias"].data_ptr() if case["bias"] else None
    s["y_ptrs"] = [y.data_ptr() for y in d["y"]]
    s["pl_ptrs"] = [p.data_ptr() for p in s["payloads"]]
    if op == "rank":  # the peers' payloads have arrived
        for i in range(1, N):
            tpq.quantize_pack(i, s["y_ptrs"][i], T, s["pl_ptrs"][i], P, row_stride=s["stride"], stream=stream)
        d["y"] = d["y"][:1]
    if op == "exchange":
        s["words"] = torch.zeros(N, dtype=torch.int32, device="cuda")
        s["word_ptrs"] = [s["words"].data_ptr() + 4 * i for i in range(N)]
        s["epoch"] = 0
    return s


def run(s):
    tpq, op, T, stream = s["tpq"], s["op"], s["T"], s["stream"]
    if op == "calibrate":
        tpq.set_ranges(s["m"], s["M"], s["counts"])
        for i, ptr in enumerate(s["seq_ptrs"]):
            tpq.calibrate_ranges(i, ptr, s["n_seq"], s["S"], stream=stream)
        features = tpq.select_features()
        m, M = tpq.get_ranges(with_R=False)
        return {"features": features, "m": m, "M": M}
    if op == "layer":
        pl = s["payload"]
        tpq.linear_quantize_pack(0, s["inputs"]["x"].data_ptr(), s["w_slots"].data_ptr(), T, s["K"], pl.data_ptr(), s["P"],
                                 stream=stream)
        return {"codes": pl[:s["code_bytes"]], "selected": pl[s["code_bytes"]:].view(torch.bfloat16)}
    out = s["out"]
    if op == "step":
        tpq.quantize_pack_batch(0, s["y_ptrs"], T, s["pl_ptrs"], s["P"], row_stride=s["stride"], stream=stream)
    elif op == "rank":
        tpq.quantize_pack(0, s["y_ptrs"][0], T, s["pl_ptrs"][0], s["P"], row_stride=s["stride"], stream=stream)
    else:
        s["epoch"] = s["epoch"] % 0x7FFFFFFF + 1
        for i in range(s["N"]):
            tpq.quantize_pack_push(i, s["y_ptrs"][i], T, [s["pl_ptrs"][i]], [s["word_ptrs"][i]], s["P"], s["epoch"],
                                   row_stride=s["stride"], stream=stream)
        tpq.dequant_reduce(s["pl_ptrs"], T, out.data_ptr(), s["dtype"], stream=stream, bias_ptr=s["bias_ptr"],
                           arrived_ptr=s["words"].data_ptr(), epoch=s["epoch"])
        return {"payloads": s["payloads"], "out": out}
    tpq.dequant_reduce(s["pl_ptrs"], T, out.data_ptr(), s["dtype"], stream=stream, bias_ptr=s["bias_ptr"])
    return {"payloads": s["payloads"][:1] if op == "rank" else s["payloads"], "out": out}


# ------------------------------------------------------------------------------------- what a pass is about
def _k(case):
    return case["E"] // 64 if case["k"] < 0 else case["k"]


def _payload_bytes(case):
    T, k = case["T"], _k(case)
    return (-(-T * (case["E"] - k) * case["bits"] // 8) + 15) // 16 * 16 + 2 * T * k


def work(case):
    """Inputs read once, payloads written once and read once, output written once."""
    N, T, E, op = case["N"], case["T"], case["E"], case["op"]
    if op == "calibrate":
        return {"bytes": 2 * N * case["n_seq"] * case["S"] * E, "flops": 0}
    P = _payload_bytes(case)
    if op == "layer":
        return {"bytes": 2 * case["K"] * (T + E) + P, "flops": 2 * T * case["K"] * E}
    shards = 1 if op == "rank" else N
    return {"bytes": shards * (2 * T * E + P) + N * P + T * E * (4 if case["out"] == "fp32" else 2), "flops": 0}


def tolerance(case):
    """Codes, payloads, features and ranges are defined to the bit, and so is the sum: binary32, devices in
    ascending order, one final rounding.  Only the layer's products may be summed in another order."""
    T = case["T"]
    if case["op"] == "layer":
        # measured against the sums in 64 bits, times four: BF16 roundings that fall the other way (of the selected
        # features 2e-4 in the 2-norm, 0.0076 at most), and the code bytes that such a rounding moves to the next
        # level (3.4e-5 of them); in a small result one such value is a larger share
        few = T * _k(case) < 4096
        codes = T * (case["E"] - _k(case)) / 2
        return {"rel": 4e-3 if few else 8e-4, "max": 3e-2, "differ": max(1.5e-4, 4 / codes)}
    return "exact"


# --------------------------------------------------------------------------------- the same in plain torch
def _steps_and_set(case, cal):
    """Steps, reciprocal steps and the selected features from one calibration sequence per device."""
    R = torch.stack([2.0 * torch.maximum(-y.float().amin(0), y.float().amax(0)) for y in cal])
    agg = R[0].clone()
    for r in R[1:]:
        agg += r
    sel = torch.sort(torch.sort(agg, descending=True, stable=True).indices[:_k(case)]).values
    # (a tensor as the divisor: by a plain number torch multiplies with its rounded reciprocal)
    s = (R / torch.full_like(R, 2.0 ** case["bits"] - 1.0)).clamp_min(2.0 ** -23)
    return s, 1.0 / s, sel


def exact(case, seed):
    N, T, E, op = case["N"], case["T"], case["E"], case["op"]
    d = _inputs(case, seed)
    if op == "calibrate":
        lo, hi = d["m"].astype(np.float64), d["M"].astype(np.float64)
        for i in range(N):
            seqs = d["seqs"][i].view(case["n_seq"], case["S"], E)
            lows, highs = seqs.amin(1).double().cpu().numpy(), seqs.amax(1).double().cpu().numpy()
            for q in range(case["n_seq"]):
                lo[i] += GAMMA * (lows[q] - lo[i])
                hi[i] += GAMMA * (highs[q] - hi[i])
        return {"features": None, "m": lo, "M": hi}
    s, inv, sel = _steps_and_set(case, d["cal"])
    if op == "layer":
        rows = [d["x"][r:r + 1024].double() @ d["w"][sel].double().t() for r in range(0, T, 1024)]
        return {"codes": None, "selected": torch.cat(rows).reshape(-1)}
    half = 2.0 ** (case["bits"] - 1)
    out = torch.empty((T, E), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 25) // E)
    for r in range(0, T, step):
        acc = torch.zeros((min(step, T - r), E), dtype=torch.float64, device="cuda")
        for i in range(N):
            y = d["y"][i][r:r + step].float()
            part = torch.round((y * inv[i]).clamp(-half, half - 1.0)).double() * s[i].double()
            part[:, sel] = y[:, sel].double()
            acc += part
        out[r:r + step] = acc + d["bias"].double() if case["bias"] else acc
    return {"payloads": [None] * (1 if op == "rank" else N), "out": out}
