"""Timed cases of the truncated-quantization path, through the calls that a data-parallel job makes.

What a case does (``kind``):

  round    one training step's compression on one GPU: statistics -> parameters -> compress all workers ->
           aggregate.  ``route`` "device": parameters designed on the device, nothing returns to the host.
           ``route`` "host": the statistics records are copied back and the parameters designed on the host.
           ``stats`` "hinted": one-pass statistics, hint kept from round to round; "two_pass": g_min = mean|g|.
  client   the sender alone: statistics -> parameters -> compress of its own rows.
  server   the receiver alone, on rows that have arrived.  ``form`` "plain": one [N, words] block; "rows": one
           address per row; "apply": aggregation fused with the momentum-SGD step.
  groups   a round with layer groups (segments of every row) that are quantized independently.

``gamma`` is the tail exponent handed to the parameter design; 0 means the maximum-likelihood estimate.
``data_gamma``, ``scale`` and ``outliers`` describe the synthetic gradients (inputs.powerlaw_gradient).
Every buffer a training loop keeps between steps (records, scratch, hint, packed rows, update) is made once.
"""
from __future__ import annotations

import ctypes
import math

import torch

from paper_2402_01798_b200 import binding as tq
from paper_2402_01798_b200 import inputs

_BITS = {2: 1, 4: 2, 8: 3, 16: 4}
_MODES = {"uniform": tq.UNIFORM, "nonuniform": tq.NONUNIFORM, "biscaled": tq.BISCALED}
_MOST_ELEMENTS = 1_000_000_000       # workers * d of a drawn case


def _case(kind, d, workers, mode, levels, dtype="float32", gamma=3.0, data_gamma=3.0, scale=5e-4, outliers=0.0,
          route="device", stats="hinted", groups=0, form="", weights=False, name=None):
    c = dict(kind=kind, d=d, workers=workers, mode=mode, levels=levels, dtype=dtype, gamma=gamma, data_gamma=data_gamma,
             scale=scale, outliers=outliers)
    if kind == "server":
        c.update(form=form, weights=weights)
    else:
        c.update(stats=stats)
        c.update(groups=groups) if kind == "groups" else c.update(route=route)
    if name is not None:
        c["name"] = name
    return c


def listed():
    bf16 = dict(dtype="bfloat16", data_gamma=3.0, scale=1e-4, outliers=0.01)
    return [
        # a small model (LeNet-sized gradient), one worker: latency and launches are all there is
        _case("round", 100_000, 1, "uniform", 4, scale=1e-3, name="round_100k"),
        # the introductory example at a small ragged size: everything by default, parameters on the host
        _case("round", 200_003, 3, "nonuniform", 8, scale=1e-3, route="host", stats="two_pass", name="round_200k_host"),
        # ResNet-18-sized gradient, 8 workers, tail exponent estimated from the data (Section 5)
        _case("round", 11_200_000, 8, "uniform", 8, gamma=0.0, data_gamma=2.5, scale=1e-3, name="round_11m"),
        # ResNet-50-sized gradient, 16 workers: the benchmark's default round
        _case("round", 25_600_000, 16, "nonuniform", 16, route="host", name="round_25m_host"),
        # the same job with its layers in 16 groups of very different sizes, as real networks have
        _case("groups", 25_557_033, 16, "nonuniform", 16, groups=16, name="groups_25m"),
        # GPT-2-small-sized gradient kept in bf16, both quantizer families and both code widths
        _case("round", 124_000_000, 8, "nonuniform", 16, name="round_124m_bf16_nonuniform", **bf16),
        _case("round", 124_000_000, 8, "uniform", 4, route="host", name="round_124m_bf16_uniform", **bf16),
        # a very large flat gradient: 16 GB of input, 3-bit codes
        _case("round", 1_000_000_000, 4, "nonuniform", 8, gamma=2.5, data_gamma=2.5, scale=1e-4, name="round_1e9"),
        # the Appendix's two-step quantizer on a medium gradient
        _case("round", 1_000_000, 8, "biscaled", 16, name="round_1m_biscaled"),
        # one sender of a distributed job: its own bf16 gradient, odd length
        _case("client", 3_500_001, 1, "nonuniform", 4, name="client_3m_bf16", **bf16),
        # the receiver: aggregation and optimiser step in one pass
        _case("server", 25_600_000, 16, "nonuniform", 16, form="apply", name="server_25m_apply"),
        # the receiver of many weighted clients, every row in a buffer of its own, odd length
        _case("server", 1_000_003, 64, "uniform", 8, form="rows", weights=True, scale=1e-3, name="server_1m_rows"),
    ]


def draw(rng):
    kind = rng.choice(["round", "round", "round", "client", "server", "groups"])
    workers = 1 if kind == "client" else rng.choice([1, 2, 3, 4, 5, 8, 11, 16, 16, 24, 32, 64])
    most = min(250_000_000, _MOST_ELEMENTS // workers)
    least = 200_000 if kind == "groups" else 20_000
    d = int(round(math.exp(rng.uniform(math.log(least), math.log(most)))))
    mode = rng.choice(["uniform", "nonuniform", "nonuniform", "biscaled"])
    levels = rng.choice({"uniform": [2, 4, 8, 16], "nonuniform": [4, 8, 16], "biscaled": [8, 16]}[mode])
    bf16 = rng.random() < 0.5
    data_gamma = rng.choice([2.5, 3.0, 4.0])
    return _case(kind, d, workers, mode, levels, dtype="bfloat16" if bf16 else "float32",
                 gamma=data_gamma if rng.random() < 0.7 else 0.0, data_gamma=data_gamma, scale=rng.choice([1e-4, 5e-4, 1e-3]),
                 outliers=0.01 if bf16 else 0.0, route=rng.choice(["device", "host"]),
                 stats=rng.choice(["hinted", "hinted", "two_pass"]), groups=rng.choice([2, 5, 16, 40]),
                 form=rng.choice(["plain", "rows", "apply"]), weights=rng.random() < 0.4)


def _group_table(d, n):
    """n segments of sizes that fall off geometrically, the smallest 1/75 of the largest, offsets 32-byte aligned."""
    share = [75.0 ** (-k / (n - 1)) for k in range(n)]
    total, table, at = sum(share), [], 0
    for k in range(n):
        length = d - at if k == n - 1 else max(16, int(d * share[k] / total) // 16 * 16)
        table.append((at, length))
        at += length
    return table[n // 2:] + table[:n // 2]          # the largest group is not the first one


def _gradients(case, seed):
    dtype = getattr(torch, case["dtype"])
    w = inputs.Workload("case", case["d"], case["workers"], case["data_gamma"], case["scale"], case["mode"], case["levels"],
                        dtype=dtype, outlier_frac=case["outliers"], base_seed=1000 * seed)
    return inputs.make_worker_gradients(w, "cuda")[0]


def _records(stats_dev):
    """The statistics records' fields as views of the record buffer: sums, counts, and (max|g|, g_min)."""
    n = stats_dev.numel() // 64
    return {"sums": stats_dev.view(torch.float64).view(n, 8)[:, 3:6], "counts": stats_dev.view(torch.int64).view(n, 8)[:, 0:3],
            "range": stats_dev.view(torch.float32).view(n, 16)[:, 12:14]}


def prepare(case, seed):
    kind, n, d = case["kind"], case["workers"], case["d"]
    bits, mode = _BITS[case["levels"]], _MODES[case["mode"]]
    s = dict(case=case, mode=mode, gamma=case["gamma"] or math.nan, seed=seed, n=n, d=d, levels=case["levels"])
    g = _gradients(case, seed)
    if kind == "server":
        stats = tq.stats_to_host(tq.tq_stats(g, d))
        s["params"] = tq.params_array([tq.tq_params(st, case["levels"], mode, s["gamma"]) for st in stats])
        packed = tq.tq_compress(g, s["params"], seed=seed, d=d)
        del g
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        s["weights"] = [(1.0 + (i % 5)) / (3.0 * n) for i in range(n)] if case["weights"] else None      # e.g. sample counts
        if case["form"] == "apply":
            s["theta"] = torch.randn(d, device="cuda", generator=gen) * 0.05
            s["momentum"] = torch.zeros(d, device="cuda")
        else:
            s["out"] = torch.empty(d, dtype=torch.float32, device="cuda")
        s["packed"] = [packed[i].clone() for i in range(n)] if case["form"] == "rows" else packed
        return s
    s["g"] = g
    jobs = n
    if kind == "groups":
        s["segments"] = tq.segments_array(_group_table(d, case["groups"]))
        jobs = n * case["groups"]
        words = tq.tq_segments_packed_words(s["segments"], bits)
    else:
        words = tq.tq_packed_words(d, bits)
    s["jobs"] = jobs
    s["stats"] = torch.empty(jobs * 64, dtype=torch.uint8, device="cuda")
    s["scratch"] = torch.empty(tq.tq_stats_workspace_bytes(jobs), dtype=torch.uint8, device="cuda")
    s["hint"] = tq.new_gmin_hint(jobs)
    s["packed"] = torch.empty((n, words), dtype=torch.int32, device="cuda")
    s["result"] = {"packed": s["packed"], **_records(s["stats"])}
    if kind != "client":
        s["out"] = s["result"]["update"] = torch.empty(d, dtype=torch.float32, device="cuda")
    if case.get("route") == "host":
        s["stats_pinned"] = torch.empty(jobs * 64, dtype=torch.uint8).pin_memory()
    else:
        record = ctypes.sizeof(tq.Params)
        s["params"] = torch.empty(jobs * record, dtype=torch.uint8, device="cuda")
        fields = s["params"].view(torch.float32).view(jobs, record // 4)
        s["result"].update(alpha=fields[:, 4], codebook=fields[:, 12:])
    return s


def _server(s):
    case = s["case"]
    if case["form"] == "apply":
        tq.tq_decompress_aggregate_apply(s["packed"], s["d"], s["params"], s["theta"], s["momentum"], lr=0.01, momentum=0.9,
                                         weight_decay=5e-4, weights=s["weights"])
        return {"theta": s["theta"], "momentum": s["momentum"]}
    call = tq.tq_decompress_aggregate_rows if case["form"] == "rows" else tq.tq_decompress_aggregate
    return call(s["packed"], s["d"], s["params"], weights=s["weights"], out=s["out"])


def _groups(s):
    g, seg = s["g"], s["segments"]
    if s["case"]["stats"] == "hinted":
        tq.tq_stats_hinted_segments(g, seg, s["hint"], stats_dev=s["stats"], workspace=s["scratch"])
    else:
        tq.tq_stats_segments(g, seg, stats_dev=s["stats"], workspace=s["scratch"])
    tq.tq_params_device(s["stats"], s["jobs"], s["levels"], s["mode"], s["gamma"], params_dev=s["params"])
    tq.tq_compress_segments(g, seg, s["params"], s["levels"], s["mode"], s["seed"], packed=s["packed"])
    tq.tq_decompress_aggregate_segments(s["packed"], seg, s["params"], s["levels"], out=s["out"])
    return s["result"]


def run(s):
    case = s["case"]
    if case["kind"] == "server":
        return _server(s)
    if case["kind"] == "groups":
        return _groups(s)
    g, n, d, mode, levels = s["g"], s["n"], s["d"], s["mode"], s["levels"]
    if case["stats"] == "hinted":
        tq.tq_stats_hinted(g, s["hint"], d, stats_dev=s["stats"], workspace=s["scratch"])
    else:
        tq.tq_stats(g, d, stats_dev=s["stats"], workspace=s["scratch"])
    if case["route"] == "host":
        s["stats_pinned"].copy_(s["stats"], non_blocking=True)
        torch.cuda.current_stream().synchronize()
        params = tq.tq_params_batch(s["stats_pinned"], n, levels, mode, s["gamma"])
        tq.tq_compress(g, params, s["seed"], d=d, packed=s["packed"])
        if case["kind"] == "round":
            tq.tq_decompress_aggregate(s["packed"], d, params, out=s["out"])
    else:
        tq.tq_params_device(s["stats"], n, levels, mode, s["gamma"], params_dev=s["params"])
        tq.tq_compress_device_params(g, s["params"], levels, mode, s["seed"], d=d, packed=s["packed"])
        if case["kind"] == "round":
            tq.tq_decompress_aggregate_device_params(s["packed"], d, s["params"], levels, out=s["out"])
    return s["result"]


def work(case):
    """Each gradient element read once, each packed word written (client side) or read (server alone) once, each update
    value written once; the fused optimiser step also reads and writes the weights and the momentum."""
    n, d, bits = case["workers"], case["d"], _BITS[case["levels"]]
    packed = n * d * bits / 8
    update = 4 * d
    if case["kind"] == "server":
        moved = 16 * d if case["form"] == "apply" else update
        return {"bytes": packed + moved, "flops": n * d}
    grad = n * d * (2 if case["dtype"] == "bfloat16" else 4)
    if case["kind"] == "client":
        return {"bytes": grad + packed, "flops": 8 * n * d}
    return {"bytes": grad + packed + update, "flops": 9 * n * d}


def tolerance(case):
    if case["kind"] == "server":
        # fp32 sums of at most 64 terms and, with "apply", three more operations
        return {"rel": 1e-6}
    # The statistics are 32-bit sums; alpha and the levels follow from them and are rounded to fp32, and an element whose
    # random draw lies on its rounding threshold then takes the neighbouring level.  Measured at these sizes with every
    # level moved by one fp32 ulp: up to 1.2e-6 of the packed words (or one word of a small row), the update by 6e-4 of its
    # norm and, where a code changed, by 0.6 of its rms.  With the tail exponent estimated, sum ln|g| from 64-bit logarithms
    # (4e-7 from the kernel's) moves alpha by 3e-6, which is fifty such ulps.
    words = case["workers"] * case["d"] * _BITS[case["levels"]] / 32
    ulps = 1 if case["gamma"] else 50
    return {"rel": 2.5e-3 * (4 if ulps > 1 else 1), "max": 0.99, "differ": 5e-6 * ulps + 4 / words}
