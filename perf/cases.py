"""The work a user of this library has it do, as cases that can be timed.

A case is a dict of plain values; ``call`` says which part of the public API it goes through:

  linear      one decode-time linear layer, threshold to y in one call      spqt_sparsify_gemv
  shared      one index list for several matrices that read the same x      spqt_sparsify, spqt_sparse_gemv
  layer       the linears of a few decoder layers, one call per x           spqt_sparsify_gemv
  dense       one linear layer without sparsity                             spqt_dense_gemv
  batch       2..8 decode rows over the union of their active sets          spqt_sparse_gemm_small
  batch_dense 2..8 rows over all columns (multi-token steps)                spqt_dense_gemm_small
  kq          the two-level format: index list, then the product            spqt_sparsify, spqt_kqw_sparse_gemv
  kq_dense    the two-level format over all columns                         spqt_kqw_dense_gemv
  pack        offline conversion of one matrix                              spqt_pack
  kq_pack     the same into the two-level format                            spqt_kqw_pack
  host        a token step of host-buffer linears, recorded once            HostStep

Weights are N(0, 0.02^2) and activations Laplace(0, 1) (Gaussian into a down-projection, 1 % of the entries times 20
where ``heavy``), the distributions of ``paper_2511_04477_b200/inputs.py``, drawn on the GPU.  Thresholds are the
order statistic of the site's own activations at the wanted sparsity.
"""
import math

import numpy as np
import torch

from paper_2511_04477_b200 import binding as spqt

MAX_WEIGHTS = 28672 * 8192   # weights of the largest matrix of any case


def listed():
    return [
        # the smallest linear of a Llama-3-8B decoder layer (k or v on its own): latency and launches count
        {"name": "kv_1024x4096", "call": "linear", "m": 1024, "n": 4096, "bits": 4, "group": 128, "sparsity": 0.5, "heavy": False, "dist": "laplace"},
        # q, k and v of a Llama-2-13B layer: one index list, three products
        {"name": "qkv_5120_shared", "call": "shared", "m": 5120, "n": 5120, "mats": 3, "bits": 4, "group": 128, "sparsity": 0.4, "heavy": False, "dist": "laplace"},
        # the ordinary decode step: four Llama-3-8B layers (q|k|v, o, gate|up, down), weights larger than L2
        {"name": "layers_8b", "call": "layer", "hidden": 4096, "kv": 1024, "inter": 14336, "copies": 4, "bits": 4, "group": 128, "sparsity": 0.5, "heavy": False},
        # the largest linear: gate or up of a Llama-2-70B layer, with outlier channels
        {"name": "up_28672x8192", "call": "linear", "m": 28672, "n": 8192, "bits": 4, "group": 128, "sparsity": 0.5, "heavy": True, "dist": "laplace"},
        # the smallest format at sizes that divide nothing: odd n, 173 block-rows
        {"name": "int3_g64_11072x4099", "call": "linear", "m": 11072, "n": 4099, "bits": 3, "group": 64, "sparsity": 0.25, "heavy": False, "dist": "laplace"},
        # a layer kept dense: the down-projection of a Llama-2-70B layer
        {"name": "dense_8192x28672", "call": "dense", "m": 8192, "n": 28672, "bits": 4, "group": 128, "sparsity": 0.0, "heavy": False, "dist": "gauss"},
        # beam search with four beams on the stacked gate|up matrix of a Llama-3-8B layer
        {"name": "beams4_28672x4096", "call": "batch", "m": 28672, "n": 4096, "bits": 4, "group": 128, "batch": 4, "beams": True, "sparsity": 0.5, "heavy": False, "dist": "laplace"},
        # eight tokens at once (a short prompt, speculative tokens) on the down-projection of a Llama-3-8B layer
        {"name": "rows8_dense_4096x14336", "call": "batch_dense", "m": 4096, "n": 14336, "bits": 4, "group": 128, "batch": 8, "beams": False, "sparsity": 0.0, "heavy": False, "dist": "gauss"},
        # the format the paper's implementation builds on, gate|up of a Llama-3-8B layer at 50 %
        {"name": "kq4_28672x4096", "call": "kq", "m": 28672, "n": 4096, "bits": 4, "sparsity": 0.5, "heavy": False, "dist": "laplace"},
        # the same family with 6-bit codes, dense: an attention matrix of a Llama-2-70B layer
        {"name": "kq6_dense_8192x8192", "call": "kq_dense", "m": 8192, "n": 8192, "bits": 6, "sparsity": 0.0, "heavy": False, "dist": "laplace"},
        # converting a model: the largest matrix of a Llama-2-70B layer
        {"name": "pack_28672x8192", "call": "pack", "m": 28672, "n": 8192, "bits": 4, "group": 128},
        # a serving loop whose activations live in host memory: the linears of two Llama-3-8B layers
        {"name": "host_step_8b", "call": "host", "hidden": 4096, "kv": 1024, "inter": 14336, "copies": 2, "bits": 4, "group": 128, "sparsity": 0.5, "heavy": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(("linear", "linear", "linear", "shared", "layer", "dense", "dense", "batch", "batch", "batch_dense", "kq", "kq_dense", "pack", "kq_pack", "host"))
    if call in ("layer", "host"):
        group = rng.choice((64, 128))
        hidden = 128 * max(8, _log(rng, 1024, 8192) // 128)
        kv = 128 * max(1, int(hidden / rng.choice((1, 4, 8))) // 128)
        inter = 128 * int(hidden * rng.uniform(2.6, 3.6) / 128)
        weights = hidden * (2 * hidden + 2 * kv) + 3 * hidden * inter
        copies = max(1, min(4, int(2.2e8 * 2 / weights)))
        return {"call": call, "hidden": hidden, "kv": kv, "inter": inter, "copies": copies, "bits": rng.choice((3, 4, 4)), "group": group,
                "sparsity": round(rng.uniform(0.25, 0.65), 2), "heavy": rng.random() < 0.3}
    two_level = call.startswith("kq")
    group = 256 if two_level else rng.choice((64, 128, 128))
    rows = _log(rng, 1024, 28672)
    n = _log(rng, 1024, 28672)
    if rng.random() < 0.6:
        n = 32 * (n // 32)      # most models; the rest are odd and ragged
    rows = min(rows, (MAX_WEIGHTS // 2 if call == "kq_pack" else MAX_WEIGHTS) // n)
    c = {"call": call, "m": group * max(1, rows // group), "n": n, "bits": rng.choice((2, 4, 4, 5, 6, 8)) if two_level else rng.choice((3, 4, 4))}
    if not two_level:
        c["group"] = group
    if call in ("pack", "kq_pack"):
        return c
    c["sparsity"] = 0.0 if "dense" in call else round(rng.uniform(0.1, 0.7), 2)
    c["heavy"] = rng.random() < 0.3
    c["dist"] = rng.choice(("laplace", "gauss"))
    if call == "shared":
        c["mats"] = rng.choice((2, 3))
        c["m"] = group * max(1, c["m"] // 3 // group)
    if call.startswith("batch"):
        c["batch"] = rng.randint(2, 8)
        c["beams"] = rng.random() < 0.6
    return c


# ---------------------------------------------------------------- inputs


def _weights(g, m, n):
    return torch.randn((m, n), generator=g, device="cuda", dtype=torch.float16).mul_(0.02)


def _activations(g, shape, dist, heavy):
    x = torch.randn(shape, generator=g, device="cuda")
    if dist == "laplace":
        u = torch.rand(shape, generator=g, device="cuda").clamp_(1e-7, 1.0)
        x = torch.sign(x) * -torch.log(u)
    if heavy:
        x = torch.where(torch.rand(shape, generator=g, device="cuda") < 0.01, x * 20.0, x)
    return x


def _threshold(x, sparsity):
    return float(spqt.spqt_calibrate_threshold(x.reshape(-1), sparsity)[0])


def _sites(case):
    """(m, n, distribution) of the matrices of a layer, stacked where they read the same x."""
    h, kv, inter = case["hidden"], case["kv"], case["inter"]
    return [(h + 2 * kv, h, "laplace"), (h, h, "laplace"), (2 * inter, h, "laplace"), (h, inter, "gauss")]


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    call = case["call"]
    state = {"call": call}
    if call in ("pack", "kq_pack"):
        state["W"] = _weights(g, case["m"], case["n"])
        state["bits"], state["group"] = case["bits"], case.get("group")
        return state
    if call in ("layer", "host"):
        sites = []
        for _ in range(case["copies"]):
            for m, n, dist in _sites(case):
                p = spqt.spqt_pack(_weights(g, m, n), case["bits"], case["group"])
                x = _activations(g, n, dist, case["heavy"]).half()
                t = _threshold(x, case["sparsity"])
                if call == "host":
                    lin = spqt.HostLinear(p)
                    lin.x_host.copy_(x)
                    sites.append((lin, t))
                else:
                    buffers = {"idx": torch.zeros(n, dtype=torch.int32, device="cuda"), "count": torch.zeros(1, dtype=torch.int32, device="cuda"),
                               "y": torch.zeros(m, dtype=torch.float16, device="cuda")}
                    sites.append((p, x, t, spqt.new_workspace(m, n, case["bits"], case["group"]), buffers))
        state["sites"] = sites
        if call == "host":
            state["step"] = spqt.HostStep([s[0] for s in sites], [s[1] for s in sites])
        return state
    m, n = case["m"], case["n"]
    state["idx"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    state["count"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    if call.startswith("batch"):
        rows = (case["batch"], n)
        if case["beams"]:   # beams share a prefix: one base vector and a smaller part of each row's own
            x = _activations(g, (1, n), case["dist"], case["heavy"]) + 0.2 * _activations(g, rows, case["dist"], False)
        else:
            x = _activations(g, rows, case["dist"], case["heavy"])
    else:
        x = _activations(g, n, case["dist"], case["heavy"])
    state["x"] = x.half()
    state["t"] = _threshold(state["x"], case["sparsity"])
    if call.startswith("kq"):
        state["p"] = spqt.spqt_kqw_pack(_weights(g, m, n), case["bits"])
        state["ws"] = spqt.new_kq_workspace(state["p"])
        return state
    state["p"] = [spqt.spqt_pack(_weights(g, m, n), case["bits"], case["group"]) for _ in range(case.get("mats", 1))]
    if call.startswith("batch"):
        state["ws"] = spqt.new_gemm_small_workspace(state["p"][0])
    else:
        state["ws"] = spqt.new_workspace(m, n, case["bits"], case["group"])
    return state


# ---------------------------------------------------------------- one pass


def run(state):
    call = state["call"]
    if call == "layer":
        return [spqt.spqt_sparsify_gemv(p, x, t, ws, **buffers) for p, x, t, ws, buffers in state["sites"]]
    if call == "host":
        state["step"].launch()
        torch.cuda.current_stream().synchronize()   # the results are in host memory only then
        return [lin.y_host for lin, _ in state["sites"]]
    if call == "pack":
        p = spqt.spqt_pack(state["W"], state["bits"], state["group"])
        return [p.codes, p.scale_zero.view(torch.int16)]
    if call == "kq_pack":
        return spqt.spqt_kqw_pack(state["W"], state["bits"]).records
    p, x, t, ws, idx, count = (state[k] for k in ("p", "x", "t", "ws", "idx", "count"))
    if call == "linear":
        return spqt.spqt_sparsify_gemv(p[0], x, t, ws, idx, count)
    if call == "shared":
        spqt.spqt_sparsify(x, t, idx, count)
        return [spqt.spqt_sparse_gemv(q, x, idx, count, ws) for q in p] + [idx, count]
    if call == "dense":
        return spqt.spqt_dense_gemv(p[0], x, ws)
    if call == "batch":
        return spqt.spqt_sparse_gemm_small(p[0], x, t, ws, idx, count)
    if call == "batch_dense":
        return spqt.spqt_dense_gemm_small(p[0], x, ws)
    if call == "kq":
        spqt.spqt_sparsify(x, t, idx, count)
        return spqt.spqt_kqw_sparse_gemv(p, x, idx, count, ws), idx, count
    if call == "kq_dense":
        return spqt.spqt_kqw_dense_gemv(p, x, ws)
    raise ValueError("unknown call %r" % (call,))


# ---------------------------------------------------------------- what a pass cannot do without


def _union(case):
    """Share of the columns active in at least one row of a batch."""
    if case["sparsity"] <= 0.0:
        return 1.0
    r = np.random.default_rng(7)
    shape = (case["batch"], 8192)
    one = (lambda s: r.laplace(size=s)) if case["dist"] == "laplace" else (lambda s: r.standard_normal(s))
    x = one((1, shape[1])) + 0.2 * one(shape) if case["beams"] else one(shape)
    a = np.abs(x)
    return float((a > np.quantile(a, case["sparsity"])).any(axis=0).mean())


def _product(m, n, block_rows, block_bytes, share, rows):
    """Active blocks, x, the list read or written once, y."""
    count = share * n
    listed_bytes = 0 if share >= 1.0 else 4 * count + 4
    return count * (m / block_rows) * block_bytes + rows * 2 * (n + m) + listed_bytes, 2.0 * rows * count * m


def work(case):
    call, bits = case["call"], case["bits"]
    if call == "pack":
        w, G = case["m"] * case["n"], case["group"]
        return {"bytes": 2 * w + w // G * (G * bits // 8 + 4), "flops": 4.0 * w}
    if call == "kq_pack":
        w = case["m"] * case["n"]
        return {"bytes": 2 * w + w // 256 * (32 * bits + 16), "flops": 4.0 * w}
    share = 1.0 - case["sparsity"]
    if call in ("layer", "host"):
        parts = [_product(m, n, case["group"], case["group"] * bits // 8 + 4, share, 1) for m, n, _ in _sites(case)] * case["copies"]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    rows = 1
    if call.startswith("batch"):
        rows, share = case["batch"], _union(case)
    if call.startswith("kq"):
        nbytes, flops = _product(case["m"], case["n"], 256, 32 * bits + 16, share, 1)
    else:
        nbytes, flops = _product(case["m"], case["n"], case["group"], case["group"] * bits // 8 + 4, share, rows)
    return {"bytes": nbytes * case.get("mats", 1), "flops": flops * case.get("mats", 1)}


def tolerance(case):
    # packed bytes are defined bit for bit; y is fp16 (2^-11 of rounding) behind fp32 sums
    if case["call"] in ("pack", "kq_pack"):
        return "exact"
    return {"rel": 5e-4, "max": 2e-3}
