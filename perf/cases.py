"""The work this framework is used for, as cases that can be timed: post-training quantization of layers.

A case is one call a user's program makes over and over while it walks a network: a single layer from its weights and
calibration activations, a layer replayed as a CUDA graph, a convolution given by its feature maps, a layer whose inputs
sit in host memory, a whole network's layers side by side, and the two variants of the column loop.  What the program
keeps between calls (output buffers, workspace, graph, landing buffers) is made in ``prepare``.

Sizes are those of the repository's workloads (``workloads.py``) and generic ones in between.  Weights are
Kaiming-normal; activations are non-negative (post-ReLU), SiLU-shaped, sparse or normal, as in ``workloads.py``.
"""
import math

import torch

from paper_2509_05576_b200 import ptq, workloads as wl

# Score modes that are used in earnest: the method's own key, and the others of its ordering study.
_MODES = {"qerr": ptq.SCORE_QERR, "prune": ptq.SCORE_PRUNE, "err": ptq.SCORE_ERR, "w": ptq.SCORE_W,
          "qerr_asc": ptq.SCORE_QERR + ptq.SCORE_ASCENDING}


def listed():
    return [
        # a small linear layer: twenty-odd launches, nothing else to it
        dict(name="layer 64x128", kind="layer", rows=64, cols=128, n=1024, bits=4, x="halfnormal", mode="qerr"),
        # the 7x7 stem of a ResNet, the path of the layer replayed as one CUDA graph; an odd number of columns
        dict(name="graph 64x147", kind="graph", rows=64, cols=147, n=4096, bits=4, x="normal", mode="qerr"),
        # the 3x3 convolution the benchmark is quoted on
        dict(name="layer 256x2304", kind="layer", rows=256, cols=2304, n=4096, bits=4, x="sparse", mode="qerr"),
        # the widest convolution of both networks, 8-bit, long calibration input
        dict(name="layer 512x4608 8-bit", kind="layer", rows=512, cols=4608, n=8192, bits=8, x="silu", mode="qerr"),
        # a classifier: rows that are no multiple of a tile; ordered by the plain rounding error
        dict(name="layer 1000x2048 err", kind="layer", rows=1000, cols=2048, n=4096, bits=4, x="halfnormal", mode="err"),
        # square projection of a large model, 3-bit
        dict(name="layer 4096x4096 3-bit", kind="layer", rows=4096, cols=4096, n=8192, bits=3, x="normal", mode="qerr"),
        # the largest layer of the scaling shapes
        dict(name="layer 4096x11008", kind="layer", rows=4096, cols=11008, n=8192, bits=4, x="normal", mode="qerr"),
        # every layer of a ResNet-50, side by side on several streams
        dict(name="set resnet50", kind="set", config=3, first=0, count=54),
        # a convolution given by its feature maps (3x3 on 14x14 maps, 21 images), read in place
        dict(name="conv 256x256x3x3", kind="conv", rows=256, channels=256, k=3, stride=1, pad=1, size=14, batch=21, bits=4,
             x="halfnormal", mode="qerr"),
        # the same layer with weights and two calibration batches in pinned host memory
        dict(name="host 256x2304", kind="host", rows=256, cols=2304, n=4096, bits=4, x="sparse", mode="qerr"),
        # re-ranking of the remaining columns while the loop runs
        dict(name="dynamic 128x1152", kind="dynamic", rows=128, cols=1152, n=4096, bits=4, x="halfnormal", mode="qerr",
             block=128),
        # the non-parallel arm: every row in its own order
        dict(name="per-row 512x128", kind="per_row", rows=512, cols=128, n=4096, bits=4, x="halfnormal", mode="qerr"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer"] * 5 + ["graph", "conv", "host", "set", "dynamic", "per_row"])
    c = dict(kind=kind, bits=rng.choice([3, 4, 8]), x=rng.choice(["halfnormal", "silu", "sparse", "normal"]),
             mode=rng.choice(["qerr"] * 3 + ["prune", "err", "w", "qerr_asc"]))
    n = _log(rng, 512, 8192)
    if kind == "set":
        # a run of consecutive layers of one of the networks
        config = rng.choice([3, 4, 6, 7])
        total = len(_set_specs(config))
        count = rng.randint(8, min(total, 54))
        return dict(kind=kind, config=config, first=rng.randint(0, total - count), count=count)
    if kind == "conv":
        k, stride = rng.choice([(1, 1), (1, 2), (3, 1), (3, 2)])
        channels = _log(rng, 16, 2048) if k == 1 else _log(rng, 3, 512)
        size = rng.randint(7, 56)
        out = (size + 2 * (k // 2) - k) // stride + 1
        return dict(c, rows=_log(rng, 16, 1024), channels=channels, k=k, stride=stride, pad=k // 2, size=size,
                    batch=max(1, n // (out * out)))
    if kind == "graph":
        return dict(c, rows=_log(rng, 16, 512), cols=_log(rng, 27, 1152), n=n)
    if kind == "host":
        return dict(c, rows=_log(rng, 32, 1024), cols=_log(rng, 64, 4608), n=2 * (n // 2))
    if kind == "dynamic":
        return dict(c, rows=_log(rng, 16, 1024), cols=_log(rng, 130, 2304), n=n, block=rng.choice([64, 128, 256]))
    if kind == "per_row":
        return dict(c, rows=_log(rng, 16, 1024), cols=rng.randint(16, 128), n=n)
    return dict(c, rows=_log(rng, 16, 4096), cols=_log(rng, 48, 8192), n=n)


def _set_specs(config):
    return wl.config4(bits=(4,)) if config == 4 else wl.CONFIGS[config]()


def _activations(shape, dist, g):
    x = torch.randn(shape, dtype=torch.float32, device="cuda", generator=g)
    if dist == "halfnormal":
        x.abs_()
    elif dist in ("sparse", "halfnormal_sparse30"):
        x.abs_().mul_(torch.rand(shape, dtype=torch.float32, device="cuda", generator=g) >= 0.3)
    elif dist == "silu":
        x = torch.nn.functional.silu(x)
    return x


def _weights(rows, cols, g):
    return torch.randn((rows, cols), dtype=torch.float32, device="cuda", generator=g) * math.sqrt(2.0 / cols)


def _conv_cols_n(case):
    k = case["k"]
    return ptq.conv_unfolded_shape((case["batch"], case["channels"], case["size"], case["size"]), k, k, case["stride"],
                                   case["pad"])


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "set":
        specs = _set_specs(case["config"])[case["first"]:case["first"] + case["count"]]
        layers = [(_weights(p.rows, p.cols, g), _activations((p.cols, p.n), p.x_dist, g), p.bits, p.damp) for p in specs]
        s["set"] = ptq.LayerSet(layers)
        # the program wants the network's results in one piece: every layer's outputs are views into shared buffers
        dev, rows, cols = "cuda", [p.rows for p in specs], [p.cols for p in specs]
        size = {"codes": [r * c for r, c in zip(rows, cols)], "What": [r * c for r, c in zip(rows, cols)], "perm": cols,
                "scale": rows, "zero": rows, "loss": [1] * len(specs)}
        flat = {}
        for key, counts in size.items():
            like = getattr(s["set"].bufs[0], key)
            starts, at = [], 0
            for m in counts:
                starts.append(at)
                at += (m + 63) // 64 * 64                  # every layer's piece starts on an aligned address
            flat[key] = torch.zeros(at, dtype=like.dtype, device=dev)
            for b, start, m in zip(s["set"].bufs, starts, counts):
                setattr(b, key, flat[key][start:start + m].view(getattr(b, key).shape))
        s["flat"] = flat
        return s
    if kind == "conv":
        k = case["k"]
        cols, _ = _conv_cols_n(case)
        s["W"] = _weights(case["rows"], cols, g)
        s["X"] = _activations((case["batch"], case["channels"], case["size"], case["size"]), case["x"], g)
        s["conv"] = (k, k, case["stride"], case["pad"])
    else:
        cols = case["cols"]
        s["W"] = _weights(case["rows"], cols, g)
        s["X"] = _activations((cols, case["n"]), case["x"], g)
    s["mode"] = _MODES[case["mode"]]
    s["ws"] = ptq.Workspace()
    s["bufs"] = ptq.LayerBuffers(case["rows"], cols)
    if kind == "graph":
        s["graph"] = ptq.LayerGraph(s["W"], s["X"], case["bits"], score_mode=s["mode"], bufs=s["bufs"], ws=s["ws"])
    elif kind == "host":
        half = case["n"] // 2
        s["W_host"] = s.pop("W").cpu().pin_memory()
        x = s.pop("X")
        s["X_host"] = [x[:, :half].contiguous().cpu().pin_memory(), x[:, half:].contiguous().cpu().pin_memory()]
        s["staging"] = ptq.HostStaging(case["rows"], cols, [half, case["n"] - half])
    elif kind == "dynamic":
        s["order"] = torch.empty(cols, dtype=torch.int32, device="cuda")
    elif kind == "per_row":
        s["perm_rows"] = torch.empty((case["rows"], cols), dtype=torch.int32, device="cuda")
    return s


def _layer_outputs(b):
    return {k: getattr(b, k) for k in ("H", "Hinv", "Hinv_diag", "lam", "scale", "zero", "S", "perm", "codes", "What", "loss")}


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "set":
        s["set"].run()
        return s["flat"]
    b, ws, bits, mode = s["bufs"], s["ws"], case["bits"], s["mode"]
    if kind == "graph":
        s["graph"].replay()
        return _layer_outputs(b)
    if kind == "host":
        ptq.quantize_layer_from_host(s["W_host"], s["X_host"], bits, score_mode=mode, bufs=b, ws=ws, staging=s["staging"])
        return _layer_outputs(b)
    if kind in ("layer", "conv"):
        ptq.quantize_layer_full(s["W"], s["X"], bits, score_mode=mode, bufs=b, ws=ws, conv=s.get("conv"))
        return _layer_outputs(b)
    # the variants of the column loop, stage by stage as their callers do it
    W, st = s["W"], b.status
    st.zero_()
    b.H.zero_()
    ptq.hessian_accumulate(b.H, s["X"], ws, st)
    ptq.prepare_hinv(b.H, 0.01, ptq.DAMP_REL_MEAN_DIAG, b.Hinv, b.Hinv_diag, b.lam, ws, st)
    ptq.minmax_grid(W, bits, b.scale, b.zero, st)
    out = {k: getattr(b, k) for k in ("H", "Hinv", "Hinv_diag", "lam", "scale", "zero", "codes", "What", "loss")}
    if kind == "dynamic":
        ptq.quantize_layer_dynamic(W, b.Hinv, b.scale, b.zero, bits, mode, case["block"], b.codes, b.What, s["order"], b.H,
                                   b.loss, ws, st)
        out["order"] = s["order"]
    else:
        ptq.quantize_layer_per_row(W, b.Hinv, b.scale, b.zero, bits, mode, b.codes, b.What, s["perm_rows"], b.H, b.loss, ws,
                                   st)
        out["perm_rows"] = s["perm_rows"]
    return out


def _layer_work(rows, cols, n, x_values, chol_rows=1):
    """Inputs once, outputs once; operations of the method: the symmetric Gram, the inverse (cols^3), the factor of the
    permuted inverse (cols^3 / 3, per row for the non-parallel arm), the deferred updates and the loss."""
    out = 16.0 * cols * cols + rows * cols * 5.0 + 20.0 * cols + 8.0 * rows
    return (4.0 * rows * cols + 4.0 * x_values + out,
            float(cols) * (cols + 1) * n + cols ** 3 + chol_rows * cols ** 3 / 3.0 + 3.0 * rows * cols * cols)


def work(case):
    if case["kind"] == "set":
        parts = [_layer_work(p.rows, p.cols, p.n, p.cols * p.n)
                 for p in _set_specs(case["config"])[case["first"]:case["first"] + case["count"]]]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    rows = case["rows"]
    if case["kind"] == "conv":
        cols, n = _conv_cols_n(case)
        x_values = case["batch"] * case["channels"] * case["size"] ** 2
    else:
        cols, n = case["cols"], case["n"]
        x_values = cols * n
    b, f = _layer_work(rows, cols, n, x_values, rows if case["kind"] == "per_row" else 1)
    return {"bytes": b, "flops": f}


def tolerance(case):
    # Everything that decides a rounding or an order is float64.  Measured: this path against itself with the Hessian
    # from plain float64 sums and the inverse from a library factorisation, over the listed cases and drawn ones.  Largest
    # relative error 2.9e-11 and largest single difference 3.8e-10 (the inverse at 6300 columns from 691 calibration
    # columns), 1e-12 and below for most; codes and orders came out the same everywhere.  About four times that, a little
    # more for worse conditioned draws; one weight in 10^5 is left for a value on a rounding boundary.
    return {"rel": 2e-10, "max": 2e-9, "differ": 1e-5}
