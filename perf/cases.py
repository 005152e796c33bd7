"""The work this library does for its users, as cases that can be timed and compared.

A program that uses the library decodes and prefills through quantized linear layers, encodes the layers of a model,
measures per-layer errors for the choice of bit widths, and fits grids.  ``listed`` names one case for each of these
over the range of sizes, ``draw`` gives further ones of the same ranges, ``prepare`` builds what such a program holds
before the call, ``run`` is one pass through the public entry points.
"""
import math
import os

import numpy as np
import torch

import paper_2411_17525_b200 as hb

GROUP = 1024
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(hb.__file__)))

# (name, rows, inputs) of the linear layers of one transformer block
SETS = {
    "1b": [("q", 2048, 2048), ("k", 512, 2048), ("v", 512, 2048), ("o", 2048, 2048),
           ("gate", 8192, 2048), ("up", 8192, 2048), ("down", 2048, 8192)],
    "8b": [("q", 4096, 4096), ("k", 1024, 4096), ("v", 1024, 4096), ("o", 4096, 4096),
           ("gate", 14336, 4096), ("up", 14336, 4096), ("down", 4096, 14336)],
    "70b": [("q", 8192, 8192), ("k", 1024, 8192), ("v", 1024, 8192), ("o", 8192, 8192),
            ("gate", 28672, 8192), ("up", 28672, 8192), ("down", 8192, 28672)],
}
SHARED_INPUT = {"q": "attn", "k": "attn", "v": "attn", "gate": "mlp", "up": "mlp"}
GRIDS = {"2x256": (2, 256), "2x64": (2, 64), "2x16": (2, 16), "1x16": (1, 16), "1x8": (1, 8), "1x4": (1, 4), "1x256": (1, 256)}
# per-matrix grids of a mixed 3/4-bit assignment (q, k, v, o, gate, up, down)
MIXED = ["2x64", "2x64", "2x64", "2x64", "2x256", "2x64", "2x256"]


# ------------------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: one layer, one token, called from Python as it stands
        dict(name="layer 512x1024 b1", kind="layer", N=512, K=1024, B=1, grid="2x256", out="f32"),
        # decode steps, captured once and replayed as a serving loop does: a small model at one token (its launches count) ...
        dict(name="decode 1b b1", kind="decode", set="1b", blocks=8, B=1, grid="2x256", out="f32"),
        # ... a medium one at a few sequences and 3 bits ...
        dict(name="decode 8b b4", kind="decode", set="8b", blocks=2, B=4, grid="2x64", out="f32"),
        # ... at the largest batch of the small-batch range, scalar grid, bf16 outputs ...
        dict(name="decode 8b b16", kind="decode", set="8b", blocks=2, B=16, grid="1x16", out="bf16"),
        # ... and the largest model with mixed bit widths (the benchmark's default step)
        dict(name="decode 70b b1", kind="decode", set="70b", blocks=1, B=1, grid="mixed", out="f32"),
        # the same step for a program whose activations and outputs live in host memory
        dict(name="host 70b b1", kind="host", set="70b", B=1, grid="mixed", out="f32"),
        # many sequences decoded together / speculative and short prompts: the tensor-core range at its small end
        dict(name="batch 8b b64", kind="batch", set="8b", B=64, grid="2x256", out="f32", lognormal=True),
        dict(name="batch 70b b32", kind="batch", set="70b", B=32, grid="mixed", out="f32", lognormal=False),
        # a prompt of ragged length
        dict(name="prefill 8b b1999", kind="batch", set="8b", B=1999, grid="2x256", out="bf16", lognormal=True),
        # encoding the layers of a block, search table prepared once per grid
        dict(name="encode 8b", kind="encode", set="8b", grid="2x256", dtype="bf16"),
        # one layer's rows of the error database behind the choice of bit widths: encode and measure at four widths
        dict(name="errors 14336x4096", kind="errors", N=14336, K=4096, dtype="bf16"),
        # a grid fitted to Gaussian samples until nothing changes
        dict(name="fit 2x256", kind="fit", p=2, n=256, log2_samples=18, max_iters=3000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    out = rng.choice(["f32", "bf16"])
    kind = rng.choice(["layer", "layer", "decode", "decode", "decode", "host", "batch", "batch", "batch", "encode", "errors", "fit"])
    if kind == "layer":
        N, K = 16 * _log_int(rng, 8, 900), 1024 * _log_int(rng, 1, 14)
        return dict(kind=kind, N=N, K=K, B=_log_int(rng, 1, 300), grid=rng.choice(list(GRIDS)), out=out)
    # a block's widths: one of the named sets or a model between them
    size = rng.choice(["1b", "8b", "70b", "other", "other", "other"])
    hidden = rng.randint(1, 7)
    shape = dict(set=size) if size != "other" else dict(hidden=1024 * hidden, kv=128 * rng.randint(2, 8), ffn=1024 * rng.randint(2 * hidden, 4 * hidden))
    weights = sum(N * K for _, N, K in _shapes(shape))
    if kind == "decode":
        return dict(kind=kind, **shape, blocks=max(1, min(8, int(4e8 / weights))), B=_log_int(rng, 1, 16),
                    grid=rng.choice(["2x256", "2x256", "2x64", "2x16", "1x16", "1x8", "mixed", "mixed"]), out=out)
    if kind == "host":
        return dict(kind=kind, **shape, B=_log_int(rng, 1, 16), grid=rng.choice(["2x256", "2x64", "mixed"]), out=out)
    if kind == "batch":
        return dict(kind=kind, **shape, B=_log_int(rng, 17, min(1950, 4e11 / weights)),
                    grid=rng.choice(["2x256", "2x64", "1x16", "2x16", "mixed"]), out=out, lognormal=rng.random() < 0.5)
    if kind == "encode":
        shape = shape if weights < 3e8 else dict(set="8b")
        return dict(kind=kind, **shape, grid=rng.choice(list(GRIDS) + ["mixed"]), dtype=rng.choice(["f32", "bf16"]))
    if kind == "errors":
        return dict(kind=kind, N=16 * _log_int(rng, 16, 890), K=1024 * rng.randint(1, 4), dtype=rng.choice(["f32", "bf16"]))
    p, n = rng.choice([(2, 256), (2, 64), (2, 16), (1, 16), (1, 8), (1, 4)])
    return dict(kind="fit", p=p, n=n, log2_samples=rng.randint(13, 18), max_iters=rng.randint(60, 200))


# ------------------------------------------------------------------------------------------------------ sizes
def _shapes(case):
    if "set" in case:
        return SETS[case["set"]]
    h, kv, f = case["hidden"], case["kv"], case["ffn"]
    return [("q", h, h), ("k", kv, h), ("v", kv, h), ("o", h, h), ("gate", f, h), ("up", f, h), ("down", h, f)]


def _layers(case):
    """(name, rows, inputs, (p, n)) of the matrices a case holds."""
    if "N" in case:
        return [("layer", case["N"], case["K"], GRIDS[case["grid"]])]
    names = MIXED if case["grid"] == "mixed" else [case["grid"]] * 7
    return [(nm, N, K, GRIDS[g]) for (nm, N, K), g in zip(_shapes(case), names)]


def _code_bytes(N, K, p, n):
    return N * K * int(math.log2(n)) // (8 * p) + 2 * N * K // GROUP


ERROR_GRIDS = ["2x16", "2x64", "2x256", "1x256"]


def work(case):
    kind = case["kind"]
    if kind == "fit":
        # samples in, grid out; one assignment pass is the least any fit computes
        m = 1 << case["log2_samples"]
        return {"bytes": 4 * case["p"] * (m + case["n"]) + 8, "flops": 3 * case["p"] * case["n"] * m}
    if kind in ("encode", "errors"):
        grids = ERROR_GRIDS if kind == "errors" else [None]
        size = {"f32": 4, "bf16": 2}[case["dtype"]]
        shapes = _layers(case) if kind == "encode" else [("layer", case["N"], case["K"], GRIDS[g]) for g in grids]
        weights = sum(N * K for _, N, K, _ in shapes)
        read = weights * size if kind == "encode" else case["N"] * case["K"] * size
        # norm and scaling 3, butterflies 10, and per tuple the distance to the one point that is chosen
        return {"bytes": read + sum(_code_bytes(N, K, p, n) + 4 * n * p for _, N, K, (p, n) in shapes), "flops": 16 * weights}
    B, esz = case["B"], {"f32": 4, "bf16": 2}[case["out"]]
    nbytes, flops, seen = 0, 0, set()
    for nm, N, K, (p, n) in _layers(case):
        key = SHARED_INPUT.get(nm, nm)
        nbytes += _code_bytes(N, K, p, n) + 4 * n * p + esz * B * N + (0 if key in seen else 2 * B * K)
        seen.add(key)
        flops += 2 * B * N * K
    return {"bytes": nbytes * case.get("blocks", 1), "flops": flops * case.get("blocks", 1)}


def tolerance(case):
    # Four times what the paths differ by from the same computation in 64 bits (from the given codes and stored scales):
    # fp16 operands 3.7e-4 of the norm and 4.8e-3 at one value, bf16 outputs 1.7e-3 and 7.5e-3; 2.4e-6 of the packed bytes
    # (points within fp32 rounding of two cells), no scale and t^2 by 2e-8.  A fit's points do not depend on the order of
    # its sums (samples permuted: the same points after the same number of iterations).
    kind = case["kind"]
    if kind == "fit":
        return {"rel": 1e-6, "max": 1e-5}
    if kind in ("encode", "errors"):
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-5}
    return {"rel": 1.5e-3, "max": 2e-2} if case["out"] == "f32" else {"rel": 7e-3, "max": 3e-2}


# ------------------------------------------------------------------------------------------------------ inputs
def _grid(p, n):
    """The fitted table of (p, n) that the repository stores."""
    g = np.loadtxt(os.path.join(ROOT, "synth", "grids", f"grid_p{p}_n{n}.txt"), comments="#", ndmin=2)
    return torch.from_numpy(g.astype(np.float32).reshape(n, p)).cuda()


def _generator(seed, k):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * seed + k)


def _weights(N, K, seed, k, dtype):
    """0.02 N(0,1) with one entry in a thousand replaced by 0.1 t(3), as layers with outliers have them."""
    g = _generator(seed, 100 + k)
    W = torch.randn(N, K, device="cuda", generator=g).mul_(0.02)
    m = N * K // 1000
    at = 1000 * torch.arange(m, device="cuda") + torch.randint(1000, (m,), device="cuda", generator=g)      # (no place twice)
    z = torch.randn(4, m, device="cuda", generator=g)
    W.view(-1)[at] = 0.1 * z[0] / (z[1:].square().mean(0)).sqrt()
    return W.to(torch.bfloat16) if dtype == "bf16" else W


def _activations(B, K, seed, k, lognormal=False):
    g = _generator(seed, 500 + k)
    x = torch.randn(B, K, device="cuda", generator=g)
    if lognormal:
        x *= torch.randn(K, device="cuda", generator=g).exp()
    return x.to(torch.bfloat16)


def _out_dtype(case):
    return {"f32": torch.float32, "bf16": torch.bfloat16}[case["out"]]


def _workspace(nbytes):
    return torch.empty(max(nbytes, 256), dtype=torch.uint8, device="cuda")


class _Block:
    """The linear layers of one transformer block for B tokens: layers that read the same input and share a grid are one
    product; otherwise the first of them leaves its rotated activations for the others."""

    def __init__(self, case, seed, index):
        B, dt = case["B"], _out_dtype(case)
        rht = 0x48494747 + seed
        self.B, self.calls, self.ys, self.xs = B, [], {}, {}
        grids = {pn: _grid(*pn) for pn in {pn for *_, pn in _layers(case)}}
        groups = {}
        for i, (nm, N, K, pn) in enumerate(_layers(case)):
            d = hb.make_desc(pn[0], pn[1], N, K, rht)
            W = _weights(N, K, seed, 10 * index + i, "bf16")
            packed, scales, _ = hb.higgs_quantize(d, W, grids[pn])
            del W
            self.ys[nm] = torch.empty(B, N, dtype=dt, device="cuda")
            groups.setdefault(SHARED_INPUT.get(nm, nm), []).append((nm, d, packed, scales, grids[pn], pn))
        for k, (key, members) in enumerate(groups.items()):
            x = _activations(B, members[0][1].K, seed, 10 * index + k, case.get("lognormal", False))
            self.xs[key] = x
            if len(members) > 1 and len({m[5] for m in members}) == 1:
                m = hb.MultiLinear([m[1] for m in members], [m[2] for m in members], [m[3] for m in members], members[0][4],
                                   [self.ys[m[0]] for m in members], B)
                self.calls.append(("multi", m, x))
                continue
            ws = _workspace(max(hb.higgs_workspace_bytes(m[1], hb.HIGGS_OP_LINEAR, B) for m in members))
            xdag, layout = None, None
            for m in members:
                nm, d, packed, scales, grid, _ = m
                if len(members) > 1 and xdag is None:
                    layout = hb.higgs_rotated_layout(d, B)
                    xdag = torch.empty(hb.higgs_rotated_bytes(d, B) // 2, dtype=torch.float16, device="cuda")
                    self.calls.append(("share", d, x, packed, scales, grid, xdag, ws, self.ys[nm]))
                elif len(members) > 1 and hb.higgs_rotated_layout(d, B) == layout:
                    self.calls.append(("rotated", d, xdag, packed, scales, grid, None, ws, self.ys[nm]))
                else:
                    self.calls.append(("plain", d, x, packed, scales, grid, None, ws, self.ys[nm]))

    def __call__(self):
        for c in self.calls:
            if c[0] == "multi":
                hb.higgs_linear_multi(c[1], c[2])
                continue
            how, d, x, packed, scales, grid, xdag, ws, y = c
            if how == "share":
                hb.higgs_linear_share(d, x, packed, scales, grid, xdag_out=xdag, workspace=ws, y=y)
            elif how == "rotated":
                hb.higgs_linear_prerotated(d, x, packed, scales, grid, workspace=ws, y=y, B=self.B)
            else:
                hb.higgs_linear(d, x, packed, scales, grid, workspace=ws, y=y)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "layer":
        p, n = GRIDS[case["grid"]]
        d = hb.make_desc(p, n, case["N"], case["K"], 0x48494747 + seed)
        grid = _grid(p, n)
        packed, scales, _ = hb.higgs_quantize(d, _weights(case["N"], case["K"], seed, 0, "bf16"), grid)
        return dict(case=case, desc=d, grid=grid, packed=packed, scales=scales, x=_activations(case["B"], case["K"], seed, 0))
    if kind == "batch":
        return dict(case=case, block=_Block(case, seed, 0))
    if kind == "decode":
        blocks = [_Block(case, seed, i) for i in range(case["blocks"])]
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(stream):
            for b in blocks:
                b()
            stream.synchronize()
            with torch.cuda.graph(graph, stream=stream):
                for b in blocks:
                    b()
        torch.cuda.current_stream().wait_stream(stream)
        return dict(case=case, blocks=blocks, graph=graph)
    if kind == "host":
        layers = _layers(case)
        grids = {pn: _grid(*pn) for pn in {pn for *_, pn in layers}}
        descs = [hb.make_desc(pn[0], pn[1], N, K, 0x48494747 + seed) for _, N, K, pn in layers]
        packed, scales = [], []
        for i, (d, (_, N, K, pn)) in enumerate(zip(descs, layers)):
            pk, sc, _ = hb.higgs_quantize(d, _weights(N, K, seed, i, "bf16"), grids[pn])
            packed.append(pk)
            scales.append(sc)
        keys = [SHARED_INPUT.get(nm, nm) for nm, *_ in layers]
        widths = {k: K for k, (_, _, K, _) in zip(keys, layers)}
        xs = [(k, _activations(case["B"], K, seed, i).cpu()) for i, (k, K) in enumerate(widths.items())]
        return dict(case=case, step=hb.HostBlock(descs, keys, xs, packed, scales, [grids[pn] for *_, pn in layers], case["B"],
                                                 y_dtype=_out_dtype(case)))
    if kind == "encode":
        layers = _layers(case)
        grids = {pn: _grid(*pn) for pn in {pn for *_, pn in layers}}
        tables = {pn: hb.higgs_make_encoder_table(*pn, g) for pn, g in grids.items()}
        descs = [hb.make_desc(pn[0], pn[1], N, K, 0x48494747 + seed) for _, N, K, pn in layers]
        ws = _workspace(max(hb.higgs_workspace_bytes(d, hb.HIGGS_OP_QUANTIZE) for d in descs))
        Ws = [_weights(N, K, seed, i, case["dtype"]) for i, (_, N, K, _) in enumerate(layers)]
        outs = [(torch.empty(hb.higgs_packed_bytes(d), dtype=torch.uint8, device="cuda"),
                 torch.empty(d.N // 16, d.K // GROUP, 16, dtype=torch.float16, device="cuda")) for d in descs]
        return dict(case=case, jobs=[(d, W, grids[pn], tables[pn], o) for d, W, (*_, pn), o in zip(descs, Ws, layers, outs)], ws=ws)
    if kind == "errors":
        W = _weights(case["N"], case["K"], seed, 0, case["dtype"])
        return dict(case=case, W=W, jobs=[(hb.make_desc(*GRIDS[g], case["N"], case["K"], 0x48494747 + seed), _grid(*GRIDS[g]))
                                          for g in ERROR_GRIDS])
    samples = torch.randn(1 << case["log2_samples"], case["p"], device="cuda", generator=_generator(seed, 0))
    return dict(case=case, samples=samples)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "layer":
        return hb.higgs_linear(state["desc"], state["x"], state["packed"], state["scales"], state["grid"], out_dtype=_out_dtype(case))
    if kind == "batch":
        state["block"]()
        return state["block"].ys
    if kind == "decode":
        state["graph"].replay()
        return [b.ys for b in state["blocks"]]
    if kind == "host":
        hb.higgs_linear_host_block(state["step"])
        torch.cuda.current_stream().synchronize()          # the outputs are read on the host
        return state["step"].y
    if kind == "encode":
        for d, W, grid, table, out in state["jobs"]:
            hb.higgs_quantize(d, W, grid, workspace=state["ws"], out=out, table=table)
        return [out for *_, out in state["jobs"]]
    if kind == "errors":
        got = []
        for d, grid in state["jobs"]:
            packed, scales, _ = hb.higgs_quantize(d, state["W"], grid)
            got.append((packed, scales, hb.higgs_layer_error(d, state["W"], packed, scales, grid)))
        return got
    grid, mse, iters = hb.higgs_make_grid(case["p"], case["n"], state["samples"], max_iters=case["max_iters"])
    return {"grid": grid, "mse": mse, "iters": iters}
