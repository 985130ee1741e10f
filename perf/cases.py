"""The work that users of this compressor have it do, as cases that can be timed.

A case names an operation, a shape, an error bound and the kind of field it works on;
`prepare` makes the inputs on the GPU, `run` is one pass through the public binding
(`paper_2105_12912_gb300.api`), `work` says what the pass cannot do without, and
`exact` gives the computed numbers (reconstructions, trained weights) in 64 bits.

Shapes and fields are those of this repository's configurations, tests and benchmark:
1-D traces of 1e4 elements and more, the 1800x3600 climate grid, 100x500x500 weather
fields, the 512^3 density, batches of many uneven fields, double-precision fields and
globally predicted ones.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2105_12912_gb300 import api, selector, synth


def listed():
    return [
        # The smallest call: a short trace of a particle code or a probe, compressed and
        # read back within a time step.  Launches, synchronisations and the code books'
        # latency are all there is to it.
        {"name": "round_trip_1d_10k", "op": "round_trip", "kind": "walk", "dims": "10007", "eb": 1e-3,
         "select": "exhaustive"},
        # An ordinary 1-D trace (the 2^20-element configuration) through the plain calls:
        # the workspace is the binding's own, the field read back is allocated per call.
        {"name": "plain_1d_1m", "op": "plain", "kind": "walk", "dims": "1048576", "eb": 1e-3,
         "select": "exhaustive"},
        # One 2-D climate variable on its 1800x3600 grid, a fifth of it exact zeros: the
        # writing side of a simulation's output step.
        {"name": "compress_2d_cesm", "op": "compress", "kind": "grf_patches", "dims": "1800x3600", "eb": 1e-4,
         "select": "exhaustive"},
        # The reading side of the same variable (post-processing, visualisation).
        {"name": "decompress_2d_cesm", "op": "decompress", "kind": "grf_patches", "dims": "1800x3600", "eb": 1e-4,
         "select": "exhaustive"},
        # The largest single field of the configurations: a cosmology snapshot's 512^3
        # density, the benchmark's own workload; the caller keeps its buffers.
        {"name": "compress_3d_512", "op": "compress_kept", "kind": "lognormal", "dims": "512x512x512", "eb": 1e-4,
         "select": "exhaustive"},
        # The same snapshot read back with no host synchronisation (restart, analysis).
        {"name": "decompress_3d_512", "op": "decompress_async", "kind": "lognormal", "dims": "512x512x512",
         "eb": 1e-4, "select": "exhaustive"},
        # A weather field with empty regions, its per-block codec picked by the trained
        # network: ragged extents (100 and 500 are no multiples of 16).
        {"name": "compress_3d_learned", "op": "compress", "kind": "grf_blocks", "dims": "100x500x500", "eb": 1e-3,
         "select": "learned"},
        # A dump of many variables of uneven shape and dimensionality as one batch,
        # planned once and replayed every output step.
        {"name": "batch_compress_40", "op": "batch_compress", "fields": 40, "scale": 0.1, "shapes": 100},
        # Reading such a dump back.
        {"name": "batch_decompress_40", "op": "batch_decompress", "fields": 40, "scale": 0.1, "shapes": 100},
        # Double-precision fields (SDRBench holds them): written and read back.
        {"name": "round_trip_f64_256", "op": "plain", "kind": "lognormal", "dims": "256x256x256", "eb": 1e-4,
         "select": "exhaustive", "f64": True},
        # Global prediction for smooth fields, chosen where archive size matters most:
        # written and read back.
        {"name": "round_trip_global_3d", "op": "plain", "kind": "grf_blocks", "dims": "100x500x500", "eb": 1e-3,
         "select": "exhaustive", "global": True},
        # Training the codec selector on the blocks of a few fields: full-batch Adam steps.
        {"name": "train_selector", "op": "train", "fields": 4, "dims": "100x500x500", "eb": 1e-3, "steps": 50},
    ]


_KINDS = {1: ("walk", "grf_blocks"), 2: ("grf_patches", "grf_blocks", "lognormal"), 3: ("grf_blocks", "lognormal")}


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_dims(rng, nd, n):
    """A shape of nd extents with about n elements, odd and ragged extents among them."""
    if nd == 1:
        return (max(64, int(n)),)
    # the extents' ratios vary by up to a factor of four either way
    cuts = [_log_uniform(rng, 0.5, 2.0) for _ in range(nd)]
    scale = (n / float(np.prod(cuts))) ** (1.0 / nd)
    return tuple(max(8, int(round(scale * c))) for c in cuts)


def draw(rng):
    """One more case: the operation by how often it is used, sizes log-uniform over the
    operation's range (10^4 elements to 512^3), bounds and selections that users set."""
    op = rng.choices(("round_trip", "plain", "compress", "decompress", "compress_kept", "decompress_async",
                      "batch_compress", "batch_decompress", "train"), (2, 3, 3, 3, 2, 2, 1, 1, 1))[0]
    if op in ("batch_compress", "batch_decompress"):
        return {"op": op, "fields": rng.randint(8, 40), "scale": round(_log_uniform(rng, 0.005, 0.1), 4),
                "shapes": rng.randrange(1000, 5000)}
    if op == "train":
        z, y, x = (rng.randint(32, 100), rng.randint(100, 500), rng.randint(100, 500))
        return {"op": op, "fields": rng.randint(1, 4), "dims": f"{z}x{y}x{x}", "eb": rng.choice((1e-2, 1e-3, 1e-4)),
                "steps": rng.randint(10, 50)}
    nd = rng.randint(1, 3)
    kind = rng.choice(_KINDS[nd])
    variant = rng.choices(("f32", "f64", "global"), (4, 1, 1))[0] if op == "plain" else "f32"
    most = {"f32": 512 ** 3 if op in ("compress_kept", "decompress_async") else 1 << 25,
            "f64": 256 ** 3, "global": 25_000_000}[variant]
    if op == "round_trip":
        most = 1 << 22
    case = {"op": op, "kind": kind, "eb": rng.choice((1e-2, 1e-3, 1e-4)),
            "select": rng.choices(("exhaustive", "learned", "heuristic", "huff", "rle_huff"), (5, 2, 2, 1, 1))[0]}
    dims = _draw_dims(rng, nd, _log_uniform(rng, 1e4, most * 0.98))
    case["dims"] = "x".join(str(d) for d in dims)
    if variant == "f64":
        case["f64"] = True
    if variant == "global":
        case["global"] = True
    return case


# -----------------------------------------------------------------------------------
# inputs
# -----------------------------------------------------------------------------------
def _dims(case):
    return tuple(int(d) for d in case["dims"].split("x"))


def _zero_some_blocks(x, frac, edge, seed):
    """About frac of the aligned edge^ndim blocks set to exactly 0 (empty regions)."""
    g = torch.Generator(device=x.device)
    g.manual_seed(seed)
    mask = torch.rand([-(-s // edge) for s in x.shape], generator=g, device=x.device) < frac
    mask.view(-1)[0] = False  # never a whole field: its value range would be empty
    for d in range(x.dim()):
        mask = mask.repeat_interleave(edge, dim=d)
    return x.masked_fill(mask[tuple(slice(0, s) for s in x.shape)], 0.0).contiguous()


def _field(kind, dims, seed, frac=None, beta=None):
    n = int(np.prod(dims))
    if kind == "walk":
        return synth.walk_sines(n, seed, "cuda").reshape(dims)
    if kind == "lognormal":
        return torch.exp(1.5 * synth.grf(dims, 2.5 if beta is None else beta, seed, "cuda")).contiguous()
    x = synth.grf(dims, 3.0 if beta is None else beta, seed, "cuda")
    if frac is None:
        frac = 0.2 if kind == "grf_patches" else float(np.random.default_rng(seed).uniform(0.0, 0.6))
    return _zero_some_blocks(x, frac, 16 if len(dims) == 3 else 64, seed + 7919)


def _selector_weights(seed):
    """A selector trained as a user trains it, on rows of two small fields of the kind."""
    fields = [(_field("grf_blocks", (48, 96, 96), 9000 + k, 0.3), 1e-3, "rel") for k in range(2)]
    rows = selector.collect_rows(fields)
    w = selector.init_weights(seed % 1000)
    api.selector_train(w, rows["feat"], rows["target"], rows["valid"], steps=40, lr=3e-3)
    return w


def _archive_cap(n):
    """Bytes a program sets aside for the archive of n elements: an element costs at most
    a record of 8 bytes and about one code byte on fields anyone compresses, and the
    books and block tables of a small field fit the rest."""
    return 10 * n + 65536


def _batch_specs(case):
    return synth.workload_batch(case["fields"], seed0=case["shapes"], scale=case["scale"])


def prepare(case, seed):
    op = case["op"]
    s = {"case": case}
    if op in ("batch_compress", "batch_decompress"):
        specs = _batch_specs(case)
        xs = []
        for i, sp in enumerate(specs):
            r = sp.recipe
            xs.append(_field("grf_blocks", sp.dims, seed * 1000 + i, float(r["zero_blocks"]), float(r["beta"])))
        bc = api.BatchCompressor(xs, [sp.eb for sp in specs], archive_caps=[_archive_cap(sp.n) for sp in specs])
        for a in bc.archives:
            a.zero_()  # bytes behind an archive's end stay as the caller left them
        if op == "batch_compress":
            s["batch"] = bc
            return s
        bc.run()
        sizes, _ = bc.results()
        archives = [a[:nb].clone() for a, nb in zip(bc.archives, sizes)]
        s["batch"] = api.BatchDecompressor(archives, [sp.dims for sp in specs])
        return s
    if op == "train":
        fields = [(_field("grf_blocks", _dims(case), seed * 16 + k), case["eb"], "rel") for k in range(case["fields"])]
        rows = selector.collect_rows(fields)
        s.update(feat=rows["feat"].contiguous(), target=rows["target"].contiguous(), valid=rows["valid"].contiguous(),
                 start=selector.init_weights(seed % 100000))
        return s
    dims = _dims(case)
    x = _field(case["kind"], dims, seed)
    if case.get("f64"):
        # a double field has digits below single precision
        x = x.double() * (1.0 + 1e-9 * math.pi)
    kw = {"select": case["select"]}
    if case["select"] == "learned":
        kw["weights"] = _selector_weights(seed)
    if case.get("global"):
        kw["global_lorenzo"] = True
    s["kw"] = kw
    if op in ("decompress", "decompress_async"):
        ar, nb, hdr = api.compress_with_header(x, case["eb"], **kw)
        s.update(archive=ar[:nb].clone(), nbytes=nb, header=hdr, out=torch.empty_like(x),
                 status=torch.zeros(1, dtype=torch.int32, device="cuda"))
        if op == "decompress_async":
            s["ws"] = api.Workspace()
        return s
    s["x"] = x
    # bytes behind an archive's end stay as the caller left them
    s["out"] = torch.zeros(_archive_cap(x.numel()), dtype=torch.uint8, device="cuda")
    if op in ("compress_kept", "round_trip"):
        s["ws"] = api.Workspace()
    if op == "round_trip":
        s["y"] = torch.empty_like(x)
        s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    return s


# -----------------------------------------------------------------------------------
# one pass
# -----------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    op = case["op"]
    if op == "batch_compress":
        b = state["batch"]
        b.run()
        sizes, statuses = b.results()  # a user needs the sizes to write the archives
        return {"archives": list(b.archives), "sizes": np.array(sizes, dtype=np.int64),
                "statuses": np.array(statuses, dtype=np.int64)}
    if op == "batch_decompress":
        b = state["batch"]
        b.run()
        return {"fields": list(b.outs), "statuses": np.array(b.results(), dtype=np.int64)}
    if op == "train":
        w = state["start"].clone()
        loss = api.selector_train(w, state["feat"], state["target"], state["valid"], steps=case["steps"], lr=3e-3)
        return {"weights": w, "loss": float(loss)}
    kw = state["kw"]
    if op == "compress":
        ar, nb, _ = api.compress(state["x"], case["eb"], out=state["out"], **kw)
        return {"archive": ar, "nbytes": nb}
    if op == "compress_kept":
        ar, nb, hdr = api.compress_with_header(state["x"], case["eb"], out=state["out"], workspace=state["ws"], **kw)
        return {"archive": ar, "nbytes": nb, "header": np.frombuffer(hdr, dtype=np.uint8)}
    if op == "decompress":
        y, _ = api.decompress(state["archive"], state["nbytes"])
        return y
    if op == "decompress_async":
        api.decompress_async(state["archive"], state["nbytes"], state["header"], state["out"], state["status"],
                             workspace=state["ws"])
        return {"field": state["out"], "status": state["status"]}
    if op == "round_trip":
        ar, nb, hdr = api.compress_with_header(state["x"], case["eb"], out=state["out"], workspace=state["ws"], **kw)
        api.decompress_async(ar, nb, hdr, state["y"], state["status"], workspace=state["ws"])
        return {"archive": ar, "nbytes": nb, "field": state["y"], "status": state["status"]}
    # plain: both plain calls
    ar, nb, _ = api.compress(state["x"], case["eb"], out=state["out"], **kw)
    y, _ = api.decompress(ar, nb)
    return {"archive": ar, "nbytes": nb, "field": y}


# -----------------------------------------------------------------------------------
# what a pass cannot do without
# -----------------------------------------------------------------------------------
def work(case):
    """The field read once and the archive written once (compression), the archive read
    and the field written (decompression); an archive is about a seventh of its FP32
    field over these kinds and bounds.  Training reads every row at every step and
    multiplies it through the network forwards and backwards."""
    op = case["op"]
    if op in ("batch_compress", "batch_decompress"):
        n = sum(int(np.prod(sp.dims)) for sp in _batch_specs(case))
        return {"bytes": 4.0 * n * (1 + 1 / 7), "flops": 0.0}
    if op == "train":
        z, y, x = _dims(case)
        rows = case["fields"] * -(-z // 16) * -(-y // 16) * -(-x // 16)
        return {"bytes": float(rows * (8 + 3) * 4 + rows) * case["steps"],
                "flops": 6.0 * api.MLP_PARAMS * rows * case["steps"]}
    n = int(np.prod(_dims(case)))
    one = (8.0 if case.get("f64") else 4.0) * n + 4.0 * n / 7
    return {"bytes": one * (2 if op in ("plain", "round_trip") else 1), "flops": 0.0}


# -----------------------------------------------------------------------------------
# the computed numbers in 64 bits
# -----------------------------------------------------------------------------------
def _reconstruction(x, eb_rel, f64):
    """The value each element is rebuilt as: the nearest multiple of the quantization
    step, twice the bound (the bound is eb times the value range, for FP32 fields
    rounded down to a float)."""
    lo, hi = float(x.min()), float(x.max())
    eb = eb_rel * (hi - lo)
    if f64:
        step = 2.0 * eb * (1.0 - 2.0 ** -24)
    else:
        f = np.float32(eb)
        if float(f) > eb:
            f = np.nextafter(f, np.float32(0))
        step = 2.0 * float(f)
    return torch.round(x.double() / step) * step


def _train_exact(state, steps, lr):
    """Full-batch Adam on the 8-32-32-3 network, mean squared error over the valid rows."""
    keep = state["valid"].bool()
    x, t = state["feat"][keep].double(), state["target"][keep].double()
    w = state["start"].double().clone()
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    loss = 0.0
    for k in range(1, steps + 1):
        p = w.clone().requires_grad_(True)
        w1, b1, w2, b2, w3, b3 = torch.split(p, [256, 32, 1024, 32, 96, 3])
        h = torch.relu(x @ w1.view(32, 8).T + b1)
        h = torch.relu(h @ w2.view(32, 32).T + b2)
        e = ((h @ w3.view(3, 32).T + b3 - t) ** 2).mean()
        e.backward()
        loss, g = float(e.detach()), p.grad
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        rate = lr * (1.0 - 0.9 * (k - 1) / steps)
        w = w - rate * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
    return w, loss


def exact(case, seed):
    op = case["op"]
    if op in ("compress", "compress_kept", "batch_compress"):
        return None  # archives are bytes
    if op == "batch_decompress":
        specs = _batch_specs(case)
        fields = []
        for i, sp in enumerate(specs):
            r = sp.recipe
            x = _field("grf_blocks", sp.dims, seed * 1000 + i, float(r["zero_blocks"]), float(r["beta"]))
            fields.append(_reconstruction(x, sp.eb, False))
        return {"fields": fields, "statuses": None}
    if op == "train":
        w, loss = _train_exact(prepare(case, seed), case["steps"], 3e-3)
        return {"weights": w, "loss": loss}
    x = _field(case["kind"], _dims(case), seed)
    if case.get("f64"):
        x = x.double() * (1.0 + 1e-9 * math.pi)
    y = _reconstruction(x, case["eb"], bool(case.get("f64")))
    if op == "decompress":
        return y
    if op == "decompress_async":
        return {"field": y, "status": None}
    if op == "round_trip":
        return {"archive": None, "nbytes": None, "field": y, "status": None}
    return {"archive": None, "nbytes": None, "field": y}
