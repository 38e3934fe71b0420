"""The work that users of this library have it do, as cases to be timed.

A case names a call of the public interface (``kind``), a sparse tensor
(mode lengths, index distribution, nonzeros) and the factors (rank, type).
The tensors follow the recipe of the package's generator: distinct coordinates,
uniform or Zipf-distributed per mode with scattered labels, in random order,
as a raw coordinate file has them.

Kinds, by what a program calls:

* ``all``       ``Tensor.mttkrp_all``: the MTTKRP of every mode with one set of
                factors (gradient methods, the paper's all-mode benchmark);
* ``one``       ``Tensor.mttkrp`` of one mode (one step of a CP-ALS sweep);
* ``f64``       ``Tensor.mttkrp_f64`` of every mode, one after another: the
                paper's precision;
* ``step``      forward and backward of the sparse CP model through autograd,
                with the residual against the stored values as the upstream
                gradient: one training step; returns model values and gradients;
* ``build``     ``Tensor.build`` from device coordinates, and the store's keys
                and values (what out-of-core tools save);
* ``als``       ``cp_als``: whole sweeps, from the given factors;
* ``update``    ``blco_cpals_update``: solve, normalization and Gram of one
                factor after its MTTKRP;
* ``streamed``  ``Tensor.mttkrp_all`` on a store held in host memory.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2201_12523_gb300 import blco

_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16, "f64": torch.float64}


def _case(name, kind, dims, dist, nnz, rank, dtype="f32", **more):
    c = {"name": name, "kind": kind, "dims": "x".join(str(d) for d in dims), "dist": dist, "nnz": int(nnz),
         "rank": int(rank), "dtype": dtype}
    c.update(more)
    return c


def listed():
    return [
        # the smallest tensor of the package's workloads: every mode of a
        # tensor that fits in L2, where launches and latency are the cost
        _case("all-3d-100k", "all", (1000, 800, 600), "uniform", 100_000, 16),
        # an ordinary tensor of a few million nonzeros and odd mode lengths
        # with bfloat16 factors: one mode's MTTKRP
        _case("one-4d-3M-bf16", "one", (183, 1140, 20011, 1717), "zipf:1.1", 3_300_017, 32, "bf16", mode=2),
        # the in-memory workloads at rank 32, every mode: three skewed modes,
        # two of them long ...
        _case("all-3d-150M", "all", (1 << 22, 1 << 21, 1 << 11), "zipf:1.2", 150_000_000, 32),
        # ... and four modes, the last one short (half of the benchmark's
        # 500M nonzeros)
        _case("all-4d-250M", "all", (1 << 20, 1 << 18, 1 << 16, 1 << 8), "zipf:1.1", 250_000_000, 32),
        # five modes at rank 16, more than 64 index bits: many blocks
        _case("all-5d-100M", "all", (1 << 24, 1 << 20, 1 << 16, 1 << 12, 1 << 8), "zipf:1.2,zipf:1.2,zipf:1.2,uniform,uniform",
              100_000_000, 16),
        # the same shape out of memory: the store in host memory, streamed
        # through device queues once per call
        _case("streamed-5d-50M", "streamed", (1 << 24, 1 << 20, 1 << 16, 1 << 12, 1 << 8),
              "zipf:1.2,zipf:1.2,zipf:1.2,uniform,uniform", 50_000_000, 16, cap=1 << 23),
        # float64 values, factors and sums, every mode
        _case("f64-3d-20M", "f64", (1 << 20, 1 << 19, 1 << 11), "zipf:1.2", 20_000_000, 32, "f64"),
        # a training step of the CP model at rank 64
        _case("step-3d-50M", "step", (1 << 20, 1 << 20, 1 << 10), "zipf:1.2", 50_000_000, 64),
        # a training step with bfloat16 factors, four modes of odd lengths
        _case("step-4d-6M-bf16", "step", (100_003, 50_021, 3001, 365), "zipf:1.1", 6_000_011, 32, "bf16"),
        # construction of a store from unordered device coordinates
        _case("build-3d-100M", "build", (1 << 22, 1 << 21, 1 << 11), "zipf:1.2", 100_000_000, 32),
        # two whole CP-ALS sweeps with the fit after each
        _case("als-3d-8M", "als", (200_003, 100_019, 2039), "zipf:1.1", 8_000_009, 32, iters=2),
        # the update of one long factor at the largest rank it takes
        _case("update-1M", "update", (1 << 20, 1 << 20, 1 << 10), "uniform", 0, 64, mode=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["all", "all", "one", "one", "streamed", "f64", "step", "build", "als", "update"])
    order = rng.choice([3, 3, 4, 4, 5])
    # mode lengths over the range of the listed ones, longest first or not
    dims = sorted((_log_int(rng, 300, (1 << 22) if k < 2 else (1 << 17)) for k in range(order)), reverse=True)
    if rng.random() < 0.3:
        rng.shuffle(dims)
    dims = [max(d, 2) for d in dims]
    cells = 1.0
    for d in dims:
        cells *= d
    dist = rng.choice(["uniform", "zipf:1.1", "zipf:1.2"])
    rank = rng.choice([8, 16, 16, 32, 32, 32, 64, 64, 128])
    dtype = rng.choice(["f32", "f32", "f32", "bf16", "f16"])
    most = {"all": 100e6, "one": 150e6, "streamed": 40e6, "f64": 20e6, "step": 50e6, "build": 100e6, "als": 20e6,
            "update": 1.0}[kind]
    # few enough nonzeros for distinct skewed coordinates to be found quickly
    most = max(20_000.0, min(most, cells / 200.0, most * 32.0 / max(rank, 32)))
    nnz = _log_int(rng, 20_000, most)
    more = {}
    if kind == "f64":
        rank, dtype = min(rank, 64), "f64"
    if kind in ("als", "build", "update"):
        dtype = "f32"
    if kind == "one":
        more["mode"] = rng.randrange(order)
    if kind == "als":
        rank = min(rank, 64)
        more["iters"] = rng.choice([1, 2, 3])
    if kind == "update":
        order = 3
        dims = [_log_int(rng, 300, 1 << 20) for _ in range(3)]
        rank, nnz, dist = rng.choice([5, 8, 10, 16, 20, 32, 50, 64]), 0, "uniform"
        more["mode"] = rng.randrange(3)
    if kind == "streamed":
        more["cap"] = 1 << rng.choice([20, 21, 22, 23])
    c = _case("", kind, dims, dist, nnz, rank, dtype, **more)
    del c["name"]
    return c


def _dims(case):
    return tuple(int(d) for d in case["dims"].split("x"))


def _draw_mode(n, dim, dist, tables, gen):
    if dist == "uniform":
        return torch.randint(0, dim, (n,), generator=gen, device="cuda", dtype=torch.int32)
    cdf, labels = tables
    out = torch.empty(n, dtype=torch.int32, device="cuda")
    for a in range(0, n, 1 << 26):
        u = torch.rand(min(n - a, 1 << 26), generator=gen, device="cuda", dtype=torch.float64)
        out[a:a + u.numel()] = labels[torch.searchsorted(cdf, u).clamp_(max=dim - 1)]
    return out


def _distinct(cols, dims):
    """The columns without repeated coordinates, in lexicographic order."""
    words, bits = [torch.zeros_like(cols[0], dtype=torch.int64)], 0
    for col, d in zip(cols, dims):
        b = (d - 1).bit_length()
        if bits + b > 62:
            words.append(torch.zeros_like(words[0]))
            bits = 0
        words[-1] = words[-1] * d + col
        bits += b
    order, keep = None, None
    for w in reversed(words):  # least significant word first
        s, o = torch.sort(w if order is None else w[order], stable=True)
        order = o if order is None else order[o]
    keep = torch.zeros(order.numel(), dtype=torch.bool, device="cuda")
    keep[:1] = True
    for w in words:
        s = w[order]
        keep[1:] |= s[1:] != s[:-1]
    order = order[keep]
    return [c[order] for c in cols]


def _coordinates(case, gen):
    """``nnz`` distinct coordinates, int32 (nnz x N), in random order. The
    tables of the skewed modes are summed on the host, in a fixed order, so
    that the same seed gives the same tensor every time."""
    dims, nnz = _dims(case), case["nnz"]
    dists = case["dist"].split(",")
    dists = dists if len(dists) == len(dims) else dists[:1] * len(dims)
    tables = []
    for d, dist in zip(dims, dists):
        if dist == "uniform":
            tables.append(None)
            continue
        cdf = np.cumsum(np.arange(1, d + 1, dtype=np.float64) ** -float(dist.split(":")[1]))
        tables.append((torch.from_numpy(cdf / cdf[-1]).cuda(),
                       torch.randperm(d, generator=gen, device="cuda").to(torch.int32)))
    have, want = None, int(nnz * 1.15) + 1024
    for _ in range(64):
        fresh = [_draw_mode(want, d, dist, tab, gen) for d, dist, tab in zip(dims, dists, tables)]
        before = 0 if have is None else have[0].numel()
        have = _distinct(fresh if have is None else [torch.cat(p) for p in zip(have, fresh)], dims)
        if have[0].numel() >= nnz:
            break
        gained = (have[0].numel() - before) / want
        want = int((nnz - have[0].numel()) / max(gained, 0.01) * 1.3) + 1024
    pick = torch.randperm(have[0].numel(), generator=gen, device="cuda")[:nnz]
    return torch.stack([c[pick] for c in have], 1)


def _inputs(case, seed):
    """Coordinates, values and factors of a case, from the seed alone:
    U(0,1) factors for training steps and CP-ALS, N(0,1) ones elsewhere."""
    dt = _DTYPES[case["dtype"]]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1009 * (int(seed) + 1))
    coords = _coordinates(case, gen)
    vals = torch.rand(case["nnz"], generator=gen, device="cuda")
    draw_f = torch.rand if case["kind"] in ("step", "als") else torch.randn
    facs = [draw_f((d, case["rank"]), generator=gen, device="cuda").to(dt) for d in _dims(case)]
    return coords, vals.double() if dt == torch.float64 else vals, facs


def _update_inputs(case, seed):
    """Factors whose Grams enter an update, and the MTTKRP it starts from."""
    dims, R = _dims(case), case["rank"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(977 * (int(seed) + 1))
    facs = [torch.randn((d, R), generator=gen, device="cuda") for d in dims]
    M = torch.randn((dims[case["mode"]], R), generator=gen, device="cuda")
    return facs, M


def prepare(case, seed):
    kind, dims, R = case["kind"], _dims(case), case["rank"]
    if kind == "update":
        facs, M = _update_inputs(case, seed)
        grams = []
        for f in facs:
            G = torch.empty((R, R), dtype=torch.float64, device="cuda")
            blco.blco_gram(f, blco.BLCO_F32, f.shape[0], R, G)
            grams.append(G)
        return {"case": case, "grams": grams, "M": M}
    coords, vals, facs = _inputs(case, seed)
    if kind == "build":
        return {"case": case, "coords": coords, "vals": vals}
    opts = {"force_stream": True, "max_nnz_per_block": case["cap"]} if kind == "streamed" else {}
    t = blco.Tensor.build(coords, vals, dims, **opts)
    state = {"case": case, "tensor": t, "factors": facs}
    if kind == "step":
        state["target"] = t.values()
        state["factors"] = [f.requires_grad_(True) for f in facs]
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "update":
        R, mode, M = case["rank"], case["mode"], state["M"]
        A = torch.empty_like(M)
        lam = torch.empty(R, dtype=torch.float64, device="cuda")
        G = torch.empty((R, R), dtype=torch.float64, device="cuda")
        info = torch.empty(1, dtype=torch.int32, device="cuda")
        blco.blco_cpals_update(state["grams"], 3, mode, R, M, M.shape[0], A, lam, G, info)
        return {"A": A, "lambda": lam, "gram": G, "info": info}
    if kind == "build":
        t = blco.Tensor.build(state["coords"], state["vals"], _dims(case))
        keys = torch.empty(case["nnz"], dtype=torch.int64, device="cuda")
        blco.blco_keys(t.handle, keys)
        vals = t.values()
        t.destroy()
        return {"keys": keys, "values": vals}
    t, facs = state["tensor"], state["factors"]
    if kind in ("all", "streamed"):
        return t.mttkrp_all(facs)
    if kind == "one":
        return t.mttkrp(case["mode"], facs)
    if kind == "f64":
        return [t.mttkrp_f64(n, facs) for n in range(t.order)]
    if kind == "step":
        xhat = blco.SparseCP.apply(t, *facs)
        grads = torch.autograd.grad(xhat, facs, xhat.detach() - state["target"])
        return {"model": xhat.detach(), "grads": list(grads)}
    if kind == "als":
        A, lam, fits = blco.cp_als(t, [f.clone() for f in facs], case["iters"])
        return {"factors": A, "lambda": lam, "fits": fits}
    raise ValueError(kind)


def work(case):
    """Bytes: the store (8-byte keys, the values), factors and outputs, each
    once. Flops: per nonzero, mode and rank element N - 1 products and a sum."""
    dims, R, nnz, kind = _dims(case), case["rank"], case["nnz"], case["kind"]
    N = len(dims)
    rows = float(sum(dims))
    fb = {"f32": 4, "bf16": 2, "f16": 2, "f64": 8}[case["dtype"]]
    if kind == "update":
        I = dims[case["mode"]]
        return {"bytes": 2.0 * 4 * I * R + 8.0 * 4 * R * R, "flops": 2.0 * I * R * R + I * R * (R + 1.0)}
    if kind == "build":  # coordinates and values in, keys, values and positions out
        return {"bytes": nnz * (4.0 * N + 4 + 12 + 4), "flops": 0}
    vb = 8 if kind == "f64" else 4
    ob = 8 if kind == "f64" else 4
    if kind == "one":
        I = dims[case["mode"]]
        return {"bytes": nnz * (8.0 + vb) + (rows - I) * R * fb + I * R * ob, "flops": float(nnz) * R * N}
    if kind == "f64":  # N calls, each over the store
        return {"bytes": N * (nnz * (8.0 + vb) + rows * R * 8), "flops": float(nnz) * R * N * N}
    if kind == "step":  # keys, target and model values, factors and gradients
        return {"bytes": nnz * (8.0 + 4 + 4) + rows * R * (fb + fb), "flops": float(nnz) * R * (N + N * N)}
    if kind == "als":
        it = case["iters"]
        return {"bytes": it * N * (12.0 * nnz + rows * R * 4) + it * rows * R * 8,
                "flops": it * (float(nnz) * R * N * N + 3.0 * rows * R * R)}
    return {"bytes": nnz * 12.0 + rows * R * (fb + 4), "flops": float(nnz) * R * N * N}


# ------------------------------------------------------------------ 64 bits
def _mttkrp(coords, vals, facs, mode):
    """Mode-`mode` MTTKRP in float64, a part of the nonzeros at a time."""
    R = facs[0].shape[1]
    out = torch.zeros((facs[mode].shape[0], R), dtype=torch.float64, device=facs[0].device)
    step = max(1, (1 << 28) // R)
    for a in range(0, coords.shape[0], step):
        c = coords[a:a + step].long()
        p = vals[a:a + step].double().unsqueeze(1).expand(-1, R).clone()
        for k, f in enumerate(facs):
            if k != mode:
                p *= f[c[:, k]].double()
        out.index_add_(0, c[:, mode], p)
    return out


def _model(coords, facs):
    xs = []
    step = max(1, (1 << 28) // facs[0].shape[1])
    for a in range(0, coords.shape[0], step):
        c = coords[a:a + step].long()
        p = facs[0][c[:, 0]].double()
        for k in range(1, len(facs)):
            p *= facs[k][c[:, k]].double()
        xs.append(p.sum(1))
    return torch.cat(xs)


def _alto_order(coords, dims):
    """Stable order of the nonzeros by their linear index: level by level, one
    bit of every mode that still has bits, lower modes at lower positions."""
    bits = [max(0, (d - 1).bit_length()) for d in dims]
    words, pos = [torch.zeros(coords.shape[0], dtype=torch.int64, device=coords.device)], 0
    for level in range(max(bits)):
        for n, b in enumerate(bits):
            if level < b:
                if pos == 60:
                    words.append(torch.zeros_like(words[0]))
                    pos = 0
                words[-1] |= ((coords[:, n].long() >> level) & 1) << pos
                pos += 1
    order = torch.arange(coords.shape[0], device=coords.device)
    for w in words:  # least significant word first
        order = order[torch.sort(w[order], stable=True)[1]]
    return order


def _update(facs, M, mode):
    V = torch.ones((M.shape[1], M.shape[1]), dtype=torch.float64, device=M.device)
    for k, f in enumerate(facs):
        if k != mode:
            V *= f.double().T @ f.double()
    A = torch.linalg.solve(V, M.double().T).T
    lam = A.norm(dim=0)
    return A / lam, lam


def exact(case, seed):
    kind, dims = case["kind"], _dims(case)
    if kind == "build":
        return None
    with torch.no_grad():
        if kind == "update":
            facs, M = _update_inputs(case, seed)
            A, lam = _update(facs, M, case["mode"])
            return {"A": A, "lambda": lam, "gram": A.T @ A, "info": None}
        coords, vals, facs = _inputs(case, seed)
        if kind in ("all", "streamed", "f64"):
            return [_mttkrp(coords, vals, facs, n) for n in range(len(dims))]
        if kind == "one":
            return _mttkrp(coords, vals, facs, case["mode"])
        if kind == "step":
            order = _alto_order(coords, dims)
            coords, vals = coords[order], vals[order]
            x = _model(coords, facs)
            return {"model": x, "grads": [_mttkrp(coords, x - vals, facs, n) for n in range(len(dims))]}
        if kind == "als":
            A = [f.double() for f in facs]
            normx = vals.double().norm()
            fits, lam = [], None
            for _ in range(case["iters"]):
                for n in range(len(dims)):
                    M = _mttkrp(coords, vals, A, n)
                    A[n], lam = _update(A, M, n)
                V = torch.ones((lam.numel(), lam.numel()), dtype=torch.float64, device=lam.device)
                for f in A:
                    V *= f.T @ f
                r2 = normx ** 2 + lam @ V @ lam - 2 * (lam * (M * A[-1]).sum(0)).sum()
                fits.append(float(1 - r2.clamp(min=0).sqrt() / normx))
            return {"factors": A, "lambda": lam, "fits": fits}
    return None
