"""What is measured: training, inference and set-up of the library, called as a user's program calls them.

A case is a dict of plain values.  ``kind`` names the call:

* ``epoch``  full-batch training: a few epochs of ``Model.epoch``, then the parameters are read back
* ``stream`` the same with the feature rows uploaded from pinned host memory in every epoch (``Model.epoch_host``)
* ``layer``  one forward and one backward pass step by step (``forward`` / ``backward`` / ``step``), gradients read back
* ``eval``   inference on the complete graph: ``Model.evaluate`` (predictions, hit count) and the logits
* ``sage``   one epoch of GraphSAGE mini-batch training (``Sage.epoch``), then the parameters are read back
* ``build``  partitioning a graph held in host memory (``Parts``) and exporting the partitions' matrices

Graphs are drawn on the GPU from the seed with the shapes of the workloads in ``gen/configs.py``: communities of
contiguous vertex ids (a share ``mu`` of the edges stays inside), degrees equal (``gamma`` 0: stochastic block model) or
power-law with tail exponent ``gamma``, or a near-regular graph without locality (``n_comm`` 0).  Features are class means
plus unit noise, labels the community modulo the number of classes with some noise.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2012_04930_b200 import gcnsa

_COMMON = dict(m=1, overlap=0.1, part="range", mask_p=0.66, agg="grad", halo_loss=True, cache_ax=False, epochs=1)


def _case(name, kind, n, nnz, f, hidden, layers, c, **kw):
    case = dict(_COMMON, name=name, kind=kind, n=n, nnz=nnz, f=f, hidden=hidden, layers=layers, c=c)
    case.update(kw)
    return case


def listed():
    return [
        # the smallest job: a 2 000-vertex block-model graph, two partitions, ten epochs; launches and latency
        _case("train-tiny", "epoch", 2000, 16000, 64, 16, 2, 5, m=2, n_comm=5, mu=0.71, gamma=0.0, mask_p=0.5, epochs=10),
        # a citation-sized graph: wide features, few edges, four partitions
        _case("train-small", "epoch", 20000, 400000, 500, 64, 2, 20, m=4, n_comm=20, mu=0.345, gamma=0.0, mask_p=0.5, epochs=10),
        # a mid-size social graph at odd sizes, vertices dealt out by hash, parameters averaged as Section 3.2 of the
        # paper states it, sampled vertices without loss
        _case("train-mid-hash", "epoch", 58241, 14300000, 301, 96, 2, 37, m=3, part="hash", n_comm=41, mu=0.9, gamma=2.1,
              agg="param", halo_loss=False, epochs=5),
        # the paper's dense dataset: 232 965 vertices, 114.6 M non-zeros, five partitions
        _case("train-paper", "epoch", 232965, 114600000, 602, 128, 2, 41, m=5, n_comm=41, mu=0.94, gamma=2.1, epochs=3),
        # the large sparse dataset: 2.45 M vertices, three layers, the first of which widens
        _case("train-large-sparse", "epoch", 2450000, 123700000, 100, 256, 3, 47, m=10, n_comm=1504, mu=0.86, gamma=2.1),
        # features that live in host memory: uploaded in every epoch, one partition ahead of the computation
        _case("train-streamed", "stream", 58241, 14300000, 602, 128, 2, 41, m=4, n_comm=41, mu=0.94, gamma=2.1),
        # a single layer of equal widths on a graph without locality (mean degree 32), stepped by the caller
        _case("layer-regular", "layer", 400000, 12800000, 256, 256, 1, 256, n_comm=0, mu=0.0, gamma=0.0),
        # validation during training of a small job: predictions and logits of every vertex
        _case("eval-small", "eval", 20000, 400000, 500, 64, 2, 20, n_comm=20, mu=0.345, gamma=0.0),
        # inference on a complete dense graph
        _case("eval-dense", "eval", 116483, 40500000, 602, 128, 2, 41, n_comm=41, mu=0.94, gamma=2.1),
        # mini-batches on the small graph: a few dozen batches per worker, the last one ragged
        _case("sage-small", "sage", 20000, 400000, 500, 128, 2, 20, m=4, n_comm=20, mu=0.345, gamma=0.0, batch=256, fan1=25, fan2=10),
        # mini-batches on a dense graph where a partition's rows no longer sit next to each other in cache
        _case("sage-dense", "sage", 116483, 40500000, 602, 128, 2, 41, m=5, n_comm=41, mu=0.94, gamma=2.1, batch=256, fan1=25, fan2=10),
        # set-up: graph in host memory to partitions on the device and their matrices back
        _case("build-dense", "build", 116483, 40500000, 301, 64, 2, 41, m=4, n_comm=41, mu=0.94, gamma=2.1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["epoch", "epoch", "epoch", "eval", "sage", "stream", "layer", "build"])
    n = int(_log(rng, 1500, 60000 if kind == "sage" else 400000))
    f = int(_log(rng, 16, min(700, max(20, 60e6 / n))))
    deg = _log(rng, 6, max(8, min(500, 30e6 / n, n / 40)))
    hidden = int(_log(rng, 8, 256))
    c = rng.randint(3, 64)
    layers = rng.choice([2, 2, 2, 3])
    shape = rng.choice(["law", "law", "block", "regular"])
    if shape == "law":
        n_comm, mu, gamma = max(2, min(int(n / _log(rng, 1000, 6000)), 1500)), round(rng.uniform(0.8, 0.95), 3), 2.1
    elif shape == "block":
        n_comm, mu, gamma = max(2, min(20, n // 400)), round(rng.uniform(0.3, 0.75), 3), 0.0
    else:
        n_comm, mu, gamma = 0, 0.0, 0.0
    extra = {}
    if kind == "sage":
        layers = 2
        extra = dict(batch=rng.choice([64, 200, 256, 512]), fan1=rng.randint(5, 25), fan2=rng.randint(3, 10))
    elif kind == "layer":
        layers = 1
        hidden = c = int(_log(rng, 16, min(602, max(17, 60e6 / n))))
        f = c
    if kind in ("epoch", "stream"):
        extra["cache_ax"] = kind == "epoch" and rng.random() < 0.12
        extra["agg"] = rng.choice(["grad", "grad", "param"])
    m = 1 if kind in ("eval", "layer") else rng.randint(2, 8)
    case = _case("", kind, n, int(n * deg) // 2 * 2, f, hidden, layers, c, m=m, n_comm=n_comm, mu=mu, gamma=gamma,
                 part=rng.choice(["range", "range", "hash"]), mask_p=rng.choice([0.3, 0.5, 0.66]),
                 overlap=rng.choice([0.0, 0.05, 0.1, 0.2]), halo_loss=rng.random() < 0.8,
                 epochs=rng.randint(2, 10) if kind == "epoch" and n < 100000 else 1, **extra)
    del case["name"]
    return case


# ----------------------------------------------------------------- inputs ---
def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h


def _graph(case, seed):
    """A simple symmetric graph with ascending rows as (rowptr int64, col int32, community) on the GPU."""
    n, nnz, n_comm = case["n"], case["nnz"], case["n_comm"]
    gen = torch.Generator(device="cuda").manual_seed(2 * seed + 1)
    want = nnz // 2
    have = torch.zeros(0, dtype=torch.int64, device="cuda")
    base = torch.arange(n, device="cuda")
    if n_comm == 0:  # union of random permutations: no locality, degrees close to the mean
        comm = base
        for _ in range(max(1, -(-nnz // (2 * n)))):
            pi = torch.randperm(n, generator=gen, device="cuda")
            have = torch.cat([have, torch.minimum(base, pi)[base != pi] * n + torch.maximum(base, pi)[base != pi]])
        have = torch.unique(have)
    else:
        rng = np.random.RandomState((seed * 7919 + 13) % (1 << 31))
        w = np.ones(n)
        if case["gamma"]:
            w = (1.0 - rng.random_sample(n)) ** (-1.0 / (case["gamma"] - 1.0))
            for _ in range(6):  # expected degrees capped at the square root of their sum
                w = np.minimum(w * (nnz / w.sum()), math.sqrt(nnz))
        bounds = np.arange(n_comm + 1, dtype=np.int64) * n // n_comm
        comm_h = np.repeat(np.arange(n_comm), np.diff(bounds))
        cw = torch.from_numpy(np.concatenate([[0.0], np.cumsum(w)])).cuda()
        comm, b = torch.from_numpy(comm_h).cuda(), torch.from_numpy(bounds).cuda()
        for _ in range(40):
            if have.numel() >= want:
                break
            draws = int((want - have.numel()) * 1.25) + 1024
            r = torch.rand((3, draws), generator=gen, dtype=torch.float64, device="cuda")
            u = (torch.searchsorted(cw, r[0] * cw[-1], right=True) - 1).clamp_(0, n - 1)
            lo, hi = cw[b[comm[u]]], cw[b[comm[u] + 1]]
            q = torch.where(r[1] < case["mu"], lo + r[2] * (hi - lo), r[2] * cw[-1])
            v = (torch.searchsorted(cw, q, right=True) - 1).clamp_(0, n - 1)
            key = (torch.minimum(u, v) * n + torch.maximum(u, v))[u != v]
            have = torch.unique(torch.cat([have, key]))
    if have.numel() > want:
        have = have[torch.randperm(have.numel(), generator=gen, device="cuda")[:want]]
    lo = have // n
    hi = have - lo * n
    key = torch.sort(torch.cat([lo * n + hi, hi * n + lo])).values
    src = key // n
    col = (key - src * n).int()
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.bincount(src, minlength=n).cumsum(0)
    return rowptr, col, comm


def _inputs(case, seed):
    """Host arrays of one graph: structure, features, labels, training mask."""
    rowptr, col, comm = _graph(case, seed)
    n, f, c = case["n"], case["f"], case["c"]
    gen = torch.Generator(device="cuda").manual_seed(2 * seed + 2)
    cls = comm % c
    x = torch.randn((n, f), generator=gen, device="cuda")
    x += 0.5 * torch.randn((c, f), generator=gen, device="cuda")[cls]
    noisy = torch.rand(n, generator=gen, device="cuda") < 0.03
    y = torch.where(noisy, torch.randint(0, c, (n,), generator=gen, device="cuda"), cls).int()
    mask = (torch.rand(n, generator=gen, device="cuda") < case["mask_p"]).to(torch.uint8)
    return {k: _pinned(v) for k, v in dict(rowptr=rowptr, col=col, x=x, y=y, mask=mask).items()}


def _parts(env, case, g, seed):
    return gcnsa.Parts(env, g["rowptr"].numpy(), g["col"].numpy(), g["x"].numpy(), g["y"].numpy(), g["mask"].numpy(),
                       case["c"], case["m"], int(case["overlap"] * 1e6) if case["m"] > 1 else 0, seed + 5,
                       part_mode=gcnsa.PART_HASH if case["part"] == "hash" else gcnsa.PART_RANGE,
                       loss_on_halo=int(case["halo_loss"]))


def _dims(case):
    return [case["f"]] + [case["hidden"]] * (case["layers"] - 1) + [case["c"]]


def _glorot(rng, fi, fo, fan_in=None):
    lim = math.sqrt(6.0 / ((fan_in or fi) + fo))
    return rng.uniform(-lim, lim, size=(fi, fo)).astype(np.float32)


_stream = None


def _own_stream():
    global _stream
    if _stream is None:  # the library records epochs on a stream other than the default one
        _stream = torch.cuda.Stream()
    return _stream


def prepare(case, seed):
    rng = np.random.RandomState((seed * 31 + 7) % (1 << 31))
    g = _inputs(case, seed)
    torch.cuda.synchronize()
    kind, dims = case["kind"], _dims(case)
    with torch.cuda.stream(_own_stream()):
        env = gcnsa.make_env()
        st = {"case": case, "env": env, "loss": torch.zeros(1, device="cuda")}
        if kind == "build":
            st["graph"], st["seed"] = {k: torch.from_numpy(v.numpy().copy()) for k, v in g.items()}, seed
            # buffers a caller can size beforehand: owned rows plus at most `overlap` of them sampled, and no more
            # stored entries than twice the graph's
            rows = int(case["n"] * (1.0 + case["overlap"])) + 2 * case["m"]
            st["out"] = {k: torch.zeros(size, dtype=t, pin_memory=True)
                         for k, size, t in (("rowptr", rows, torch.int32), ("col", 2 * case["nnz"] + rows, torch.int32),
                                            ("val", 2 * case["nnz"] + rows, torch.float32), ("members", rows, torch.int64))}
            return st
        st["parts"] = parts = _parts(env, case, g, seed)
        if kind == "sage":
            pairs = list(zip(dims[:-1], dims[1:]))
            st["model"] = gcnsa.Sage(env, parts, dims, [_glorot(rng, a, b, 2 * a) for a, b in pairs],
                                     [_glorot(rng, a, b, 2 * a) for a, b in pairs], fanout=(case["fan1"], case["fan2"]),
                                     batch=case["batch"], lr=1e-4, seed=seed + 9)
        else:
            agg = gcnsa.AGG_PARAM_AVG if case["agg"] == "param" else gcnsa.AGG_GRAD_AVG
            st["model"] = gcnsa.Model(env, parts, dims, [_glorot(rng, a, b) for a, b in zip(dims[:-1], dims[1:])], lr=0.02,
                                      agg_mode=agg, cache_ax=int(case["cache_ax"]))
        if kind == "stream":
            x = g["x"].cuda()
            st["x_host"] = [_pinned(x[torch.from_numpy(parts.members(p)).cuda()]) for p in range(case["m"])]
            st["loss_host"] = np.zeros(1, np.float32)
        if kind == "eval":
            st["mask"] = 1 - g["mask"].numpy()
            st["logits"] = torch.empty((case["n"], case["c"]), pin_memory=True)
    _own_stream().synchronize()
    return st


# -------------------------------------------------------------------- run ---
def _gcn_params(model):
    return [model.get(what, l) for l in range(model.L) for what in (gcnsa.GET_W, gcnsa.GET_B)]


def _run_build(st):
    case, lib = st["case"], gcnsa.lib()
    parts = _parts(st["env"], case, st["graph"], st["seed"])
    at = dict.fromkeys(st["out"], 0)
    for p in range(case["m"]):
        i = parts.info(p)
        got = {}
        for k, size in (("rowptr", i.n + 1), ("col", i.nnz), ("val", i.nnz), ("members", i.n)):
            got[k] = st["out"][k][at[k]:at[k] + size]
            at[k] += size
        h = gcnsa.PartHost(**{k: v.data_ptr() for k, v in got.items()})
        if lib.gcnsa_parts_export(parts.handle, p, ctypes.byref(h)):
            raise RuntimeError(lib.gcnsa_last_error())
    assignment = parts.assignment()
    parts.close()
    return [assignment, st["out"]]


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "build":
        with torch.cuda.stream(_own_stream()):
            return _run_build(st)
    model = st["model"]
    if kind == "epoch":
        for _ in range(case["epochs"]):
            model.epoch(st["loss"].data_ptr())
        return [_gcn_params(model), st["loss"]]
    if kind == "stream":
        model.epoch_host([x.data_ptr() for x in st["x_host"]], st["loss_host"])
        return [_gcn_params(model), st["loss_host"]]
    if kind == "layer":
        model.forward(0, st["loss"].data_ptr())
        model.backward(0)
        grads = [model.get(what, l) for l in range(model.L) for what in (gcnsa.GET_GRAD_W, gcnsa.GET_GRAD_B)]
        model.step()
        return [grads, st["loss"]]
    if kind == "eval":
        correct, total, pred = model.evaluate(st["parts"], 0, st["mask"])
        logits = st["logits"]
        if gcnsa.lib().gcnsa_model_get(model.handle, gcnsa.GET_ACT, model.L, logits.data_ptr(), 4 * logits.numel()):
            raise RuntimeError(gcnsa.lib().gcnsa_last_error())
        return [pred, logits, total, correct / total]
    model.epoch(st["loss"].data_ptr())
    return [[model.get(what, l) for l in (0, 1) for what in (gcnsa.SAGE_W_SELF, gcnsa.SAGE_W_NEIGH, gcnsa.SAGE_B)], st["loss"]]


# ------------------------------------------------------------- accounting ---
def _extended(case):
    """Expected rows and stored entries of A + I over all extended partitions."""
    n, m = case["n"], case["m"]
    if m == 1:
        return n, case["nnz"] + n
    grow = 1.0 + case["overlap"]
    inside = 1.0 / m if case["part"] == "hash" else case["mu"] + (1.0 - case["mu"]) / m
    rows = n * grow
    return rows, case["nnz"] * inside * grow + rows


def work(case):
    kind, dims = case["kind"], _dims(case)
    rows, nnz = _extended(case)
    f, c = case["f"], case["c"]
    params = sum(a * b + b for a, b in zip(dims[:-1], dims[1:]))
    if kind == "build":  # graph, features, labels and mask in; matrices, members and feature rows out
        return {"bytes": 8.0 * case["n"] + 4.0 * case["nnz"] + (4.0 * f + 5.0) * case["n"] + 8.0 * nnz + (4.0 * f + 12.0) * rows,
                "flops": 2.0 * nnz}
    if kind == "sage":
        b, r1, r2 = case["batch"], case["fan1"], case["fan2"]
        batches = case["mask_p"] * rows / b
        h = case["hidden"]
        gemm = b * (1 + r2) * 2 * f * h * 4.0 + b * 2 * h * c * 6.0
        gather = b * (1 + r2) * (1 + r1) * f * 1.0
        part = rows / case["m"]  # a batch draws with repetition from the rows of its partition: each row read once
        read = part * (1.0 - math.exp(-gather / (f * part))) * f
        return {"bytes": batches * (4.0 * read + 12.0 * 2 * (2 * f * h + 2 * h * c)), "flops": batches * (gemm + gather)}
    narrow = [min(a, b) for a, b in zip(dims[:-1], dims[1:])]
    dense = sum(2.0 * a * b for a, b in zip(dims[:-1], dims[1:])) * rows
    sparse = sum(2.0 * w for w in narrow) * nnz
    read = 4.0 * nnz + 4.0 * rows + (4.0 * f + 5.0) * rows + 4.0 * params
    if kind == "eval":
        return {"bytes": read + (4.0 * c + 4.0) * rows, "flops": dense + sparse}
    # backward: two dense products per layer but the first (one there), one transposed sparse product per layer (none
    # for a first layer that aggregates before it multiplies)
    back = 2.0 * dense - 2.0 * dims[0] * dims[1] * rows + sparse - (2.0 * dims[0] * nnz if dims[1] > dims[0] else 0.0)
    return {"bytes": case["epochs"] * (read + 24.0 * params), "flops": case["epochs"] * (dense + sparse + back)}


def tolerance(case):
    """About four times the difference between the default path and the same path with fp32 FMA products and stored
    matrix values (other roundings, sums in another order) after two passes."""
    kind = case["kind"]
    if kind == "build":  # structure exact, matrix values to the last bits of fp32
        return {"rel": 1e-6, "max": 1e-6, "differ": 0.0}
    if kind == "eval":  # two classes within rounding of each other may swap
        return {"rel": 2.5e-5, "max": 1e-4, "differ": 1e-4}
    if kind == "layer":  # gradients after a step on gradients that differ by rounding
        return {"rel": 1e-3, "max": 3e-2}
    if kind == "sage":
        return {"rel": 2e-4, "max": 2e-3}
    # weights after a few Adam steps: a step moves an entry by lr sign(g) at first, so entries whose gradient is
    # rounding noise go either way; more of them the smaller the gradients, i.e. in deeper models on larger graphs
    return {"rel": 4e-3, "max": 0.7} if case["n"] > 1000000 else {"rel": 1e-3, "max": 0.1}
