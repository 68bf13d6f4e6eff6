"""GPU parity of the GraphSAGE variant (mean aggregator, sampled neighbours,
mini-batches, per-worker Adam, parameters averaged per epoch) through the C-ABI
against the fp64 checker on the same seeded inputs.

Bars: batch membership and sampled neighbour sets identical (compared as sets:
every draw is a set of unique keys); embeddings, logits, gradients within
1e-4 * max|reference|; epoch loss within 1e-3 relative at every epoch."""
import copy

import numpy as np
import pytest
import torch

from gen import configs
from oracle import oracle, sage
from paper_2012_04930_b200 import gcnsa

from parity_helpers import TOL, ambiguous_units, close

pytestmark = pytest.mark.gpu


def _setup(w, hidden, fanout, batch, lr, gemm_mode):
    dims = [w.dims[0], hidden, w.dims[-1]]
    ws, wn, bs = configs.sage_weights(dims, w.seed + 77)
    env = gcnsa.make_env(0)
    parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                        w.part_mode, w.user_part, w.loss_on_halo)
    model = gcnsa.Sage(env, parts, dims, ws, wn, bs, fanout=fanout, batch=batch, lr=lr, seed=w.seed, gemm_mode=gemm_mode)
    _, rparts = oracle.build_partitions(w.rowptr, w.col, w.m, w.overlap_ppm, w.seed, w.part_mode, w.user_part)
    params = [ws[0].astype(np.float64), wn[0].astype(np.float64), bs[0].astype(np.float64),
              ws[1].astype(np.float64), wn[1].astype(np.float64), bs[1].astype(np.float64)]
    xs = [w.x[pt.members].astype(np.float64) for pt in rparts]
    ys = [w.y[pt.members] for pt in rparts]
    trs = [oracle.train_set(pt, w.train_mask[pt.members], w.loss_on_halo) for pt in rparts]
    return env, parts, model, rparts, params, xs, ys, trs


def _relu_decisions(fw, e):
    """ReLU on / off per hidden unit for the checker's backward pass: its own sign of z, except where |z| is
    within fp32 resolution of zero (parity_helpers.ambiguous_units, from the checker's values alone); there the
    kernel's decision is taken, after checking that its value is equally tiny.  Away from zero both must agree."""
    z = fw["z1"]
    amb = ambiguous_units([z])[0]
    on = z > 0.0
    seen = np.zeros(z.shape[0], bool)
    for j, v in enumerate(e["vertices"]):
        if v < 0:
            continue
        k = fw["where"][int(v)]
        h = e["hidden"][j]
        assert np.all(np.abs(h[amb[k]]) < 2e-5 * np.abs(z).max())
        assert np.array_equal((h > 0)[~amb[k]], on[k][~amb[k]]), "ReLU decisions differ away from zero"
        if not seen[k]:
            on[k] = np.where(amb[k], h > 0, on[k])
            seen[k] = True
    assert amb.sum() <= 1e-3 * z.size + 2
    return on


def _gpu_params(model, base):
    return [model.get(base + k, l) for l in (0, 1) for k in (0, 1, 2)]


def _check_batch(model, pt, x, y, params, tg, seed, epoch, fanout, p, b):
    """One batch on both sides: membership, both layers' sample sets, embeddings, logits, loss, logit gradient and
    the six parameter gradients."""
    fw = sage.batch_forward(pt, x, params, tg, y, seed, epoch, fanout)
    model.run_batch(p, epoch, b, apply=False)
    e = model.batch_export()
    grads, g = sage.batch_backward(fw, x, params, relu_on=_relu_decisions(fw, e))
    nb, r1, r2 = tg.size, fanout[0], fanout[1]
    assert e["nb"] == nb and np.array_equal(e["vertices"][:nb], tg), "batch membership and order"
    # the output layer's samples: slots nb + i r2 + s
    slots = e["vertices"][nb:].reshape(nb, r2)
    for i in range(nb):
        c = int(e["count2"][i])
        assert c == fw["c2"][i] and sorted(slots[i, :c]) == list(fw["s2"][i, :c]) and np.all(slots[i, c:] == -1)
    # the hidden layer's samples and embeddings, row by row against the checker's record of that vertex
    for j, v in enumerate(e["vertices"]):
        if v < 0:
            assert e["count1"][j] == 0
            continue
        k = fw["where"][int(v)]
        c = int(e["count1"][j])
        assert c == fw["c1"][k] and sorted(e["samples1"][j, :c]) == list(fw["s1"][k, :c])
    valid = e["vertices"] >= 0
    rows = np.array([fw["where"][int(v)] for v in e["vertices"][valid]])
    close(e["hidden"][valid], fw["h1"][rows], what=f"p{p} b{b} hidden layer")
    close(e["logits"], fw["logits"], what=f"p{p} b{b} logits")
    close(e["dlogits"], g, what=f"p{p} b{b} dlogits")
    assert abs(float(e["loss"][0]) - fw["loss"]) <= 1e-5 * abs(fw["loss"])
    for got, want, nm in zip(_gpu_params(model, gcnsa.SAGE_GRAD_W_SELF), grads,
                             ("dWs1", "dWn1", "db1", "dWs2", "dWn2", "db2")):
        close(got, want, what=f"p{p} b{b} {nm}")


@pytest.mark.parametrize("hidden,c,fanout,batch", [(1, 3, (2, 1), 7), (17, 33, (3, 4), 63), (100, 129, (4, 3), 64),
                                                   (16, 256, (3, 2), 65), (16, 257, (3, 2), 64), (256, 41, (2, 5), 33),
                                                   (512, 5, (2, 3), 40), (600, 41, (2, 3), 40), (24, 5, (3, 0), 32)])
def test_output_layer_of_every_width(hidden, c, fanout, batch, tiny_wl):
    """The output layer of small batches runs in one kernel up to 256 classes and 32 768 weights, two vertices to a block (odd
    batches), and launch by launch beyond: a full and the ragged last batch against the checker."""
    w = copy.copy(tiny_wl)
    w.dims = [w.dims[0], hidden, c]
    w.y = np.random.default_rng(c).integers(0, c, len(w.y)).astype(np.int32)
    env, parts, model, rparts, params, xs, ys, trs = _setup(w, hidden, fanout, batch, 0.01, gcnsa.GEMM_TF32X3)
    want = sage.batches(rparts[0], trs[0], w.seed, 0, batch)
    for b in (0, len(want) - 1):
        _check_batch(model, rparts[0], xs[0], ys[0], params, want[b], w.seed, 0, fanout, 0, b)
    assert gcnsa.tc_status() == 0
    model.close(); parts.close()


@pytest.mark.parametrize("hidden,c,batch,one_kernel", [
    (128, 41, 256, 1), (128, 41, 1023, 1), (128, 47, 1024, 0), (256, 256, 64, 0), (64, 256, 175, 1), (64, 256, 176, 0), (256, 64, 384, 1),
    (256, 64, 385, 0), (512, 16, 4096, 1), (32, 17, 2647, 1), (32, 17, 2648, 0)])
def test_output_layers_that_are_work_stay_on_the_tensor_cores(hidden, c, batch, one_kernel, tiny_wl):
    """A batch has three products on the tensor cores where the output layer runs in one kernel, and five otherwise."""
    w = copy.copy(tiny_wl)
    w.dims = [w.dims[0], hidden, c]
    w.y = np.random.default_rng(c).integers(0, c, len(w.y)).astype(np.int32)
    env, parts, model, *_ = _setup(w, hidden, (2, 2), batch, 0.01, gcnsa.GEMM_TF32X3)
    tc0, fb0 = gcnsa.gemm_path_counts()
    model.run_batch(0, 0, 0)
    tc1, fb1 = gcnsa.gemm_path_counts()
    assert (tc1 - tc0, fb1 - fb0) == (3 if one_kernel else 5, 0) and gcnsa.tc_status() == 0
    model.close(); parts.close()


@pytest.mark.parametrize("gemm_mode", [gcnsa.GEMM_FP32, gcnsa.GEMM_TF32X3])
@pytest.mark.parametrize("name,hidden,fanout,batch", [("tiny", 16, (5, 3), 64), ("tiny", 16, (25, 10), 256),
                                                      ("small", 64, (25, 10), 256), ("small", 32, (2, 40), 100)])
def test_one_batch_matches_checker(name, hidden, fanout, batch, gemm_mode, tiny_wl, small_wl):
    w = tiny_wl if name == "tiny" else small_wl
    env, parts, model, rparts, params, xs, ys, trs = _setup(w, hidden, fanout, batch, 0.01, gemm_mode)
    tc0, fb0 = gcnsa.gemm_path_counts()
    for p, epoch in ((0, 0), (w.m - 1, 3)):
        pt = rparts[p]
        want_batches = sage.batches(pt, trs[p], w.seed, epoch, batch)
        assert model.n_batches(p) == len(want_batches)
        for b in sorted({0, len(want_batches) - 1}):         # a full batch and the ragged last one
            _check_batch(model, pt, xs[p], ys[p], params, want_batches[b], w.seed, epoch, fanout, p, b)
    if gemm_mode == gcnsa.GEMM_TF32X3:
        tc1, fb1 = gcnsa.gemm_path_counts()
        assert tc1 > tc0 and fb1 == fb0 and gcnsa.tc_status() == 0
    # one Adam step of worker 0 on the last computed gradient of a fresh batch
    pt = rparts[0]
    tg = sage.batches(pt, trs[0], w.seed, 0, batch)[0]
    fw = sage.batch_forward(pt, xs[0], params, tg, ys[0], w.seed, 0, fanout)
    model.run_batch(0, 0, 0, apply=False)
    grads, _ = sage.batch_backward(fw, xs[0], params, relu_on=_relu_decisions(fw, model.batch_export()))
    g_own = [a.astype(np.float64) for a in _gpu_params(model, gcnsa.SAGE_GRAD_W_SELF)]
    model.run_batch(0, 0, 0, apply=True)
    ref = oracle.Adam(params, 0.01).step(params, grads)
    own = oracle.Adam(params, 0.01).step(params, g_own)
    for got, r, o, gr in zip(_gpu_params(model, gcnsa.SAGE_WORK_W_SELF), ref, own, grads):
        scale = max(np.abs(r).max(), 0.01)
        assert np.abs(got - o).max() <= 1e-5 * scale          # the kernel's step on its own gradient
        firm = np.abs(gr) >= 1e-3 * np.abs(gr).max()          # where the sign of the gradient is determined in fp32
        if firm.any():
            assert np.abs(got - r)[firm].max() <= TOL * scale
    for got, p0 in zip(_gpu_params(model, gcnsa.SAGE_W_SELF), params):
        assert np.array_equal(got, p0.astype(np.float32)), "the aggregated parameters move at the end of an epoch only"
    model.close(); parts.close()


@pytest.mark.parametrize("hidden", [64, 128])
def test_products_of_workers_side_by_side_keep_fp32_accuracy(hidden, small_wl):
    """Four workers' products are cut for several that run at once: hidden layer and its weight gradients of three batches
    against the checker in the 2-norm.  A slice has at most 16 k-blocks with one cut of at most 2^-23 per 8 k, half of that on
    average, on a sum that is half its end on average: 2^-23 per k-block, 1.9e-6, with the dropped terms 2.1e-6; 0.4e-6 for
    the rest of the batch."""
    w = small_wl
    env, parts, model, rparts, params, xs, ys, trs = _setup(w, hidden, (25, 10), 256, 0.01, gcnsa.GEMM_TF32X3)
    errs = []
    for b, tg in enumerate(sage.batches(rparts[0], trs[0], w.seed, 0, 256)[:3]):
        fw = sage.batch_forward(rparts[0], xs[0], params, tg, ys[0], w.seed, 0, (25, 10))
        model.run_batch(0, 0, b, apply=False)
        e = model.batch_export()
        grads, _ = sage.batch_backward(fw, xs[0], params, relu_on=_relu_decisions(fw, e))
        valid = e["vertices"] >= 0
        rows = np.array([fw["where"][int(v)] for v in e["vertices"][valid]])
        pairs = [(e["hidden"][valid], fw["h1"][rows])] + list(zip(_gpu_params(model, gcnsa.SAGE_GRAD_W_SELF)[:2], grads[:2]))
        errs.append([np.linalg.norm(got - want) / np.linalg.norm(want) for got, want in pairs])
    assert gcnsa.tc_status() == 0 and np.max(errs) <= 2.5e-6, errs
    model.close(); parts.close()


@pytest.mark.parametrize("name,hidden,fanout,batch,epochs,lr", [("tiny", 16, (25, 10), 256, 10, 0.003),
                                                               ("small", 64, (25, 10), 256, 5, 0.0005)])
def test_loss_curve_and_averaged_parameters_match_checker(name, hidden, fanout, batch, epochs, lr, tiny_wl, small_wl):
    w = tiny_wl if name == "tiny" else small_wl
    env, parts, model, rparts, params, xs, ys, trs = _setup(w, hidden, fanout, batch, lr, gcnsa.GEMM_TF32X3)
    opts = [oracle.Adam(params, lr) for _ in rparts]
    loss = torch.zeros(1, device="cuda")
    first = None
    for e in range(epochs):
        params, want = sage.epoch(rparts, xs, ys, trs, params, opts, w.seed, e, fanout, batch)
        model.epoch(loss.data_ptr())
        got = loss.item()
        assert abs(got - want) <= 1e-3 * abs(want), (e, got, want)
        first = want if first is None else first
    assert want < first, "training must reduce the loss"
    assert model.epochs_done == epochs and gcnsa.tc_status() == 0
    for got, ref, nm in zip(_gpu_params(model, gcnsa.SAGE_W_SELF), params, ("Ws1", "Wn1", "b1", "Ws2", "Wn2", "b2")):
        close(got, ref, tol=5e-3, what=f"{nm} after {epochs} epochs")
    model.close(); parts.close()


def test_batches_at_paper_scale_match_checker():
    """The configuration the benchmark's GraphSAGE line times (232 965 vertices, 602 -> 128 -> 41, fan-outs 25 / 10,
    batches of 256, tensor-core products): the first, a middle and the ragged last batch of two workers, in two
    different epochs, against the checker."""
    w = configs.paper_scale()
    fanout, batch = (25, 10), 256
    env, parts, model, rparts, params, xs, ys, trs = _setup(w, 128, fanout, batch, 1e-4, gcnsa.GEMM_TF32X3)
    tc0, fb0 = gcnsa.gemm_path_counts()
    for p, epoch in ((1, 0), (4, 2)):
        pt = rparts[p]
        want_batches = sage.batches(pt, trs[p], w.seed, epoch, batch)
        assert model.n_batches(p) == len(want_batches) > 100
        for b in (0, len(want_batches) // 2, len(want_batches) - 1):
            _check_batch(model, pt, xs[p], ys[p], params, want_batches[b], w.seed, epoch, fanout, p, b)
    tc1, fb1 = gcnsa.gemm_path_counts()
    assert tc1 > tc0 and fb1 == fb0 and gcnsa.tc_status() == 0
    model.close(); parts.close()


def test_recorded_batches_equal_plain_launches(small_wl):
    """batch_graph: a worker's full-size batches replay one recorded kernel sequence whose batch index and epoch
    live in device memory.  Losses, parameters and the launch counter equal those of plain launches, bit for bit,
    over three epochs (ten full batches and a ragged one per worker)."""
    w = small_wl
    dims = [w.dims[0], 64, w.dims[-1]]
    ws, wn, bs = configs.sage_weights(dims, w.seed + 77)
    results = []
    with torch.cuda.stream(torch.cuda.Stream()):      # a recording needs a stream other than the legacy default one
        for batch_graph in (0, 1):
            env = gcnsa.make_env(0)
            parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                                w.part_mode, w.user_part, w.loss_on_halo)
            model = gcnsa.Sage(env, parts, dims, ws, wn, bs, fanout=(25, 10), batch=256, lr=5e-4, seed=w.seed,
                               gemm_mode=gcnsa.GEMM_TF32X3, batch_graph=batch_graph)
            assert all(model.n_batches(p) >= 5 for p in range(w.m))
            loss = torch.zeros(1, device="cuda")
            losses, n0 = [], gcnsa.launch_count()
            for _ in range(3):
                model.epoch(loss.data_ptr())
                losses.append(loss.item())
            launches = gcnsa.launch_count() - n0
            results.append((losses, _gpu_params(model, gcnsa.SAGE_W_SELF), launches))
            assert gcnsa.tc_status() == 0
            model.close(); parts.close()
    (l0, p0, n0), (l1, p1, n1) = results
    assert l0 == l1, (l0, l1)
    for a, b in zip(p0, p1):
        assert np.array_equal(a, b)
    # the recorded sequence has one kernel more per full batch (its first, which advances the index and takes the
    # batch's vertices, where the plain sequence has a copy) and one per worker and epoch that resets the index
    assert n1 > n0


@pytest.mark.parametrize("m", [1, 8, 11])
def test_workers_side_by_side_equal_workers_one_after_another(tiny_wl, m):
    """An epoch runs up to eight workers at once; while profiling it runs them one after another.  Losses, parameters
    and the last worker's last batch are the same bit for bit (fewer, as many and more workers than lanes)."""
    w = tiny_wl
    dims = [w.dims[0], 16, w.dims[-1]]
    ws, wn, bs = configs.sage_weights(dims, w.seed + 77)
    results = []
    with torch.cuda.stream(torch.cuda.Stream()):
        for serial in (False, True):
            env = gcnsa.make_env(0)
            parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], m, w.overlap_ppm, w.seed)
            model = gcnsa.Sage(env, parts, dims, ws, wn, bs, fanout=(5, 4), batch=32, lr=5e-4, seed=w.seed)
            model.profile(serial)
            loss = torch.zeros(1, device="cuda")
            losses = []
            for _ in range(2):
                model.epoch(loss.data_ptr())
                losses.append(loss.item())
            results.append((losses, _gpu_params(model, gcnsa.SAGE_W_SELF), model.batch_export()))
            model.close(); parts.close()
    (l0, p0, b0), (l1, p1, b1) = results
    assert l0 == l1
    for a, b in zip(p0, p1):
        assert np.array_equal(a, b)
    for key in ("vertices", "samples1", "hidden", "logits", "nb"):
        assert np.array_equal(b0[key], b1[key]), key


@pytest.mark.parametrize("idle", [1, 2, 3])
def test_latest_batch_of_an_epoch_whose_last_workers_have_none(tiny_wl, idle):
    """The last `idle` of four workers have no training vertices: after an epoch the export describes the last batch of the
    last worker that has any, workers side by side as one after another (default stream)."""
    w = tiny_wl
    n = w.rowptr.size - 1
    user = (np.arange(n) * 4 // n).astype(np.int32)
    mask = ((user < 4 - idle) & (np.arange(n) % 3 > 0)).astype(np.uint8)
    dims = [w.dims[0], 16, w.dims[-1]]
    ws, wn, bs = configs.sage_weights(dims, 3)
    got = []
    for stream in (torch.cuda.default_stream(), torch.cuda.Stream()):
        with torch.cuda.stream(stream):
            env = gcnsa.make_env(0)
            parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, mask, w.dims[-1], 4, 100_000, 5, gcnsa.PART_USER, user,
                                loss_on_halo=0)
            assert [parts.info(p).n_train > 0 for p in range(4)] == [True] * (4 - idle) + [False] * idle
            model = gcnsa.Sage(env, parts, dims, ws, wn, bs, fanout=(4, 3), batch=64, seed=9)
            for _ in range(2):
                model.epoch()
            got.append(model.batch_export())
            model.run_batch(0, 0, 0)
            got.append(model.batch_export())
            got.append({"grad": model.get(gcnsa.SAGE_GRAD_W_SELF, 0)})
            assert got[-1]["grad"].any()
            model.close()
            parts.close()
    for one, other in zip(got[:3], got[3:]):
        for key in one:
            assert np.array_equal(one[key], other[key]), key


def test_partitions_with_more_training_vertices_than_the_model_has_room_for_are_refused(tiny_wl):
    w = tiny_wl
    n = w.rowptr.size - 1
    dims = [w.dims[0], 16, w.dims[-1]]
    ws, wn, bs = configs.sage_weights(dims, 3)
    env = gcnsa.make_env(0)
    few, more = (gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, (np.arange(n) % k == 0).astype(np.uint8), w.dims[-1], 2, 0, 5)
                 for k in (3, 2))
    model = gcnsa.Sage(env, few, dims, ws, wn, bs, batch=64)
    model.epoch()
    model.parts = more
    for call in (model.epoch, lambda: model.run_batch(0, 0, 0), lambda: model.n_batches(0)):
        with pytest.raises(gcnsa.GcnsaError) as ei:
            call()
        assert ei.value.code == gcnsa.ERR_ARG
    other = gcnsa.Sage(env, more, dims, ws, wn, bs, batch=64)
    other.parts = few
    other.epoch()
    torch.cuda.synchronize()
    for closing in (model, other, few, more):
        closing.close()


def test_runs_are_bitwise_reproducible_and_arguments_are_checked(tiny_wl):
    w = tiny_wl
    outs = []
    for _ in range(2):
        env, parts, model, *_ = _setup(w, 16, (4, 3), 128, 0.01, gcnsa.GEMM_TF32X3)
        for _ in range(2):
            model.epoch()
        outs.append(_gpu_params(model, gcnsa.SAGE_W_SELF))
        if len(outs) == 2:
            for bad in (lambda: model.run_batch(0, 0, 10_000), lambda: model.run_batch(9, 0, 0),
                        lambda: model.run_batch(0, -1, 0), lambda: model.get(99, 0), lambda: model.get(0, 2)):
                with pytest.raises(gcnsa.GcnsaError) as ei:
                    bad()
                assert ei.value.code == gcnsa.ERR_ARG
        model.close(); parts.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
    env = gcnsa.make_env(0)
    parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed, w.part_mode,
                        w.user_part)
    ws, wn, bs = configs.sage_weights([64, 16, 5], 1)
    for kw in (dict(batch=0), dict(fanout=(-1, 3)), dict(lr=0.0)):
        with pytest.raises(gcnsa.GcnsaError) as ei:
            gcnsa.Sage(env, parts, [64, 16, 5], ws, wn, bs, **kw)
        assert ei.value.code == gcnsa.ERR_ARG
    with pytest.raises(gcnsa.GcnsaError):
        gcnsa.Sage(env, parts, [63, 16, 5], ws, wn, bs)        # width does not match the partitions
    parts.close()
