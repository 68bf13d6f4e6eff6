"""GPU parity of the whole path through the C-ABI: gcnsa_build_partitions,
gcnsa_forward, gcnsa_backward, gcnsa_step against the fp64 checker on the same
seeded inputs.

Bars: bit-exact partition assignment, sampled vertex sets, CSR and transposed
CSR indices; fp32 tensors within 1e-4 * max|reference| after one step; epoch
loss within 1e-3 relative at every epoch."""
import copy
import threading

import numpy as np
import pytest
import torch

from gen import configs, graphs
from oracle import oracle
from paper_2012_04930_b200 import gcnsa

from parity_helpers import TOL, close as _close, relu_decisions as _relu_decisions

pytestmark = pytest.mark.gpu


def _make(w, **kw):
    env = gcnsa.make_env(0)
    parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                        w.part_mode, w.user_part, kw.get("loss_on_halo", w.loss_on_halo))
    model = gcnsa.Model(env, parts, w.dims, w.w0, w.b0, use_bias=kw.get("use_bias", 1), lr=w.lr, beta1=w.beta1,
                        beta2=w.beta2, eps=w.eps, gemm_mode=kw.get("gemm_mode", gcnsa.GEMM_FP32),
                        factored_norm=kw.get("factored_norm", 0), loss_rows_only=0, epoch_graph=0)
    return env, parts, model


def _check_structure(parts, ref_part, ref_parts):
    assert np.array_equal(parts.assignment(), ref_part)
    for p, pt in enumerate(ref_parts):
        e = parts.export(p)
        i = parts.info(p)
        assert (i.n_owned, i.n, i.nnz, i.nts) == (pt.n_owned, pt.n, pt.nnz, pt.nts)
        assert np.array_equal(e["members"], pt.members)
        for k in ("rowptr", "col", "t_rowptr", "t_col"):
            assert np.array_equal(e[k], getattr(pt, k)), k
        assert np.abs(e["val"] - pt.val).max() <= 2e-7 * pt.val.max()
        assert np.abs(e["t_val"] - pt.t_val).max() <= 2e-7 * pt.t_val.max()


@pytest.mark.parametrize("factored_norm", [0, 1])
@pytest.mark.parametrize("gemm_mode", [gcnsa.GEMM_FP32, gcnsa.GEMM_TF32X3])
@pytest.mark.parametrize("name", ["tiny", "small", "small_seed_7", "small_seed_123457"])
def test_one_step_matches_checker(name, gemm_mode, factored_norm, tiny_wl, small_wl):
    if name.startswith("small_seed_"):       # other draws of graph, features, weights and sampling keys
        w = configs.small(seed=int(name.rsplit("_", 1)[1]))
    else:
        w = tiny_wl if name == "tiny" else small_wl
    ref = oracle.train(w, epochs=1, keep_first=True)
    env, parts, model = _make(w, gemm_mode=gemm_mode, factored_norm=factored_norm)
    _check_structure(parts, ref["part"], ref["parts"])
    recs, _, _ = ref["first"]
    L = len(w.w0)
    ws0 = [a.astype(np.float64) for a in w.w0]
    bs0 = [b.astype(np.float64) for b in w.b0]
    gw = [np.zeros_like(a) for a in ws0]
    gb = [np.zeros_like(b) for b in bs0]
    losses = torch.zeros(w.m, device="cuda")
    for p, pt in enumerate(ref["parts"]):
        model.forward(p, losses[p:p + 1].data_ptr())
        fw, _ = recs[p]
        h_gpu = [model.get(gcnsa.GET_ACT, l, rows=pt.n) for l in range(1, L + 1)]
        for l in range(1, L + 1):
            _close(h_gpu[l - 1], fw["H"][l], what=f"p{p} H{l}")
        bw = oracle.backward(pt, fw, ws0, w.y[pt.members], relu_on=_relu_decisions(fw, h_gpu[:-1]))
        _close(model.get(gcnsa.GET_DLOGITS, rows=pt.n), bw["G"][L - 1], what=f"p{p} dlogits")
        model.backward(p)
        for l in range(L):
            gw[l] += bw["dW"][l]; gb[l] += bw["db"][l]
    assert np.allclose(losses.cpu().numpy(), [r[0]["loss"] for r in recs], rtol=1e-5)
    for l in range(L):  # the gradient sum before the step
        _close(model.get(gcnsa.GET_GRAD_W, l), gw[l], what=f"dW{l}")
        _close(model.get(gcnsa.GET_GRAD_B, l), gb[l], what=f"db{l}")
    g_own = [model.get(gcnsa.GET_GRAD_W, l).astype(np.float64) for l in range(L)] + \
            [model.get(gcnsa.GET_GRAD_B, l).astype(np.float64) for l in range(L)]
    model.step()
    assert model.t == 1 and gcnsa.tc_status() == 0
    # Adam's first step moves every entry by about lr * sign(g): an entry whose gradient is below fp32
    # resolution has no determined sign.  Entries with |g| >= 1e-3 max|g| are compared with the checker's step
    # on the checker's gradient; every entry is compared with the checker's step on the kernel's own gradient.
    opt = oracle.Adam(ws0 + bs0, w.lr, w.beta1, w.beta2, w.eps)
    new = opt.step(ws0 + bs0, [g / w.m for g in gw + gb])
    own = oracle.Adam(ws0 + bs0, w.lr, w.beta1, w.beta2, w.eps).step(ws0 + bs0, [g / w.m for g in g_own])
    got = [model.get(gcnsa.GET_W, l) for l in range(L)] + [model.get(gcnsa.GET_B, l) for l in range(L)]
    for i, (a, ref, mine, g) in enumerate(zip(got, new, own, gw + gb)):
        scale = max(np.abs(ref).max(), w.lr)
        assert np.abs(a - mine).max() <= 1e-5 * scale, f"param {i}: Adam kernel on its own gradient"
        firm = np.abs(g) >= 1e-3 * np.abs(g).max()
        assert firm.mean() >= 0.9
        assert np.abs(a - ref)[firm].max() <= TOL * scale, f"param {i} after one step"
    for l in range(L):
        assert np.all(model.get(gcnsa.GET_GRAD_W, l) == 0)
        _close(model.get(gcnsa.GET_ADAM_M_W, l), opt.m[l], what=f"adam m W{l}")
        _close(model.get(gcnsa.GET_ADAM_V_W, l), opt.v[l], what=f"adam v W{l}")
    model.close(); parts.close()


@pytest.mark.parametrize("factored_norm", [0, 1])
@pytest.mark.parametrize("gemm_mode", [gcnsa.GEMM_FP32, gcnsa.GEMM_TF32X3])
@pytest.mark.parametrize("name,epochs", [("tiny", 10), ("small", 50)])
def test_loss_curve_matches_checker(name, epochs, gemm_mode, factored_norm, tiny_wl, small_wl):
    w = tiny_wl if name == "tiny" else small_wl
    ref = oracle.train(w, epochs=epochs)
    env, parts, model = _make(w, gemm_mode=gemm_mode, factored_norm=factored_norm)
    loss = torch.zeros(1, device="cuda")
    got = []
    for _ in range(epochs):
        model.epoch(loss.data_ptr())
        got.append(loss.item())
    got, want = np.array(got), np.array(ref["losses"])
    assert np.abs(got - want).max() <= 1e-3 * np.abs(want).max(), (got, want)
    assert np.all(np.abs(got - want) <= 1e-3 * np.abs(want) + 1e-6)
    model.close(); parts.close()


def test_three_layers_with_a_widening_layer_and_options():
    """Deeper variant: 100 -> 256 -> 256 -> 47 runs the first layer as
    (A_hat H) W and the others as A_hat (H W); also without bias, with the
    loss restricted to owned vertices, and with the normalization factored out
    of the sparse products."""
    w = configs.large_sparse(scale=0.004)
    for use_bias, loh, mode, fact in ((1, 1, gcnsa.GEMM_FP32, 0), (0, 0, gcnsa.GEMM_TF32X3, 1), (1, 1, gcnsa.GEMM_TF32X3, 1)):
        w.loss_on_halo = loh
        if not use_bias:
            w.b0 = [np.zeros_like(b) for b in w.b0]
        env, parts, model = _make(w, use_bias=use_bias, loss_on_halo=loh, gemm_mode=mode, factored_norm=fact)
        part, rparts = oracle.build_partitions(w.rowptr, w.col, w.m, w.overlap_ppm, w.seed, w.part_mode, w.user_part)
        _check_structure(parts, part, rparts)
        ws = [a.astype(np.float64) for a in w.w0]
        bs = [b.astype(np.float64) for b in w.b0]
        gw = [np.zeros_like(a) for a in ws]
        gb = [np.zeros_like(b) for b in bs]
        for p, pt in enumerate(rparts):
            fw = oracle.forward(pt, w.x[pt.members], ws, bs if use_bias else None, w.y[pt.members],
                                w.train_mask[pt.members], loh)
            model.forward(p)
            h_gpu = [model.get(gcnsa.GET_ACT, l, rows=pt.n) for l in range(1, 4)]
            for l in range(1, 4):
                _close(h_gpu[l - 1], fw["H"][l], what=f"p{p} H{l}")
            bw = oracle.backward(pt, fw, ws, w.y[pt.members], relu_on=_relu_decisions(fw, h_gpu[:-1]))
            model.backward(p)
            for l in range(3):
                gw[l] += bw["dW"][l]; gb[l] += bw["db"][l]
        for l in range(3):
            _close(model.get(gcnsa.GET_GRAD_W, l), gw[l], what=f"dW{l}")
            if use_bias:
                _close(model.get(gcnsa.GET_GRAD_B, l), gb[l], what=f"db{l}")
            else:
                assert np.all(model.get(gcnsa.GET_GRAD_B, l) == 0)
        model.close(); parts.close()


def test_runs_are_bitwise_reproducible(small_wl):
    outs = []
    for _ in range(2):
        env, parts, model = _make(small_wl)
        for _ in range(3):
            model.epoch()
        outs.append([model.get(gcnsa.GET_W, l) for l in range(2)])
        model.close(); parts.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


def test_call_order_errors_and_checkpoint(tiny_wl):
    w = tiny_wl
    env, parts, model = _make(w)
    with pytest.raises(gcnsa.GcnsaError) as ei:
        model.backward(0)                      # no forward yet
    assert ei.value.code == gcnsa.ERR_ORDER
    with pytest.raises(gcnsa.GcnsaError) as ei:
        model.step()                           # nothing accumulated
    assert ei.value.code == gcnsa.ERR_ORDER
    model.forward(0)
    with pytest.raises(gcnsa.GcnsaError) as ei:
        model.backward(1)                      # forward was on another partition
    assert ei.value.code == gcnsa.ERR_ORDER
    with pytest.raises(gcnsa.GcnsaError) as ei:
        model.forward(5)
    assert ei.value.code == gcnsa.ERR_ARG
    model.backward(0)
    with pytest.raises(gcnsa.GcnsaError):
        model.step()                           # only one of two partitions
    model.forward(1); model.backward(1); model.step()
    # checkpoint: 2 epochs, save, 2 more  ==  restore into a fresh model, 2 more
    model.epoch()
    state = {(what, l): model.get(what, l) for what in range(8) for l in range(2)}
    t = model.t
    model.epoch(); model.epoch()
    want = [model.get(gcnsa.GET_W, l) for l in range(2)]
    env2, parts2, model2 = _make(w)
    for (what, l), v in state.items():
        model2.set(what, l, v)
    model2.t = t
    model2.epoch(); model2.epoch()
    for l in range(2):
        assert np.array_equal(model2.get(gcnsa.GET_W, l), want[l])
    for m_, p_ in ((model, parts), (model2, parts2)):
        m_.close(); p_.close()


def test_epoch_from_host_buffers_matches_resident_epoch(small_wl):
    w = small_wl
    env, parts, model = _make(w)
    env2, parts2, model2 = _make(w)
    xs = [torch.from_numpy(np.ascontiguousarray(w.x[parts.members(p)])).pin_memory() for p in range(w.m)]
    loss_h = np.zeros(1, np.float32)
    loss_d = torch.zeros(1, device="cuda")
    for _ in range(3):
        model.epoch_host([x.data_ptr() for x in xs], loss_h)
        model2.epoch(loss_d.data_ptr())
        assert loss_h[0] == loss_d.item()
    for l in range(2):
        assert np.array_equal(model.get(gcnsa.GET_W, l), model2.get(gcnsa.GET_W, l))
    for m_, p_ in ((model, parts), (model2, parts2)):
        m_.close(); p_.close()


def test_single_partition_and_zero_overlap(tiny_wl):
    """M = 1 (no sampling at all) and O = 0 (isolated partitions) are the
    method's degenerate cases."""
    import copy
    for m, o_ppm, mode in ((1, 100_000, configs.PART_RANGE), (3, 0, configs.PART_HASH)):
        w = copy.copy(tiny_wl)
        w.m, w.overlap_ppm, w.part_mode, w.user_part, w.epochs = m, o_ppm, mode, None, 2
        ref = oracle.train(w)
        env, parts, model = _make(w)
        assert all(parts.info(p).n_halo == 0 for p in range(m))
        loss = torch.zeros(1, device="cuda")
        for e in range(2):
            model.epoch(loss.data_ptr())
            assert abs(loss.item() - ref["losses"][e]) <= 1e-3 * ref["losses"][e]
        for l in range(2):
            _close(model.get(gcnsa.GET_W, l), ref["ws"][l], tol=2e-4, what=f"W{l}")
        model.close(); parts.close()


def test_profile_counters(small_wl):
    env, parts, model = _make(small_wl)
    model.profile(True)
    before = gcnsa.launch_count()
    model.epoch()
    pr = model.profile_read()
    assert pr["spmm"]["launches"] == 4 * small_wl.m and pr["spmm"]["ms"] > 0
    assert pr["gemm"]["launches"] >= 5 * small_wl.m
    assert sum(v["launches"] for v in pr.values()) == gcnsa.launch_count() - before
    nnz = sum(parts.info(p).nnz for p in range(small_wl.m))
    # the last layer's transposed product skips the columns that carry no loss, hence "<="
    assert 2.0 * nnz * (64 + 64 + 20) < pr["spmm"]["flops"] <= 2.0 * nnz * (64 + 64 + 20 + 20)
    model.close(); parts.close()


@pytest.mark.parametrize("name,epochs", [("tiny", 10), ("small", 20)])
def test_parameter_averaging_mode_matches_checker(name, epochs, tiny_wl, small_wl):
    """Section 3.2 as written: every partition takes its own Adam step (own
    moments) from the aggregated parameters; the parameters are averaged."""
    w = tiny_wl if name == "tiny" else small_wl
    env = gcnsa.make_env(0)
    parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                        w.part_mode, w.user_part, w.loss_on_halo)
    model = gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr, beta1=w.beta1, beta2=w.beta2, eps=w.eps,
                        gemm_mode=gcnsa.GEMM_TF32X3, agg_mode=gcnsa.AGG_PARAM_AVG, factored_norm=1, loss_rows_only=0,
                        epoch_graph=0)
    _, rparts = oracle.build_partitions(w.rowptr, w.col, w.m, w.overlap_ppm, w.seed, w.part_mode, w.user_part)
    xs = [w.x[pt.members].astype(np.float64) for pt in rparts]
    ys = [w.y[pt.members] for pt in rparts]
    mks = [w.train_mask[pt.members] for pt in rparts]
    ws = [a.astype(np.float64) for a in w.w0]
    bs = [b.astype(np.float64) for b in w.b0]
    opts = [oracle.Adam(ws + bs, w.lr, w.beta1, w.beta2, w.eps) for _ in rparts]
    loss = torch.zeros(1, device="cuda")
    L = len(ws)
    for e in range(epochs):
        ws, bs, want = oracle.epoch_param_avg(rparts, xs, ys, mks, ws, bs, opts, w.loss_on_halo)
        model.epoch(loss.data_ptr())
        assert abs(loss.item() - want) <= 1e-3 * abs(want), (e, loss.item(), want)
        if e == 0:
            # the first step moves each entry by about lr * sign(g_p) per partition: compare where every
            # partition's gradient sign is determined, i.e. away from |first moment| ~ 0
            for l in range(L):
                got = model.get(gcnsa.GET_W, l)
                firm = np.ones(got.shape, bool)
                for o in opts:
                    firm &= np.abs(o.m[l]) >= 1e-3 * np.abs(o.m[l]).max()
                assert firm.mean() > 0.9
                assert np.abs(got - ws[l])[firm].max() <= 1e-4 * np.abs(ws[l]).max()
            for p, o in enumerate(opts):      # every partition keeps its own moments
                model.select_partition(p)
                for l in range(L):
                    _close(model.get(gcnsa.GET_ADAM_M_W, l), o.m[l], what=f"m p{p} W{l}")
                    _close(model.get(gcnsa.GET_ADAM_V_W, l), o.v[l], what=f"v p{p} W{l}")
    assert model.t == epochs and gcnsa.tc_status() == 0
    for l in range(L):
        _close(model.get(gcnsa.GET_W, l), ws[l], tol=2e-3, what=f"W{l} after {epochs} epochs")
    model.close(); parts.close()


def test_full_graph_evaluation_matches_checker(small_wl):
    """Micro-F1 on the complete graph (Section 2.2): train on the extended
    partitions, copy the parameters into a model built on the un-partitioned
    graph, predict, count.  Predictions are compared with the checker's argmax
    on the same parameters; rows whose two best logits are closer than fp32
    resolution may go either way."""
    w = small_wl
    env, parts, model = _make(w, gemm_mode=gcnsa.GEMM_TF32X3)
    for _ in range(15):
        model.epoch()
    full = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], 1, 0, w.seed, gcnsa.PART_RANGE)
    # the evaluating model uses the options bench.py trains with: evaluation still has to compute every row
    ev = gcnsa.Model(env, full, w.dims, w.w0, w.b0, **gcnsa.MEASURED)
    ev.copy_params_from(model)
    test_mask = (1 - w.train_mask).astype(np.uint8)
    correct, total, pred = ev.evaluate(full, 0, test_mask)
    ws = [model.get(gcnsa.GET_W, l).astype(np.float64) for l in range(2)]
    bs = [model.get(gcnsa.GET_B, l).astype(np.float64) for l in range(2)]
    _, (pt,) = oracle.build_partitions(w.rowptr, w.col, 1, 0, w.seed)
    want_pred, logits = oracle.predict(pt, w.x.astype(np.float64), ws, bs)
    top2 = np.sort(logits, axis=1)[:, -2:]
    firm = (top2[:, 1] - top2[:, 0]) > 1e-4 * np.abs(logits).max()
    assert firm.mean() > 0.99
    assert np.array_equal(pred[firm], want_pred[firm])
    f1, tp, fp, fn = oracle.micro_f1(want_pred, w.y, test_mask, w.dims[-1])
    assert total == int(test_mask.sum()) == tp + fn
    assert abs(correct - tp) <= int((~firm & test_mask.astype(bool)).sum())
    assert correct / total > 0.8          # the synthetic classes are learnable: training worked
    # no mask = every vertex; evaluation leaves the training state alone
    c_all, t_all, _ = ev.evaluate(full, 0)
    assert t_all == w.n and c_all >= correct
    with pytest.raises(gcnsa.GcnsaError):   # a model built for smaller partitions cannot take the full graph
        model.evaluate(full, 0)
    model.epoch()
    for m_, p_ in ((ev, full), (model, parts)):
        m_.close(); p_.close()


def test_loss_rows_only_gives_the_same_training(small_wl):
    """With loss_rows_only the last layer is computed on the rows that carry
    loss only; training (losses, parameters) must be bit-identical, and an
    evaluation in between still sees every row."""
    w = small_wl
    env = gcnsa.make_env(0)
    parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                        w.part_mode, w.user_part, w.loss_on_halo)
    models = [gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr, gemm_mode=gcnsa.GEMM_TF32X3, loss_rows_only=k,
                          factored_norm=0, epoch_graph=0) for k in (0, 1)]
    loss = torch.zeros(2, device="cuda")
    for e in range(5):
        for k, m_ in enumerate(models):
            m_.epoch(loss[k:k + 1].data_ptr())
        assert loss[0].item() == loss[1].item()
        if e == 2:
            a = models[0].evaluate(parts, 1)
            b = models[1].evaluate(parts, 1)
            assert a[0] == b[0] and np.array_equal(a[2], b[2])
    for l in range(2):
        assert np.array_equal(models[0].get(gcnsa.GET_W, l), models[1].get(gcnsa.GET_W, l))
    for m_ in models:
        m_.close()
    parts.close()


@pytest.mark.parametrize("agg_mode", [gcnsa.AGG_GRAD_AVG, gcnsa.AGG_PARAM_AVG])
def test_recorded_epoch_equals_plain_launches(small_wl, agg_mode):
    """epoch_graph replays one recorded epoch: losses, parameters, step count
    and the launch counter must be those of plain launches, also after the
    step count is set by hand, while profiling, and with another loss pointer."""
    w = small_wl
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        env = gcnsa.make_env(0)
        assert env.stream          # a stream of its own, not the legacy default stream (NULL)
        parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                            w.part_mode, w.user_part, w.loss_on_halo)
        models = [gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr, gemm_mode=gcnsa.GEMM_TF32X3, agg_mode=agg_mode,
                              loss_rows_only=1, factored_norm=0, epoch_graph=k) for k in (0, 1)]
        loss = torch.zeros(3, device="cuda")
        counts = [0, 0]
        for e in range(8):
            if e == 3:
                for m_ in models:
                    m_.t = 40            # as after restoring a checkpoint
            if e == 5:
                models[1].profile(True)  # profiling suspends the replay
            if e == 6:
                models[1].profile(False)
            for k, m_ in enumerate(models):
                before = gcnsa.launch_count()
                m_.epoch(loss[2 if (k == 1 and e == 7) else k:].data_ptr())
                counts[k] = gcnsa.launch_count() - before
            stream.synchronize()
            got = loss[2].item() if e == 7 else loss[1].item()
            assert loss[0].item() == got, e
            assert counts[0] == counts[1] > 0
            assert models[0].t == models[1].t
        for what in (gcnsa.GET_W, gcnsa.GET_B):
            for l in range(2):
                assert np.array_equal(models[0].get(what, l), models[1].get(what, l))
        assert gcnsa.tc_status() == 0
        for m_ in models:
            m_.close()
        parts.close()


@pytest.mark.parametrize("m", [1, 2, 8, 11])
def test_partitions_of_a_recorded_epoch_run_side_by_side(tiny_wl, m):
    """A recorded epoch works on up to eight partitions at once (fewer, as many and more partitions than that): bit for
    bit the plain launches, and the activations left behind are those of the last partition."""
    w = tiny_wl
    with torch.cuda.stream(torch.cuda.Stream()):
        env = gcnsa.make_env(0)
        parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], m, w.overlap_ppm, w.seed)
        models = [gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr, epoch_graph=k) for k in (0, 1)]
        loss = torch.zeros(2, device="cuda")
        for _ in range(3):
            for k, m_ in enumerate(models):
                m_.epoch(loss[k:].data_ptr())
        rows = parts.info(m - 1).n
        for what, l in [(gcnsa.GET_W, 0), (gcnsa.GET_W, 1), (gcnsa.GET_B, 0), (gcnsa.GET_B, 1), (gcnsa.GET_ADAM_V_W, 0)]:
            assert np.array_equal(models[0].get(what, l), models[1].get(what, l))
        assert np.array_equal(models[0].get(gcnsa.GET_ACT, 1, rows), models[1].get(gcnsa.GET_ACT, 1, rows))
        assert loss[0].item() == loss[1].item()
        for m_ in models:
            m_.close()
        parts.close()


@pytest.mark.parametrize("name,dims,m,factored_norm,use_bias,loss_rows_only", [
    ("tiny", [64, 32, 24, 16, 5], 11, 1, 1, 1), ("tiny", [64, 50, 33, 7], 3, 0, 1, 0), ("tiny", [64, 100, 96, 80, 5], 11, 1, 1, 1),
    ("tiny", [64, 96, 32, 90, 24, 9], 3, 1, 1, 0), ("tiny", [30, 64, 96, 41], 4, 1, 1, 1), ("tiny", [40, 48, 20, 33, 5], 9, 0, 1, 1),
    ("tiny", [64, 70, 24, 16, 5], 5, 1, 0, 1), ("small", [500, 96, 80, 20], 4, 1, 1, 1), ("small", [500, 64, 40, 24, 20], 4, 0, 1, 0)])
def test_recorded_epochs_of_deep_models_equal_plain_launches(name, dims, m, factored_norm, use_bias, loss_rows_only, tiny_wl, small_wl):
    """In a recorded epoch loss, bias gradients and the weight gradients of all layers but the first run beside the pass, whose
    next layer writes the buffers that they read: three to five layers, narrow products and tensor-core ones alone and in turn,
    a widening layer, without bias, more partitions than are worked on at once.  Bit for bit the plain launches."""
    w = tiny_wl if name == "tiny" else small_wl
    rng = np.random.default_rng(len(dims) + dims[1] + m)
    x = np.ascontiguousarray(w.x[:, :dims[0]])
    y = rng.integers(0, dims[-1], len(w.y)).astype(np.int32)
    shapes = list(zip(dims[:-1], dims[1:]))
    w0 = [(rng.standard_normal(s) / np.sqrt(s[0])).astype(np.float32) for s in shapes]
    b0 = [(0.1 * rng.standard_normal(s[1])).astype(np.float32) for s in shapes] if use_bias else None
    with torch.cuda.stream(torch.cuda.Stream()):
        env = gcnsa.make_env(0)
        parts = gcnsa.Parts(env, w.rowptr, w.col, x, y, w.train_mask, dims[-1], m, w.overlap_ppm, w.seed)
        models = [gcnsa.Model(env, parts, dims, w0, b0, use_bias=use_bias, lr=w.lr, gemm_mode=gcnsa.GEMM_TF32X3,
                              factored_norm=factored_norm, loss_rows_only=loss_rows_only, epoch_graph=k) for k in (0, 1)]
        loss = torch.zeros(2, device="cuda")
        for e in range(4):
            for k, m_ in enumerate(models):
                m_.epoch(loss[k:].data_ptr())
            assert loss[0].item() == loss[1].item(), e
        for l in range(len(shapes)):
            for what in (gcnsa.GET_W, gcnsa.GET_ADAM_M_W, gcnsa.GET_ADAM_V_W) + ((gcnsa.GET_B, gcnsa.GET_ADAM_M_B) if use_bias else ()):
                assert np.array_equal(models[0].get(what, l), models[1].get(what, l)), (what, l)
        assert gcnsa.tc_status() == 0
        for m_ in models:
            m_.close()
        parts.close()


def test_recorded_epoch_on_the_default_stream_falls_back(tiny_wl):
    """The legacy default stream cannot be recorded: epoch_graph then runs
    plain launches with the same results."""
    w = tiny_wl
    env = gcnsa.make_env(0)
    if env.stream:
        pytest.skip("torch's current stream is not the default stream")
    parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                        w.part_mode, w.user_part, w.loss_on_halo)
    models = [gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr, **{**gcnsa.PLAIN, "epoch_graph": k}) for k in (0, 1)]
    for _ in range(3):
        for m_ in models:
            m_.epoch()
    for l in range(2):
        assert np.array_equal(models[0].get(gcnsa.GET_W, l), models[1].get(gcnsa.GET_W, l))
    for m_ in models:
        m_.close()
    parts.close()


@pytest.mark.parametrize("epoch_graph", [0, 1])
def test_cached_aggregated_features_give_the_same_training(epoch_graph, small_wl):
    """cache_ax keeps A_hat X of every partition and runs layer 1 as (A_hat X) W (Section 4.1: the same
    H^1 = sigma(A_hat X W^1), multiplied in the other order): gradients and loss curve match the checker, and a
    partition whose feature rows are rewritten gets its product recomputed."""
    w = small_wl
    epochs = 12
    ref = oracle.train(w, epochs=epochs, keep_first=True)
    stream = torch.cuda.Stream() if epoch_graph else torch.cuda.current_stream()
    with torch.cuda.stream(stream):
        env = gcnsa.make_env(0)
        parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                            w.part_mode, w.user_part, w.loss_on_halo)
        kw = dict(lr=w.lr, beta1=w.beta1, beta2=w.beta2, eps=w.eps, gemm_mode=gcnsa.GEMM_TF32X3, loss_rows_only=1,
                  factored_norm=1, epoch_graph=epoch_graph)
        cached = gcnsa.Model(env, parts, w.dims, w.w0, w.b0, cache_ax=1, **kw)
        # gradient sum of the first epoch against the checker's
        recs, _, _ = ref["first"]
        L = len(w.w0)
        ws0 = [a.astype(np.float64) for a in w.w0]
        gw = [np.zeros_like(a) for a in ws0]
        for p, pt in enumerate(ref["parts"]):
            cached.forward(p)
            fw, _ = recs[p]
            h1 = cached.get(gcnsa.GET_ACT, 1, rows=pt.n)
            _close(h1, fw["H"][1], what=f"p{p} H1 from the cached product")
            bw = oracle.backward(pt, fw, ws0, w.y[pt.members], relu_on=_relu_decisions(fw, [h1]))
            cached.backward(p)
            for l in range(L):
                gw[l] += bw["dW"][l]
        for l in range(L):
            _close(cached.get(gcnsa.GET_GRAD_W, l), gw[l], what=f"dW{l}")
        cached.step()
        # loss curve of the following epochs (the first one is spent above)
        loss = torch.zeros(1, device="cuda")
        for e in range(1, epochs):
            cached.epoch(loss.data_ptr())
            assert abs(loss.item() - ref["losses"][e]) <= 1e-3 * abs(ref["losses"][e]), (e, loss.item(), ref["losses"][e])
        # rewrite one partition's feature rows: the cached product must follow
        plain = gcnsa.Model(env, parts, w.dims, w.w0, w.b0, **kw)
        for l in range(L):
            for what in (gcnsa.GET_W, gcnsa.GET_B):
                plain.set(what, l, cached.get(what, l))
        newx = np.ascontiguousarray(w.x[parts.members(1)] * np.float32(0.5))
        parts.set_features(1, newx.ctypes.data)
        la, lb = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
        cached.forward(1, la.data_ptr()); plain.forward(1, lb.data_ptr())
        _close(cached.get(gcnsa.GET_ACT, 1, rows=parts.info(1).n), plain.get(gcnsa.GET_ACT, 1, rows=parts.info(1).n),
               what="H1 after the feature rows changed")
        assert abs(la.item() - lb.item()) <= 1e-5 * abs(lb.item())
        cached.close(); plain.close(); parts.close()


@pytest.mark.parametrize("dims,factored_norm,use_bias", [
    ([64, 1, 1], 1, 1), ([64, 64, 64], 1, 1), ([64, 65, 3], 1, 1), ([5, 3, 2], 1, 0), ([33, 33, 17, 5], 1, 1), ([61, 50, 29, 13], 0, 1),
    ([30, 64, 33, 7], 1, 1)])
def test_narrow_layers_of_small_partitions_match_checker(tiny_wl, dims, factored_norm, use_bias):
    """Products of at most 64 inner columns and 64 wide run outside the tensor cores on partitions of up to 4 096 rows: widths at
    and beside the quads and the limit, a widening layer, without bias, with stored values.  Bars of the other tests."""
    w = copy.copy(tiny_wl)
    rng = np.random.default_rng(len(dims) + dims[1])
    w.dims, w.x = dims, np.ascontiguousarray(w.x[:, :dims[0]])
    w.y = rng.integers(0, dims[-1], len(w.y)).astype(np.int32)
    shapes = list(zip(dims[:-1], dims[1:]))
    w.w0 = [(rng.standard_normal(s) / np.sqrt(s[0])).astype(np.float32) for s in shapes]
    w.b0 = [(rng.standard_normal(s[1]) * (0.1 if use_bias else 0.0)).astype(np.float32) for s in shapes]
    env, parts, model = _make(w, gemm_mode=gcnsa.GEMM_TF32X3, factored_norm=factored_norm, use_bias=use_bias)
    _, rparts = oracle.build_partitions(w.rowptr, w.col, w.m, w.overlap_ppm, w.seed, w.part_mode, w.user_part)
    ws, bs = [a.astype(np.float64) for a in w.w0], [b.astype(np.float64) for b in w.b0]
    L = len(shapes)
    gw, gb = [np.zeros_like(a) for a in ws], [np.zeros_like(b) for b in bs]
    for p, pt in enumerate(rparts):
        fw = oracle.forward(pt, w.x[pt.members], ws, bs if use_bias else None, w.y[pt.members], w.train_mask[pt.members],
                            w.loss_on_halo)
        model.forward(p)
        h_gpu = [model.get(gcnsa.GET_ACT, l, rows=pt.n) for l in range(1, L + 1)]
        for l in range(L):
            _close(h_gpu[l], fw["H"][l + 1], what=f"p{p} H{l + 1}")
        bw = oracle.backward(pt, fw, ws, w.y[pt.members], relu_on=_relu_decisions(fw, h_gpu[:-1]))
        model.backward(p)
        for l in range(L):
            gw[l] += bw["dW"][l]; gb[l] += bw["db"][l]
    for l in range(L):
        _close(model.get(gcnsa.GET_GRAD_W, l), gw[l], what=f"dW{l}")
        if use_bias:
            _close(model.get(gcnsa.GET_GRAD_B, l), gb[l], what=f"db{l}")
    assert gcnsa.tc_status() == 0
    model.close(); parts.close()


@pytest.mark.parametrize("dims,on_tensor_cores", [([64, 16, 5], 2), ([64, 48, 10], 2), ([64, 48, 40], 2), ([64, 48, 41], 4),
                                                  ([64, 64, 5], 3), ([64, 64, 30], 3), ([64, 64, 31], 5), ([64, 64, 64], 5)])
def test_wide_products_of_small_partitions_stay_on_the_tensor_cores(tiny_wl, dims, on_tensor_cores):
    """Of a partition's five products the two weight gradients always run there, the others where they have more than 48 x 40
    weights (the first of the forward pass: 64 x 48)."""
    w = copy.copy(tiny_wl)
    rng = np.random.default_rng(1)
    w.dims, w.y = dims, rng.integers(0, dims[-1], len(w.y)).astype(np.int32)
    w.w0 = [(rng.standard_normal(s) / np.sqrt(s[0])).astype(np.float32) for s in zip(dims[:-1], dims[1:])]
    w.b0 = [np.zeros(d, np.float32) for d in dims[1:]]
    env, parts, model = _make(w, gemm_mode=gcnsa.GEMM_TF32X3, factored_norm=1)
    tc0, fb0 = gcnsa.gemm_path_counts()
    model.forward(0)
    model.backward(0)
    tc1, fb1 = gcnsa.gemm_path_counts()
    assert (tc1 - tc0, fb1 - fb0) == (on_tensor_cores, 0)
    model.close(); parts.close()


def test_weight_gradients_of_partitions_side_by_side_keep_fp32_accuracy(small_wl):
    """Partitions of 5 500 rows (172 k-blocks) whose products are cut for several that run at once: the first layer's weight
    gradient against the checker in the 2-norm.  A slice has at most 18 k-blocks with one cut of at most 2^-23 per 8 k, half of
    that on average, on a sum that is half its end on average: 2^-23 per k-block, 2.1e-6, with the dropped terms 2.3e-6;
    0.4e-6 for the sparse products and the softmax in front of it."""
    w = small_wl
    env, parts, model = _make(w, gemm_mode=gcnsa.GEMM_TF32X3, factored_norm=1)
    _, rparts = oracle.build_partitions(w.rowptr, w.col, w.m, w.overlap_ppm, w.seed, w.part_mode, w.user_part)
    ws, bs = [a.astype(np.float64) for a in w.w0], [b.astype(np.float64) for b in w.b0]
    gw = np.zeros_like(ws[0])
    for p, pt in enumerate(rparts):
        assert pt.n > 5000
        fw = oracle.forward(pt, w.x[pt.members], ws, bs, w.y[pt.members], w.train_mask[pt.members], w.loss_on_halo)
        model.forward(p)
        h_gpu = [model.get(gcnsa.GET_ACT, l, rows=pt.n) for l in (1, 2)]
        gw += oracle.backward(pt, fw, ws, w.y[pt.members], relu_on=_relu_decisions(fw, h_gpu[:-1]))["dW"][0]
        model.backward(p)
    err = np.linalg.norm(model.get(gcnsa.GET_GRAD_W, 0) - gw) / np.linalg.norm(gw)
    assert gcnsa.tc_status() == 0 and err <= 2.7e-6, err
    model.close(); parts.close()


@pytest.mark.parametrize("rows,dims", [((9500, 9215, 8200), [500, 64, 5]), ((8500, 8245, 4500), [602, 128, 7])])
@pytest.mark.parametrize("epoch_graph", [0, 1])
def test_products_of_partitions_of_any_size_have_their_workspace(rows, dims, epoch_graph):
    """Partitions with fewer rows than the largest may be cut into more k-slices (500 x 64: 33 of 9 500 rows, 36 of 9 215): no
    product falls back to the fp32 FMA kernel."""
    n = sum(rows)
    rowptr, col = graphs.permutation_graph(n, 3, 5)
    rng = np.random.default_rng(n)
    x = rng.standard_normal((n, dims[0]), dtype=np.float32)
    w0 = [(rng.standard_normal(s) / np.sqrt(s[0])).astype(np.float32) for s in zip(dims[:-1], dims[1:])]
    with torch.cuda.stream(torch.cuda.Stream()):
        env = gcnsa.make_env(0)
        parts = gcnsa.Parts(env, rowptr, col, x, rng.integers(0, dims[-1], n), np.ones(n, np.uint8), dims[-1], len(rows), 0, 3,
                            gcnsa.PART_USER, np.repeat(np.arange(len(rows)), rows).astype(np.int32))
        assert tuple(parts.info(p).n for p in range(len(rows))) == rows
        model = gcnsa.Model(env, parts, dims, w0, gemm_mode=gcnsa.GEMM_TF32X3, epoch_graph=epoch_graph)
        tc0, fb0 = gcnsa.gemm_path_counts()
        for _ in range(2):
            model.epoch()
        tc1, fb1 = gcnsa.gemm_path_counts()
        assert tc1 > tc0 and fb1 == fb0 and gcnsa.tc_status() == 0
        model.close(); parts.close()


@pytest.mark.parametrize("c", [1, 32, 33, 64, 65, 128, 129, 256, 257])
def test_last_layer_gradients_for_every_number_of_classes(tiny_wl, c):
    """The softmax kernel holds a row in 8, 16 or 32 lanes, one or two float4 each (up to 32, 64, 128, 256 columns), and
    writes the scaled copy and the partial column sums the last layer's backward pass starts from; wider rows take the
    row kernel and the column-sum kernel.  Loss, logit gradient, dW and db against the checker, at the bars of the
    other tests (fp32 sums over at most a partition's rows)."""
    w = copy.copy(tiny_wl)
    rng = np.random.default_rng(c)
    f, h = w.dims[0], 300
    w.dims = [f, h, c]
    w.y = rng.integers(0, c, len(w.y)).astype(np.int32)
    w.w0 = [(rng.standard_normal(s) / np.sqrt(s[0])).astype(np.float32) for s in ((f, h), (h, c))]
    w.b0 = [rng.standard_normal(s).astype(np.float32) * 0.1 for s in (h, c)]
    env, parts, model = _make(w, gemm_mode=gcnsa.GEMM_TF32X3, factored_norm=1)
    _, rparts = oracle.build_partitions(w.rowptr, w.col, w.m, w.overlap_ppm, w.seed, w.part_mode, w.user_part)
    ws, bs = [a.astype(np.float64) for a in w.w0], [b.astype(np.float64) for b in w.b0]
    gw, gb = [np.zeros_like(a) for a in ws], [np.zeros_like(b) for b in bs]
    loss = torch.zeros(1, device="cuda")
    for p, pt in enumerate(rparts):
        fw = oracle.forward(pt, w.x[pt.members], ws, bs, w.y[pt.members], w.train_mask[pt.members], w.loss_on_halo)
        model.forward(p, loss.data_ptr())
        assert abs(loss.item() - fw["loss"]) <= 1e-5 * max(abs(fw["loss"]), 1e-6)
        h_gpu = [model.get(gcnsa.GET_ACT, l, rows=pt.n) for l in (1, 2)]
        bw = oracle.backward(pt, fw, ws, w.y[pt.members], relu_on=_relu_decisions(fw, h_gpu[:-1]))
        _close(model.get(gcnsa.GET_DLOGITS, rows=pt.n), bw["G"][1], what=f"p{p} dlogits")
        model.backward(p)
        for l in range(2):
            gw[l] += bw["dW"][l]; gb[l] += bw["db"][l]
    for l in range(2):
        _close(model.get(gcnsa.GET_GRAD_W, l), gw[l], what=f"dW{l}")
        _close(model.get(gcnsa.GET_GRAD_B, l), gb[l], what=f"db{l}")
    assert gcnsa.tc_status() == 0
    model.close(); parts.close()


@pytest.mark.parametrize("agg_mode", [gcnsa.AGG_GRAD_AVG, gcnsa.AGG_PARAM_AVG])
def test_a_gradient_set_before_an_epoch_is_part_of_its_sum(tiny_wl, agg_mode):
    """gcnsa_model_set may put a gradient into the sum (a penalty on the weights, say): the epoch that follows adds the
    partitions' gradients to it and clears it, bit for bit as the calls step by step do."""
    w = tiny_wl
    rng = np.random.default_rng(5)
    extra = {(what, l): rng.standard_normal(s).astype(np.float32) for l, (a, b) in enumerate(zip(w.dims[:-1], w.dims[1:]))
             for what, s in ((gcnsa.GET_GRAD_W, (a, b)), (gcnsa.GET_GRAD_B, (b,)))}
    results = []
    for how in ("steps", "plain", "recorded", "host"):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            env = gcnsa.make_env(0)
            parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                                w.part_mode, w.user_part, w.loss_on_halo)
            model = gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr, agg_mode=agg_mode, epoch_graph=how == "recorded")
            for e in range(3):
                if e != 1:
                    for (what, l), g in extra.items():
                        model.set(what, l, g)
                if how == "steps":
                    for p in range(w.m):
                        model.forward(p)
                        model.backward(p)
                    model.step()
                elif how == "host":
                    xs = [np.ascontiguousarray(w.x[parts.members(p)]) for p in range(w.m)]
                    model.epoch_host([x.ctypes.data for x in xs], np.zeros(1, np.float32))
                else:
                    model.epoch()
                assert not any(model.get(what, l).any() for what, l in extra)
            results.append([model.get(what, l) for what in (gcnsa.GET_W, gcnsa.GET_B, gcnsa.GET_ADAM_M_W) for l in range(2)])
            model.close()
            parts.close()
    for other in results[1:]:
        for a, b in zip(results[0], other):
            assert np.array_equal(a, b)


def test_an_empty_partition_leaves_no_bias_gradient_of_other_partitions(tiny_wl):
    """One model trained in turn on two cuts of a graph, the second with an empty partition: that partition adds nothing to
    the sum, so an epoch is bit for bit that of the calls step by step."""
    w = tiny_wl
    n = w.rowptr.size - 1
    even = (np.arange(n) * 3 // n).astype(np.int32)
    got = []
    for how in ("steps", "epoch"):
        env = gcnsa.make_env(0)
        cuts = [gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], 3, 0, 5, gcnsa.PART_USER, user)
                for user in (np.zeros(n, np.int32), even, np.where(even == 1, 2, even).astype(np.int32))]
        assert cuts[2].info(1).n == 0
        model = gcnsa.Model(env, cuts[0], w.dims, w.w0, w.b0, lr=w.lr, epoch_graph=0)
        for parts in (cuts[1], cuts[2], cuts[2]):
            model.parts = parts
            if how == "epoch":
                model.epoch()
                continue
            for p in range(3):
                model.forward(p)
                model.backward(p)
            model.step()
        got.append([model.get(what, l) for what in (gcnsa.GET_W, gcnsa.GET_B, gcnsa.GET_ADAM_M_B) for l in range(2)])
        model.close()
        for parts in cuts:
            parts.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("epoch_graph", [0, 1])
def test_no_backward_pass_after_an_epoch_has_replaced_the_activations(tiny_wl, epoch_graph):
    """forward, epoch, backward is refused whether the epoch is launched, recorded or replayed."""
    w = tiny_wl
    with torch.cuda.stream(torch.cuda.Stream()):
        env = gcnsa.make_env(0)
        parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                            w.part_mode, w.user_part, w.loss_on_halo)
        model = gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr, epoch_graph=epoch_graph)
        for _ in range(3):
            model.forward(0)
            model.epoch()
            with pytest.raises(gcnsa.GcnsaError) as ei:
                model.backward(0)
            assert ei.value.code == gcnsa.ERR_ORDER
        model.close()
        parts.close()


def test_several_threads_may_read_a_models_tensors(small_wl):
    """gcnsa_model_get leaves the model as it is: threads that read different layers at the same time get what one thread
    gets (rows whose width is not that of the device's are packed on the way)."""
    w = small_wl
    env = gcnsa.make_env(0)
    dims = [w.dims[0], 45, 37, w.dims[-1]]
    rng = np.random.default_rng(4)
    w0 = [rng.standard_normal(s).astype(np.float32) * 0.1 for s in zip(dims[:-1], dims[1:])]
    parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                        w.part_mode, w.user_part, w.loss_on_halo)
    model = gcnsa.Model(env, parts, dims, w0, loss_rows_only=0, epoch_graph=0)
    model.forward(0)
    n = parts.info(0).n
    want = {l: model.get(gcnsa.GET_ACT, l, n) for l in (1, 2, 3)}
    wrong = []

    def read(l):
        for _ in range(60):
            if not np.array_equal(model.get(gcnsa.GET_ACT, l, n), want[l]):
                wrong.append(l)

    threads = [threading.Thread(target=read, args=(l,)) for l in (1, 2, 3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
    model.close()
    parts.close()
