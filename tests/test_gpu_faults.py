"""Failures made on the host, handled on the GPU machine: an allocator callback
that returns NULL on its k-th call (a simulated out-of-memory condition) for
every k until the call succeeds.  Each failing call must report GCNSA_ERR_OOM,
hand back everything it was given (the callback counts), and leave the context
usable for the next call.  Nothing here faults, traps or hangs the GPU."""
import ctypes as C

import numpy as np
import pytest
import torch

from gen import configs, graphs
from paper_2012_04930_b200 import gcnsa

pytestmark = pytest.mark.gpu


class FailingAllocator:
    """gcnsa_env callbacks on top of torch's caching allocator; call number `fail_at` (1-based) returns NULL."""

    def __init__(self):
        self.calls, self.fail_at, self.on, self.live = 0, 0, False, {}
        self.alloc_cb = gcnsa.ALLOC_FN(self._alloc)
        self.free_cb = gcnsa.FREE_FN(self._free)

    def arm(self, fail_at, on=False):
        """on: every call from number fail_at on is refused, not that one alone."""
        self.calls, self.fail_at, self.on = 0, fail_at, on

    def _alloc(self, nbytes, user):
        self.calls += 1
        if self.calls == self.fail_at or (self.on and self.calls > self.fail_at):
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), stream=torch.cuda.current_stream())
        self.live[p] = int(nbytes)
        return p

    def _free(self, ptr, user):
        assert ptr in self.live, "free of a pointer the allocator never handed out (or a second free)"
        del self.live[ptr]
        torch.cuda.caching_allocator_delete(ptr)

    def env(self):
        e = gcnsa.make_env(0)
        e.alloc, e.free = self.alloc_cb, self.free_cb
        return e


def _until_success(alloc, call, keeps=False, limit=400):
    """Runs call() with the k-th allocation failing for k = 1, 2, ...; returns (k of the first success, result).
    keeps: the object under test may keep what a failed call had already obtained (buffers made on first use)."""
    for k in range(1, limit):
        alloc.arm(k)
        live_before = set(alloc.live)
        try:
            out = call()
        except gcnsa.GcnsaError as e:
            assert e.code == gcnsa.ERR_OOM, (k, e)
            assert alloc.calls >= k
            torch.cuda.synchronize()
            if not keeps:
                leaked = set(alloc.live) - live_before
                assert not leaked, f"allocation {k} failed and {len(leaked)} buffers were not handed back"
            continue
        assert alloc.calls < k, "the call succeeded although one of its allocations was refused"
        return k, out
    raise AssertionError("no success within the limit")


@pytest.mark.parametrize("builder", [gcnsa.BUILD_DEVICE, gcnsa.BUILD_HOST])
def test_out_of_memory_while_building_partitions(builder, tiny_wl):
    w = tiny_wl
    alloc = FailingAllocator()
    env = alloc.env()

    def build():
        return gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                           w.part_mode, w.user_part, w.loss_on_halo, builder=builder)

    k, parts = _until_success(alloc, build)
    assert k > 10, "the build makes many allocations: each of them was made to fail once"
    alloc.arm(0)
    # the object built right after the failures is a good one: same structure as a build with torch's allocator
    good = gcnsa.Parts(gcnsa.make_env(0), w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                       w.part_mode, w.user_part, w.loss_on_halo, builder=builder)
    for p in range(w.m):
        a, b = parts.export(p), good.export(p)
        for key in a:
            assert np.array_equal(a[key], b[key]), key
    good.close()
    parts.close()
    torch.cuda.synchronize()
    assert not alloc.live, "destroy releases every buffer"


@pytest.mark.parametrize("agg_mode,cache_ax", [(gcnsa.AGG_GRAD_AVG, 0), (gcnsa.AGG_PARAM_AVG, 1)])
def test_out_of_memory_while_creating_and_using_a_model(agg_mode, cache_ax, tiny_wl):
    w = tiny_wl
    alloc = FailingAllocator()
    env = alloc.env()
    parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                        w.part_mode, w.user_part, w.loss_on_halo)
    held = set(alloc.live)

    def create():
        return gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr, agg_mode=agg_mode, cache_ax=cache_ax,
                           **{**gcnsa.MEASURED, "epoch_graph": 0})

    k, model = _until_success(alloc, create)
    assert k > 10
    alloc.arm(0)
    loss = torch.zeros(1, device="cuda")
    model.epoch(loss.data_ptr())
    first = loss.item()
    assert np.isfinite(first)
    # the buffers evaluation and the host-buffer epoch allocate on first use: a failure there is an error code, and
    # the call works when it is made again
    k_ev, (correct, total, _) = _until_success(alloc, lambda: model.evaluate(parts, 0), keeps=True)
    assert k_ev >= 2 and 0 <= correct <= total == parts.info(0).n
    xs = [np.ascontiguousarray(w.x[parts.members(p)]) for p in range(w.m)]
    loss_h = np.zeros(1, np.float32)
    k_eh, _ = _until_success(alloc, lambda: model.epoch_host([x.ctypes.data for x in xs], loss_h), keeps=True)
    assert k_eh >= 2 and np.isfinite(loss_h[0]) and loss_h[0] <= first
    alloc.arm(0)
    model.close()
    torch.cuda.synchronize()
    assert held <= set(alloc.live) and len(set(alloc.live) - held) <= 2   # the partitions and their two staging buffers
    parts.close()
    torch.cuda.synchronize()
    assert not alloc.live


def _planned_graph(n, target_nnz):
    rowptr, col, comm = graphs.chung_lu_communities(n, target_nnz, 2.1, 3, 0.93, 5)
    rng = np.random.default_rng(n)
    return (rowptr, col, rng.standard_normal((n, 20)).astype(np.float32), (comm % 7).astype(np.int32),
            (rng.random(n) < 0.9).astype(np.uint8), 7, 1, 0, 3)


@pytest.mark.parametrize("builder", [gcnsa.BUILD_DEVICE, gcnsa.BUILD_HOST])
@pytest.mark.parametrize("n,target_nnz", [(3001, 640_000), (12_003, 300_000)])
def test_no_memory_for_a_plan_or_for_row_lists_is_no_failure(builder, n, target_nnz):
    """The plan of the tensor-core products (first graph) and the row lists by length (second graph) only save time: where
    one of their allocations is refused, alone or with all after it, the build succeeds and the products are right."""
    alloc = FailingAllocator()
    env = alloc.env()
    small = _planned_graph(200, 2000)
    alloc.arm(0)
    gcnsa.Parts(env, *small, builder=builder).close()
    required = alloc.calls                     # with one partition, the same for every graph
    args = _planned_graph(n, target_nnz)
    w0 = [np.random.default_rng(1).standard_normal((20, 7)).astype(np.float32)]

    def logits(parts):
        m = gcnsa.Model(gcnsa.make_env(0), parts, [20, 7], w0, loss_rows_only=0, epoch_graph=0)
        m.forward(0)
        out = m.get(gcnsa.GET_ACT, 1, n)
        m.close()
        return out

    alloc.arm(0)
    parts = gcnsa.Parts(env, *args, builder=builder)
    total, want, full = alloc.calls, logits(parts), len(alloc.live)
    parts.close()
    assert total >= required + 6 and not alloc.live
    for k in range(required + 1, total + 1):
        for on in (False, True):
            alloc.arm(k, on)
            parts = gcnsa.Parts(env, *args, builder=builder)
            assert len(alloc.live) <= full
            if on:
                # sums of up to a few hundred terms in another order, and another rounding of the three terms
                assert np.abs(logits(parts) - want).max() <= 2e-5 * np.abs(want).max(), k
            parts.close()
            assert not alloc.live, k


def test_a_rejected_plan_keeps_no_memory():
    """A graph that is looked at for a plan and gets none holds as many buffers as one that is not looked at."""
    alloc = FailingAllocator()
    env = alloc.env()
    small = gcnsa.Parts(env, *_planned_graph(200, 2000))
    held = len(alloc.live)
    small.close()
    n = 10_001
    rowptr, col = graphs.permutation_graph(n, 27, 5)
    assert col.size + n >= 1 << 19
    rng = np.random.default_rng(2)
    parts = gcnsa.Parts(env, rowptr, col, rng.standard_normal((n, 4)).astype(np.float32), np.zeros(n, np.int32),
                        np.ones(n, np.uint8), 2, 1, 0, 3)
    assert len(alloc.live) == held
    parts.close()
    assert not alloc.live


def test_scratch_of_the_build_stays_within_the_stated_bound():
    """A partition so large for its degree that the tables of a plan would outgrow its matrix: it is not looked at (no
    request is larger than the graph's own arrays), and the scratch of the whole build is what gcnsa.h states."""
    n, f = 720_001, 4
    rowptr, col = graphs.permutation_graph(n, 21, 5)
    assert col.size >= 40 * n
    rng = np.random.default_rng(2)

    class Recorder(FailingAllocator):
        peak = largest = 0

        def _alloc(self, nbytes, user):
            p = super()._alloc(nbytes, user)
            self.largest, self.peak = max(self.largest, int(nbytes)), max(self.peak, sum(self.live.values()))
            return p

    alloc = Recorder()
    parts = gcnsa.Parts(alloc.env(), rowptr, col, rng.standard_normal((n, f)).astype(np.float32), np.zeros(n, np.int32),
                        np.ones(n, np.uint8), 2, 1, 0, 3)
    nnz = parts.info(0).nnz
    assert alloc.largest <= 4 * (nnz + n + 1)
    scratch = alloc.peak - sum(alloc.live.values())
    assert scratch <= 37 * n + 4 * col.size + 4 * n * f + 24 * nnz + 64 * n + (8 << 20)
    parts.close()


@pytest.mark.parametrize("agg_mode,cache_ax", [(gcnsa.AGG_GRAD_AVG, 0), (gcnsa.AGG_PARAM_AVG, 1)])
def test_a_model_without_memory_for_planned_products_gathers(agg_mode, cache_ax):
    """The workspace of the planned products is asked for after everything a model needs; without it the model trains on
    the gathers, with the losses of a model that has it up to rounding."""
    alloc = FailingAllocator()
    env = alloc.env()
    args = _planned_graph(3001, 640_000)
    parts = gcnsa.Parts(gcnsa.make_env(0), *args)
    rng = np.random.default_rng(1)
    w0 = [rng.standard_normal(s).astype(np.float32) / np.float32(np.sqrt(s[0])) for s in ((20, 12), (12, 7))]
    losses = {}
    for fail_at in (0, -1):      # -1: the last allocation of the first model
        alloc.arm(0 if fail_at == 0 else calls)
        m = gcnsa.Model(env, parts, [20, 12, 7], w0, agg_mode=agg_mode, cache_ax=cache_ax, epoch_graph=0)
        calls = alloc.calls
        loss = torch.zeros(1, device="cuda")
        before = gcnsa.launch_count()
        out = []
        for _ in range(3):
            m.epoch(loss.data_ptr())
            out.append(loss.item())
        losses[fail_at] = out, gcnsa.launch_count() - before
        m.close()
        assert not alloc.live
    assert losses[-1][1] < losses[0][1], "planned products take more launches than gathers"
    assert np.allclose(losses[0][0], losses[-1][0], rtol=1e-4)
    parts.close()


def _sparse_parts(env, m, rows, f, c):
    """m partitions of the same ring of `rows` vertices: few entries, many rows."""
    rp, cl = graphs.from_edge_list(rows, np.stack([np.arange(rows), (np.arange(rows) + 1) % rows], 1))
    rowptr = np.concatenate([[0], np.cumsum(np.tile(np.diff(rp), m))])
    col = (np.tile(cl.astype(np.int64), m) + np.repeat(np.arange(m) * rows, cl.size)).astype(np.int32)
    rng = np.random.default_rng(m)
    x = rng.standard_normal((m * rows, f)).astype(np.float32)
    return gcnsa.Parts(env, rowptr, col, x, np.zeros(m * rows, np.int32), np.ones(m * rows, np.uint8), c, m, 0, 3)


def test_side_by_side_partitions_take_bounded_memory():
    """The buffers with which a recorded epoch runs partitions side by side: at most 1 GiB above the model of a caller who
    records nothing, whatever the rows; none on the default stream, which cannot be recorded."""
    rng = np.random.default_rng(1)
    for rows, dims in ((1000, [16, 8, 3]), (40_000, [256, 256, 3])):
        w0 = [rng.standard_normal(s).astype(np.float32) * 0.05 for s in zip(dims[:-1], dims[1:])]
        held = {}
        for name, stream, graph in (("plain", torch.cuda.Stream(), 0), ("recorded", torch.cuda.Stream(), 1),
                                    ("default", torch.cuda.default_stream(), 1)):
            with torch.cuda.stream(stream):
                alloc = FailingAllocator()
                env = alloc.env()
                parts = _sparse_parts(gcnsa.make_env(0), 8, rows, dims[0], dims[-1])
                m = gcnsa.Model(env, parts, dims, w0, epoch_graph=graph)
                held[name] = sum(alloc.live.values())
                m.close()
                parts.close()
        assert held["default"] == held["plain"]
        assert held["plain"] < held["recorded"] <= held["plain"] + (1 << 30)


def test_many_partitions_of_a_large_model_share_one_gradient_sum():
    """The gradients of the partitions of an epoch are kept apart up to 64 MB; beyond that the memory of a model does not
    grow with the number of partitions times its parameters, and an epoch is bit for bit that of the calls step by step."""
    rng = np.random.default_rng(1)
    dims = [4000, 64, 3]
    w0 = [rng.standard_normal(s).astype(np.float32) * 0.05 for s in zip(dims[:-1], dims[1:])]
    with torch.cuda.stream(torch.cuda.Stream()):
        held = {}
        for m in (1, 100):
            parts = _sparse_parts(gcnsa.make_env(0), m, 50, dims[0], dims[-1])
            alloc = FailingAllocator()
            model = gcnsa.Model(alloc.env(), parts, dims, w0, epoch_graph=0)
            held[m] = sum(alloc.live.values())
            model.close()
        assert held[100] <= held[1]
        for agg_mode in (gcnsa.AGG_GRAD_AVG, gcnsa.AGG_PARAM_AVG):
            got = []
            for how in ("steps", "plain", "recorded"):
                model = gcnsa.Model(gcnsa.make_env(0), parts, dims, w0, agg_mode=agg_mode, epoch_graph=how == "recorded")
                for _ in range(3):
                    if how != "steps":
                        model.epoch()
                        continue
                    for p in range(100):
                        model.forward(p)
                        model.backward(p)
                    model.step()
                got.append([model.get(what, l) for what in (gcnsa.GET_W, gcnsa.GET_B) for l in range(2)])
                model.close()
            for other in got[1:]:
                for x, y in zip(got[0], other):
                    assert np.array_equal(x, y)
        parts.close()


@pytest.mark.parametrize("agg_mode,cache_ax", [(gcnsa.AGG_GRAD_AVG, 1), (gcnsa.AGG_PARAM_AVG, 0)])
def test_buffers_a_model_needs_come_before_those_that_save_time(agg_mode, cache_ax):
    """An allocator with just the memory of a model that records nothing: the same model that records is created too."""

    class Limited(FailingAllocator):
        room = 1 << 62

        def _alloc(self, nbytes, user):
            if sum(self.live.values()) + nbytes > self.room:
                return None
            return super()._alloc(nbytes, user)

    rng = np.random.default_rng(1)
    dims = [32, 16, 3]
    w0 = [rng.standard_normal(s).astype(np.float32) * 0.05 for s in zip(dims[:-1], dims[1:])]
    with torch.cuda.stream(torch.cuda.Stream()):
        parts = _sparse_parts(gcnsa.make_env(0), 8, 3000, dims[0], dims[-1])
        alloc = Limited()
        env = alloc.env()
        losses = []
        for graph in (0, 1):
            m = gcnsa.Model(env, parts, dims, w0, agg_mode=agg_mode, cache_ax=cache_ax, epoch_graph=graph)
            alloc.room = min(alloc.room, sum(alloc.live.values()))
            loss = torch.zeros(1, device="cuda")
            for _ in range(2):
                m.epoch(loss.data_ptr())
            losses.append(loss.item())
            m.close()
        assert losses[0] == losses[1] and not alloc.live
        parts.close()


def test_workers_side_by_side_take_bounded_memory():
    """GraphSAGE: the buffers of the workers after the first, at most 1 GiB together; none on the default stream."""
    dims = [16, 8, 3]
    rng = np.random.default_rng(1)
    ws = [rng.standard_normal(s).astype(np.float32) * 0.05 for s in zip(dims[:-1], dims[1:])]
    held = {}
    for fanout, batch in (((2000, 1), 16_000), ((4, 3), 64)):   # a quarter of a gigabyte of sample lists a worker; little
        for name, stream in (("own", torch.cuda.Stream()), ("default", torch.cuda.default_stream())):
            with torch.cuda.stream(stream):
                alloc = FailingAllocator()
                parts = _sparse_parts(gcnsa.make_env(0), 8, 300, dims[0], dims[-1])
                model = gcnsa.Sage(alloc.env(), parts, dims, ws, ws, fanout=fanout, batch=batch)
                held[name] = sum(alloc.live.values())
                model.epoch()
                stream.synchronize()
                model.close()
                parts.close()
                assert not alloc.live
        assert held["default"] < held["own"] <= held["default"] + (1 << 30)
