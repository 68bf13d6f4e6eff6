"""The products that run on the tensor cores through a partition's plan (256-row tiles of bits, a remainder of gathers),
against a dense fp64 computation of the same layers."""
import numpy as np
import pytest
import torch

from gen import graphs
from paper_2012_04930_b200 import gcnsa

pytestmark = pytest.mark.gpu

# fp32 sums of a few hundred terms (1e-6 of the largest entry) after dense products with a bound of 1e-5 of it
TOL = 2e-5


def _close(got, want, what):
    got, want = torch.as_tensor(got, dtype=torch.float64), want.double().cpu()
    err = ((got - want).abs().max() / want.abs().max()).item()
    assert err <= TOL, (what, err)


# widths of one to three slabs, each with the 16-, 32-, 48- and 64-wide kernel; rows that fill their tiles and rows that
# do not; every, no and some rows with loss; a hidden layer that narrows and one that widens (source rows scaled while
# they are split)
@pytest.mark.parametrize("n,dims,mask_p", [
    (3072, [20, 16], 0.5), (3001, [40, 7], 0.66), (2817, [40, 29], 0.66), (3001, [48, 41], 1.0), (2999, [70, 64], 0.3),
    (3001, [130, 100], 0.66), (3010, [150, 130], 0.66), (3001, [90, 33, 9], 0.66), (3001, [24, 72, 40, 5], 0.5),
    (3001, [40, 24, 7], 0.0)])
def test_planned_products_match_fp64(n, dims, mask_p):
    rowptr, col, comm = graphs.chung_lu_communities(n, 640_000, 2.1, 3, 0.93, 5)
    rng = np.random.default_rng(n + dims[0])
    x = rng.standard_normal((n, dims[0]), dtype=np.float32)
    y = (comm % dims[-1]).astype(np.int32)
    mask = (rng.random(n) < mask_p).astype(np.uint8)
    w0 = [rng.standard_normal((a, b), dtype=np.float32) / np.float32(np.sqrt(a)) for a, b in zip(dims[:-1], dims[1:])]
    env = gcnsa.make_env(0)
    parts = gcnsa.Parts(env, rowptr, col, x, y, mask, dims[-1], 1, 0, 3)
    A = torch.zeros((n, n), dtype=torch.float64)
    A[np.repeat(np.arange(n), np.diff(rowptr)), torch.from_numpy(col.astype(np.int64))] = 1.0
    A += torch.eye(n, dtype=torch.float64)
    dinv = A.sum(1).rsqrt()
    A = (dinv[:, None] * A * dinv[None, :]).cuda()
    ws = [torch.from_numpy(w).double().cuda().requires_grad_() for w in w0]
    acts, h = [], torch.from_numpy(x).double().cuda()
    for l, w in enumerate(ws):
        h = A @ (h @ w)
        if l < len(ws) - 1:
            h = torch.relu(h)
        acts.append(h)
    on = torch.from_numpy(mask).bool().cuda()
    if mask.any():
        torch.nn.functional.cross_entropy(h[on], torch.from_numpy(y).long().cuda()[on]).backward()
    launches = {}
    for loss_rows_only in (0, 1):
        for fact in (0, 1):
            m = gcnsa.Model(env, parts, dims, w0, loss_rows_only=loss_rows_only, factored_norm=fact, epoch_graph=0)
            before = gcnsa.launch_count()
            m.forward(0)
            launches[fact] = gcnsa.launch_count() - before
            m.backward(0)
            if fact:
                for l in range(1, len(dims)):
                    got, want = m.get(gcnsa.GET_ACT, l, n), acts[l - 1].detach()
                    if l == len(dims) - 1 and loss_rows_only:
                        got, want = got[mask.astype(bool)], want[on]
                    if want.numel():
                        _close(got, want, ("H", l, loss_rows_only))
                for l, w in enumerate(ws):
                    g = m.get(gcnsa.GET_GRAD_W, l)
                    if mask.any():
                        _close(g, w.grad, ("dW", l, loss_rows_only))
                    else:
                        assert not g.any()
            m.close()
    assert launches[1] > launches[0], "the planned path did not run"
    assert gcnsa.tc_status() == 0
    parts.close()


def _reference(rowptr, col, n):
    A = torch.zeros((n, n), dtype=torch.float64)
    A[np.repeat(np.arange(n), np.diff(rowptr)), torch.from_numpy(col.astype(np.int64))] = 1.0
    A += torch.eye(n, dtype=torch.float64)
    dinv = A.sum(1).rsqrt()
    return (dinv[:, None] * A * dinv[None, :]).cuda()


# what a source row does to the rows that do not have it as a neighbour (nothing), and to sums between half of the largest
# fp32 number and that number (they are finite); one layer that multiplies first and one that aggregates first
@pytest.mark.parametrize("dims", [[16, 16], [16, 20], [80, 80]])
@pytest.mark.parametrize("loss_rows_only", [0, 1])
def test_planned_products_with_values_that_are_not_finite_or_very_large(dims, loss_rows_only):
    n = 3001
    rowptr, col, comm = graphs.chung_lu_communities(n, 640_000, 2.1, 3, 0.93, 5)
    rng = np.random.default_rng(7)
    x = rng.standard_normal((n, dims[0]), dtype=np.float32)
    mask = (rng.random(n) < 0.66).astype(np.uint8)
    w0 = [np.eye(dims[0], dims[1], dtype=np.float32)]
    env = gcnsa.make_env(0)
    parts = gcnsa.Parts(env, rowptr, col, x, (comm % 3).astype(np.int32), mask, dims[1], 1, 0, 3)
    A = _reference(rowptr, col, n)
    m = gcnsa.Model(env, parts, dims, w0, use_bias=0, loss_rows_only=loss_rows_only, epoch_graph=0)
    rows = mask.astype(bool) if loss_rows_only else np.ones(n, bool)

    def forward(values):
        values = np.ascontiguousarray(values)
        parts.set_features(0, values.ctypes.data)
        before = gcnsa.launch_count()
        m.forward(0)
        assert gcnsa.launch_count() - before >= 5, "the planned path did not run"
        return m.get(gcnsa.GET_ACT, 1, n)[rows]

    clean = forward(x)
    v = int(np.argmin(np.diff(rowptr)))
    near = np.zeros(n, bool)
    near[col[rowptr[v]:rowptr[v + 1]]] = True
    near[v] = True
    assert 0 < near[rows].sum() < rows.sum() // 2
    for bad in (np.inf, -np.inf, np.nan):
        broken = x.copy()
        broken[v, 3] = bad
        got = forward(broken)
        assert not np.isfinite(got[near[rows]][:, 3]).any()
        # (the same sums in another order and another rounding of the three terms)
        assert np.abs(got[~near[rows]] - clean[~near[rows]]).max() <= 2e-5 * np.abs(clean).max()
        assert np.array_equal(forward(x), clean), "the next product is planned again"
    # sums of about 0.9 of the largest fp32 number, before the rows are scaled by d^-1/2
    big = np.abs(x)
    deg = torch.from_numpy(np.diff(rowptr) + 1).double().cuda().sqrt()
    top = (deg[:, None] * (A @ torch.from_numpy(big).double().cuda())).max().item()
    big *= np.float32(0.9 * np.finfo(np.float32).max / top)
    want = (A @ torch.from_numpy(big).double().cuda()) @ torch.from_numpy(w0[0]).double().cuda()
    _close(forward(big), want[torch.from_numpy(rows).cuda()], "large values")
    # and values whose terms are subnormal: the planned product's absolute error is that of the smallest normal number
    tiny = x * np.float32(2.0 ** -112)
    want = (A @ torch.from_numpy(tiny).double().cuda()) @ torch.from_numpy(w0[0]).double().cuda()
    _close(forward(tiny), want[torch.from_numpy(rows).cuda()], "small values")
    m.close()
    parts.close()


# rows of at most 64 entries go to a group of lanes, longer ones to a warp, those above 256 to a block; one width per
# kernel shape, and a graph without locality whose gathered matrix exceeds L2 (column slabs)
@pytest.mark.parametrize("n,width", [(12_003, 7), (12_003, 30), (12_003, 41), (12_003, 64), (12_003, 100), (12_003, 130),
                                     (12_003, 300), (12_003, 400), (12_003, 520), (300_001, 101)])
def test_rows_by_length_match_fp64(n, width):
    if n < 100_000:
        rowptr, col, _ = graphs.chung_lu_communities(n, 300_000, 2.1, 12, 0.7, 5)
        assert (np.diff(rowptr) > 256).any() and (np.diff(rowptr) <= 64).mean() > 0.5
    else:
        rowptr, col = graphs.permutation_graph(n, 4, 5)
    rng = np.random.default_rng(n + width)
    x = rng.standard_normal((n, width), dtype=np.float32)
    y = rng.integers(0, width, n).astype(np.int32)
    mask = (rng.random(n) < 0.9).astype(np.uint8)
    w0 = [np.eye(width, dtype=np.float32)]
    env = gcnsa.make_env(0)
    parts = gcnsa.Parts(env, rowptr, col, x, y, mask, width, 1, 0, 3)
    ex = parts.export(0)
    crow, ccol = (torch.from_numpy(ex[k].astype(np.int64)).cuda() for k in ("rowptr", "col"))
    dinv = (crow[1:] - crow[:-1]).double().rsqrt()
    pattern = torch.sparse_csr_tensor(crow, ccol, torch.ones(ccol.numel(), dtype=torch.float64, device="cuda"), size=(n, n))
    on = mask.astype(bool)

    def product(v):
        return dinv[:, None] * (pattern @ (dinv[:, None] * v))

    want = product(torch.from_numpy(x).double().cuda())
    for fact in (0, 1):
        m = gcnsa.Model(env, parts, [width, width], w0, use_bias=0, factored_norm=fact, epoch_graph=0)
        m.forward(0)
        _close(m.get(gcnsa.GET_ACT, 1, n)[on], want[torch.from_numpy(on).cuda()], ("logits", fact))
        g = torch.from_numpy(m.get(gcnsa.GET_DLOGITS, 1, n)).double().cuda()
        m.backward(0)
        _close(m.get(gcnsa.GET_GRAD_W, 0), torch.from_numpy(x).double().cuda().T @ product(g), ("dW", fact))
        m.close()
    parts.close()


def test_profile_charges_a_planned_product_with_its_own_bytes():
    """l1_bytes of a product through a plan: three launches, more than the compulsory bytes and far less than one gather of a
    source row per stored entry, which is what the product without the plan is charged with."""
    n, f = 3001, 41
    rowptr, col, comm = graphs.chung_lu_communities(n, 640_000, 2.1, 3, 0.93, 5)
    x = np.random.default_rng(3).standard_normal((n, f), dtype=np.float32)
    env = gcnsa.make_env(0)
    parts = gcnsa.Parts(env, rowptr, col, x, (comm % 3).astype(np.int32), np.ones(n, np.uint8), f, 1, 0, 3)
    got = {}
    for fact in (0, 1):
        m = gcnsa.Model(env, parts, [f, f], [np.eye(f, dtype=np.float32)], factored_norm=fact, epoch_graph=0)
        m.profile(True)
        m.forward(0)
        got[fact] = m.profile_read()["spmm"]
        m.close()
    gathers = 4.0 * f * parts.info(0).nnz
    assert got[0]["launches"] == 1 and got[0]["l1_bytes"] > gathers
    assert got[1]["launches"] == 3 and got[1]["alg_bytes"] < got[1]["l1_bytes"] < 0.5 * gathers
    assert got[0]["flops"] == got[1]["flops"]
    parts.close()
