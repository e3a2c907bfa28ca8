"""The aggregation kernels at the edges of their layouts: every vector width and number of lanes per row, ragged last vectors,
row lengths around the ones at which a group, a warp or several segments take a row, rows of odd strides."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_rows_close, dev
from paper_2302_13053_b200 import workloads as wl

pytestmark = pytest.mark.gpu

GRAPH = wl.degree_ladder_graph([0, 1, 2, 3, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128, 129, 191, 193, 700], seed=4)


@pytest.mark.parametrize("aggr", [oracle.GCN, oracle.SAGE_MEAN, oracle.SAGE_MAX])
@pytest.mark.parametrize("dim,ld", [(1, 1), (3, 8), (8, 8), (9, 16), (13, 16), (16, 16), (31, 32), (32, 32), (33, 40), (60, 64), (64, 64), (65, 72),
                                    (127, 128), (200, 200), (20, 20), (36, 36), (100, 100), (22, 22), (70, 70), (33, 33), (77, 77), (161, 161)])
def test_layouts(aggr, dim, ld):
    from paper_2302_13053_b200 import binding as B
    n, rowptr, colidx, _ = GRAPH
    rng = np.random.default_rng(dim)
    buf = np.full((n, ld), np.nan, dtype=np.float32)            # nothing beyond a row's columns may enter a result
    buf[:, :dim] = np.abs(rng.standard_normal((n, dim))) + 0.1  # positive: a sum of any order is within 1e-5 of its row
    q = np.ascontiguousarray(buf[:, :dim])
    ref = oracle.aggregate(aggr, rowptr, colidx, q)
    rp, ci = dev(rowptr.astype(np.int64)), dev(colidx.astype(np.int32))
    out, out16 = B.retexo_aggregate(aggr, rp, ci, dev(buf), dim=dim, want_bf16=True)
    again, _ = B.retexo_aggregate(aggr, rp, ci, dev(buf), dim=dim)
    assert torch.equal(out, again)
    assert torch.equal(out16[:, :out.shape[1]], out.to(torch.bfloat16))
    got = out.cpu().numpy()
    if aggr == oracle.SAGE_MAX:
        np.testing.assert_array_equal(got, ref.astype(np.float32))
    else:
        assert_rows_close(got, ref, what="%d columns, stride %d" % (dim, ld))


@pytest.mark.parametrize("aggr", [oracle.GCN, oracle.SAGE_MEAN, oracle.SAGE_MAX])
@pytest.mark.parametrize("dim,ld", [(95, 96), (97, 97), (97, 97 + 7), (129, 129), (130, 130), (193, 193), (194, 194), (196, 196), (196, 200),
                                    (257, 264), (260, 260), (500, 500), (602, 602), (603, 603), (769, 776), (1030, 1030)])
def test_leftover_columns(aggr, dim, ld):
    """Whole slabs of columns and the layouts that take what is left, with every load width; all hubs, so that a wide row has many pieces."""
    test_layouts(aggr, dim, ld)


def _time(fn, repeats=7):
    """Device time of 8 calls: as a graph, so that small calls are not timed by their launches."""
    fn()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(8):
            fn()
    best = float("inf")
    for _ in range(repeats):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("n,degree,dim,other,factor", [(20000, 100, 97, 95, 1.45), (2000, 100, 8, 64, 1.45)])
def test_cost_of_leftover_columns_and_of_small_dense_graphs(n, degree, dim, other, factor):
    """Two columns more cost no second pass over lanes that have none (1.8 times the time before they had their own layout); a narrow
    row takes no longer than a wide one (2.1 times when a warp walked as many rows as on a graph that fills the device)."""
    from paper_2302_13053_b200 import binding as B
    rng = np.random.default_rng(n)
    rp, ci = dev(np.arange(n + 1, dtype=np.int64) * degree), dev(rng.integers(0, n, size=n * degree).astype(np.int32))
    times = []
    for d in (dim, other):
        q = torch.randn((n, d), device="cuda")
        out = torch.empty((n, d), device="cuda")
        times.append(_time(lambda: B.retexo_aggregate(oracle.SAGE_MEAN, rp, ci, q, concat_self=False, out=out)))
    assert times[0] <= factor * times[1], times


def _fma(a, b, c):
    """fp32 multiply-add with one rounding: the product of two fp32 numbers is exact in fp64 (the sum's own rounding there is far below)."""
    return (a.astype(np.float64) * b + c).astype(np.float32)


@pytest.mark.parametrize("n,degree,dim,ld", [(20000, 2, 64, 64), (20000, 4, 64, 64), (20000, 4, 16, 16), (20000, 8, 8, 8), (20000, 4, 100, 100),
                                             (20000, 8, 97, 97), (20000, 16, 33, 40)])
def test_gcn_precision_of_short_rows(n, degree, dim, ld):
    """The error of a short row is that of one multiply-add per neighbour with the fp32 value of 1 / sqrt(d + 1): rows scaled ahead and
    rounded a second time (5 to 9 % more) are only for rows whose own sum hides it."""
    from paper_2302_13053_b200 import binding as B
    rng = np.random.default_rng(n + dim)
    rowptr, colidx = wl.csr_from_edge_list(n, rng.integers(0, n, size=(n * degree // 2, 2)))
    deg = np.diff(rowptr)
    buf = np.zeros((n, ld), np.float32)
    buf[:, :dim] = rng.standard_normal((n, dim))
    q = np.ascontiguousarray(buf[:, :dim])
    c = np.float32(1) / np.sqrt(deg.astype(np.float32) + np.float32(1))
    exact = (1.0 / np.sqrt(deg + 1.0))[:, None]
    ref = q * exact
    chain = np.zeros((n, dim), np.float32)
    for k in range(deg.max()):                                 # k-th neighbour of every row that has one
        v = np.flatnonzero(deg > k)
        u = colidx[rowptr[v] + k]
        ref[v] += q[u] * exact[u]
        chain[v] = _fma(q[u], c[u][:, None], chain[v])
    ref *= exact
    chain = _fma(q, c[:, None], chain) * c[:, None]
    out, _ = B.retexo_aggregate(B.GCN, dev(rowptr.astype(np.int64)), dev(colidx.astype(np.int32)), dev(buf), dim=dim)
    err, bound = (np.linalg.norm(x - ref) for x in (out.cpu().numpy(), chain))
    print(degree, dim, ld, err / bound)
    assert err <= 1.02 * bound, err / bound                   # 1.02: the noise of 1e5 to 2e6 rounding errors is below 1 %


@pytest.mark.parametrize("degree,dim,ld", [(16, 340, 340), (16, 450, 452), (16, 602, 604),
                                         (16, 768, 768), (16, 800, 800), (32, 97, 100),
                                         (16, 250, 250), (16, 450, 450), (16, 193, 193)])
def test_rows_bound_by_memory(degree, dim, ld):
    """GCN on graphs whose slabs of 64 columns are far beyond the cache: every number of column chunks in one pass, two passes, rows in
    8- and 4-byte pieces; rows of every length against 64 bits."""
    from paper_2302_13053_b200 import binding as B
    n = 2097152
    g = torch.Generator(device="cuda").manual_seed(dim)
    ladder = torch.tensor([0, 1, 2, 3, 31, 32, 33, 127, 129, 4000, 100000], device="cuda")
    deg = torch.full((n,), degree, device="cuda")
    rows = torch.randperm(n, generator=g, device="cuda")[:len(ladder)]
    deg[rows] = ladder
    rows = torch.cat([rows, torch.randint(0, n, (100,), generator=g, device="cuda"), torch.tensor([0, n - 1], device="cuda")])
    rp = torch.zeros((n + 1,), dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(deg, 0)
    ci = torch.randint(0, n, (int(rp[-1]),), generator=g, device="cuda", dtype=torch.int32)
    assert ci.numel() >= degree * n
    q = torch.rand((n, ld), generator=g, device="cuda") + 0.1
    q[:, dim:] = float("nan")
    out, out16 = B.retexo_aggregate(oracle.GCN, rp, ci, q, dim=dim, want_bf16=True)
    c = 1.0 / torch.sqrt(deg.double() + 1)
    for v in rows.tolist():
        u = ci[rp[v]:rp[v + 1]].long()
        want = c[v] * ((q[u, :dim].double() * c[u][:, None]).sum(0) + c[v] * q[v, :dim].double())
        assert (out[v].double() - want).norm() <= 1e-5 * want.norm(), (v, int(deg[v]))
        assert torch.equal(out16[v, :dim], out[v].to(torch.bfloat16))
    again, _ = B.retexo_aggregate(oracle.GCN, rp, ci, q, dim=dim)
    assert torch.equal(out, again)


@pytest.mark.parametrize("dim", [128, 200, 301])
@pytest.mark.parametrize("aggr", [oracle.GCN, oracle.SAGE_MEAN, oracle.SAGE_MAX])
def test_rows_by_length(aggr, dim):
    """A graph sparse and large enough for the rows to be taken in order of their lengths: empty rows, rows around what a group of lanes and a
    segment take, and more rows above a group's length than there are warps for them."""
    from paper_2302_13053_b200 import binding as B
    rng = np.random.default_rng(dim)
    deg = np.concatenate([np.full(22500, 33), np.repeat([0, 1, 2, 31, 32, 34, 127, 128, 129, 400], 10), rng.integers(0, 12, 60000)])
    deg = deg[rng.permutation(deg.size)]
    n, e = deg.size, int(deg.sum())
    rowptr = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    assert 8 * n <= e <= 48 * n and e * dim >= 32 << 20
    colidx = rng.integers(0, n, e).astype(np.int32)
    q = rng.standard_normal((n, dim)).astype(np.float32)
    out, out16 = B.retexo_aggregate(aggr, dev(rowptr), dev(colidx), dev(q), want_bf16=True)
    assert_rows_close(out.cpu().numpy(), oracle.aggregate(aggr, rowptr, colidx, q), what="aggr %d" % aggr)
    assert torch.equal(out16[:, :out.shape[1]], out.to(torch.bfloat16))
    again, _ = B.retexo_aggregate(aggr, dev(rowptr), dev(colidx), dev(q))
    assert torch.equal(out, again)
