"""The GAT kernels' lane layout at its edges: every number of lanes per entry (1 .. 32, 4 or 8 columns each), lanes without
columns, rows around the lengths at which a group, a warp or a block takes them, and rows the layout does not cover."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_rows_close, dev
from paper_2302_13053_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,dh,pad", [(1, 4, 0), (3, 4, 0), (8, 4, 0), (1, 8, 0), (3, 16, 0), (7, 8, 0), (1, 256, 0), (2, 128, 0), (5, 32, 8),
                                          (4, 16, 4)])
def test_gat_forward_and_backward(heads, dh, pad):
    """pad > 0: the rows have a stride of heads * dh + pad floats (4: in 16-byte pieces only, four columns a lane)."""
    from paper_2302_13053_b200 import binding as B
    n, rowptr, colidx, _ = wl.degree_ladder_graph([0, 1, 2, 3, 7, 8, 9, 30, 31, 32, 33, 61, 62, 63, 64, 65, 127, 129, 300], seed=heads)
    rng = np.random.default_rng(dh)
    d = heads * dh
    buf = rng.standard_normal((n, d + pad)).astype(np.float32)
    p = np.ascontiguousarray(buf[:, :d])
    dz = rng.standard_normal((n, d)).astype(np.float32)
    dz[rng.random(n) < 0.4] = 0.0
    scale = 1.0 / np.sqrt(dh)
    gat = dict(heads=heads, head_dim=dh, negative_slope=0.2, add_self_loop=1,
               a_src=(rng.standard_normal((heads, dh)) * scale).astype(np.float32),
               a_dst=(rng.standard_normal((heads, dh)) * scale).astype(np.float32))
    g = dict(gat, a_src=torch.from_numpy(gat["a_src"]), a_dst=torch.from_numpy(gat["a_dst"]))
    rp, ci = dev(rowptr.astype(np.int64)), dev(colidx.astype(np.int32))
    q = dev(buf)[:, :d]
    out, out16 = B.retexo_aggregate(B.GAT, rp, ci, q, gat=g, want_bf16=True)
    assert_rows_close(out.cpu().numpy(), oracle.aggregate(oracle.GAT, rowptr, colidx, p, gat=gat), what="%d x %d" % (heads, dh))
    assert torch.equal(out16[:, :d], out.to(torch.bfloat16))
    dp, dp16, da_src, da_dst = B.retexo_gat_backward(rp, ci, q, g, dev(dz), want_bf16=True)
    again = B.retexo_gat_backward(rp, ci, q, g, dev(dz))
    assert torch.equal(dp, again[0]) and torch.equal(da_src, again[2]) and torch.equal(da_dst, again[3])
    assert torch.equal(dp16[:, :d], dp.to(torch.bfloat16))
    ref_dp, ref_as, ref_ad = oracle.gat_backward(rowptr, colidx, p, gat, dz.astype(np.float64))
    # a row of up to 300 fp32 terms: 2e-5 of its norm, or of the largest gradient where its terms cancel
    err = np.abs(dp.cpu().numpy() - ref_dp).max(axis=1)
    assert np.all(err <= 2e-5 * np.linalg.norm(ref_dp, axis=1) + 1e-5 * np.abs(ref_dp).max()), float(err.max())
    for got, ref in ((da_src, ref_as), (da_dst, ref_ad)):      # sums over the n nodes, as in the other backward tests
        np.testing.assert_allclose(got.cpu().numpy(), ref, rtol=0, atol=2e-6 * max(1.0, np.abs(ref).max()) * np.sqrt(n))


@pytest.mark.parametrize("heads,dh", [(2, 8), (1, 32)])
def test_more_long_rows_than_warps_for_them(heads, dh):
    """24000 rows of 41 entries with the node itself, longer than a group takes: the grid has 21312 warps for such rows, the others share."""
    from paper_2302_13053_b200 import binding as B
    n, half, d = 24000, 20, heads * dh
    steps = np.concatenate([np.arange(-half, 0), np.arange(1, half + 1)])
    colidx = np.sort((np.arange(n)[:, None] + steps) % n, axis=1).astype(np.int32).ravel()
    rowptr = np.arange(n + 1, dtype=np.int64) * (2 * half)
    rng = np.random.default_rng(heads)
    p, dz = (rng.standard_normal((n, d)).astype(np.float32) for _ in range(2))
    dz[rng.random(n) < 0.4] = 0.0
    gat = dict(heads=heads, head_dim=dh, negative_slope=0.2, add_self_loop=1,
               a_src=(rng.standard_normal((heads, dh)) / np.sqrt(dh)).astype(np.float32),
               a_dst=(rng.standard_normal((heads, dh)) / np.sqrt(dh)).astype(np.float32))
    g = dict(gat, a_src=torch.from_numpy(gat["a_src"]), a_dst=torch.from_numpy(gat["a_dst"]))
    out, _ = B.retexo_aggregate(B.GAT, dev(rowptr), dev(colidx), dev(p), gat=g)
    assert_rows_close(out.cpu().numpy(), oracle.aggregate(oracle.GAT, rowptr, colidx, p, gat=gat))
    dp, _, _, _ = B.retexo_gat_backward(dev(rowptr), dev(colidx), dev(p), g, dev(dz))
    ref = oracle.gat_backward(rowptr, colidx, p, gat, dz.astype(np.float64))[0]
    err = np.abs(dp.cpu().numpy() - ref).max(axis=1)      # (as above)
    assert np.all(err <= 2e-5 * np.linalg.norm(ref, axis=1) + 1e-5 * np.abs(ref).max()), float(err.max())


@pytest.mark.parametrize("heads,dh,pad", [(4, 16, 0), (8, 4, 0), (1, 64, 0), (4, 16, 4), (2, 6, 0)])
@pytest.mark.parametrize("level", [4000.0, -4000.0])
def test_weights_of_large_scores(heads, dh, pad, level):
    """Scores of +-4000 with gaps of order 1, all exact in fp32 (multiples of 1 / 64, slope 1 / 4): what is left is the error of the
    weights, which may depend on the gap to the row's maximum but not on the scores' size."""
    from paper_2302_13053_b200 import binding as B
    n, rowptr, colidx, _ = wl.degree_ladder_graph([0, 1, 2, 3, 7, 31, 33, 63, 65, 129, 300], seed=heads)
    rng = np.random.default_rng(dh)
    d = heads * dh
    buf = rng.standard_normal((n, d + pad)).astype(np.float32)
    rows = buf[:, :d].reshape(n, heads, dh).copy()
    rows[..., 0] = np.round(rows[..., 0] * 64) / 64       # s_u
    rows[..., 1] = 1.0                                    # t_v = level
    buf[:, :d] = rows.reshape(n, d)
    p = np.ascontiguousarray(buf[:, :d])
    dz = rng.standard_normal((n, d)).astype(np.float32)
    gat = dict(heads=heads, head_dim=dh, negative_slope=0.25, add_self_loop=1, a_src=np.zeros((heads, dh), np.float32),
               a_dst=np.zeros((heads, dh), np.float32))
    gat["a_src"][:, 0] = 1.0
    gat["a_dst"][:, 1] = level
    g = dict(gat, a_src=torch.from_numpy(gat["a_src"]), a_dst=torch.from_numpy(gat["a_dst"]))
    rp, ci = dev(rowptr.astype(np.int64)), dev(colidx.astype(np.int32))
    dzb = torch.zeros((n, d + pad), device="cuda")
    dzb[:, :d] = dev(dz)
    out, _ = B.retexo_aggregate(B.GAT, rp, ci, dev(buf)[:, :d], gat=g)
    # a weight: 2^-22 of the exponential and as much of the product at gaps up to 8 (2.4e-7 each); rows of up to 300 terms that cancel to
    # a tenth of their size.  Half a unit in the last place of the scores on the exponent instead would be 1.7e-4.
    assert_rows_close(out.cpu().numpy(), oracle.aggregate(oracle.GAT, rowptr, colidx, p, gat=gat), rel=6e-6)
    dp, _, _, _ = B.retexo_gat_backward(rp, ci, dev(buf)[:, :d], g, dzb[:, :d])
    ref = oracle.gat_backward(rowptr, colidx, p, gat, dz.astype(np.float64))[0]
    # columns that neither attention vector reaches: sums of weighted gradients alone
    free = np.delete(np.arange(d).reshape(heads, dh), [0, 1], axis=1).ravel()
    assert_rows_close(dp.cpu().numpy()[:, free], ref[:, free], rel=6e-6)


@pytest.mark.parametrize("heads,dh", [(1, 8), (4, 16), (8, 4), (8, 32)])
def test_gradients_of_rows_with_a_common_part(heads, dh):
    """Rows around 20 and gradients around 1: <dz_v, p_u> and its mean over the row agree to one part in a hundred, and their difference is
    what reaches ds and dt.  Its error may be a few units in the last place of <dz_v, p_u> for every unit of attention a node
    receives (about ten for the node of 300 rows), not that of sums of the products themselves."""
    from paper_2302_13053_b200 import binding as B
    n, rowptr, colidx, _ = wl.degree_ladder_graph([1, 2, 3, 7, 15, 31, 32, 33, 63, 129, 300], seed=heads)
    rng = np.random.default_rng(dh)
    d = heads * dh
    p = (20 + rng.standard_normal((n, d))).astype(np.float32)
    dz = (1 + 0.1 * rng.standard_normal((n, d))).astype(np.float32)

    def vector():      # (mean zero: scores of order 1 although the rows are not)
        a = rng.standard_normal((heads, dh)) / np.sqrt(dh)
        return (a - a.mean(axis=1, keepdims=True)).astype(np.float32)
    gat = dict(heads=heads, head_dim=dh, negative_slope=0.2, add_self_loop=1, a_src=vector(), a_dst=vector())
    g = dict(gat, a_src=torch.from_numpy(gat["a_src"]), a_dst=torch.from_numpy(gat["a_dst"]))
    dp, _, _, _ = B.retexo_gat_backward(dev(rowptr.astype(np.int64)), dev(colidx.astype(np.int32)), dev(p), g, dev(dz))
    ref = oracle.gat_backward(rowptr, colidx, p, gat, dz.astype(np.float64))[0]
    size = 20.0 * dh                                        # of <dz_v, p_u>
    assert np.abs(dp.cpu().numpy() - ref).max() <= 20 * 2.0 ** -24 * size


def _time(fn, repeats=5):
    fn()
    best = float("inf")
    for _ in range(repeats):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("heads,dh,ld,offset", [(1, 8, 12, 0), (4, 16, 68, 0), (4, 16, 64, 4), (2, 32, 68, 0), (1, 64, 68, 0), (8, 8, 76, 4),
                                                (8, 4, 36, 0), (3, 16, 52, 4)])
def test_rows_in_16_byte_pieces(heads, dh, ld, offset):
    """Rows of up to 64 columns that start on 16-byte but not on 32-byte boundaries: the same results, and no more than a few times
    the time of rows that do (the general kernels take ten to thirty times as long)."""
    from paper_2302_13053_b200 import binding as B
    n, rowptr, colidx, _ = wl.degree_ladder_graph([1, 5, 31, 33, 64, 200, 400], seed=heads)
    rng = np.random.default_rng(dh + ld)
    d = heads * dh
    scale = 1.0 / np.sqrt(dh)
    gat = dict(heads=heads, head_dim=dh, negative_slope=0.2, add_self_loop=1,
               a_src=(rng.standard_normal((heads, dh)) * scale).astype(np.float32),
               a_dst=(rng.standard_normal((heads, dh)) * scale).astype(np.float32))
    g = dict(gat, a_src=torch.from_numpy(gat["a_src"]), a_dst=torch.from_numpy(gat["a_dst"]))
    rp, ci = dev(rowptr.astype(np.int64)), dev(colidx.astype(np.int32))

    def laid_out(a):
        rows = torch.full((offset + n * ld,), float("nan"), device="cuda")[offset:].view(n, ld)
        rows[:, :d] = dev(a)
        return rows[:, :d]
    p, dz = rng.standard_normal((n, d)).astype(np.float32), rng.standard_normal((n, d)).astype(np.float32)
    dz[rng.random(n) < 0.4] = 0.0
    q, gz = laid_out(p), laid_out(dz)
    out, _ = B.retexo_aggregate(B.GAT, rp, ci, q, gat=g)
    assert_rows_close(out.cpu().numpy(), oracle.aggregate(oracle.GAT, rowptr, colidx, p, gat=gat), what="%d x %d" % (heads, dh))
    dp, _, da_src, da_dst = B.retexo_gat_backward(rp, ci, q, g, gz)
    ref_dp, ref_as, ref_ad = oracle.gat_backward(rowptr, colidx, p, gat, dz.astype(np.float64))
    err = np.abs(dp.cpu().numpy() - ref_dp).max(axis=1)      # as for aligned rows above
    assert np.all(err <= 2e-5 * np.linalg.norm(ref_dp, axis=1) + 1e-5 * np.abs(ref_dp).max()), float(err.max())
    for got, ref in ((da_src, ref_as), (da_dst, ref_ad)):
        np.testing.assert_allclose(got.cpu().numpy(), ref, rtol=0, atol=2e-6 * max(1.0, np.abs(ref).max()) * np.sqrt(n))
    if dh >= 8:
        m = 20000                                            # a graph large enough to be bound by its entries: 200 a row
        step = torch.arange(1, 201, device="cuda", dtype=torch.int64) * 37
        cols = ((torch.arange(m, device="cuda")[:, None] + step) % m).sort(1).values
        rp2, ci2 = torch.arange(m + 1, device="cuda") * 200, cols.to(torch.int32).flatten().contiguous()
        base = torch.randn(m * 80 + 64, device="cuda")
        odd, even = base[offset:offset + m * ld].view(m, ld)[:, :d], base[:m * d].view(m, d)
        slow = _time(lambda: B.retexo_gat_backward(rp2, ci2, odd, g, odd))
        fast = _time(lambda: B.retexo_gat_backward(rp2, ci2, even, g, even))
        assert slow < 4 * fast, (slow, fast)
