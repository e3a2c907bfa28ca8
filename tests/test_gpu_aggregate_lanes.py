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
