"""The weight-gradient launch of the per-node model (both layers' [dW ; db] in one grid) at the edges of its tiles (128 x 64 /
128 / 256), of its 64-row steps and of its row ranges, against the same arithmetic in fp64 on operands rounded to bf16."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,hidden,n_classes,n", [(1, 1, 1, 1), (128, 0, 64, 64), (129, 0, 64, 65), (300, 0, 3, 9000), (64, 65, 1, 63),
                                                     (127, 128, 64, 129), (65, 129, 33, 200), (257, 256, 47, 4500),
                                                     (130, 257, 5, 700), (1030, 512, 41, 1500),
                                                     # two kernels an iteration up to 512 rows and 128 hidden units, and just beyond
                                                     (1433, 64, 7, 140), (63, 128, 41, 512), (200, 33, 17, 33), (64, 63, 8, 31), (1000, 128, 3, 60),
                                                     (2400, 100, 9, 300), (4400, 0, 40, 65), (64, 128, 9, 513), (128, 0, 64, 513), (129, 0, 64, 600),
                                                     (65, 64, 1, 600), (127, 128, 64, 700), (4481, 128, 3, 60)])
def test_gradients_at_the_edges(d_in, hidden, n_classes, n):
    from paper_2302_13053_b200 import binding as B
    rng = np.random.default_rng(1000 * d_in + hidden)
    out1 = hidden or n_classes
    bf = lambda t: t.to(torch.bfloat16).double()
    w1, b1 = rng.standard_normal((d_in, out1)) / np.sqrt(d_in), rng.standard_normal(out1) * 0.1
    w2, b2 = (rng.standard_normal((hidden, n_classes)) / np.sqrt(hidden), rng.standard_normal(n_classes) * 0.1) if hidden else (None, None)
    x = bf(torch.from_numpy(rng.standard_normal((n, d_in)).astype(np.float32)))
    y = torch.zeros(n, dtype=torch.int64)      # one label for all rows: the bias sums do not cancel, so a range left out shows
    gpu = B.Mlp(d_in, hidden, n_classes, w1, b1, w2, b2, optimizer=oracle.SGD, lr=0.1)
    x16, _ = B.retexo_pack_rows(dev(x.float().numpy()))
    _, gg = B.retexo_mlp_train_step(gpu, x16, dev(y.numpy().astype(np.int32)), return_grad=True)
    gg = gg.double().cpu()

    f32 = lambda v: torch.from_numpy(np.asarray(v, dtype=np.float32))
    z = x @ bf(f32(w1)) + f32(b1).double()
    logits, hd = z, None
    if hidden:
        hd = bf(z.clamp(min=0).float())
        logits = hd @ bf(f32(w2)) + f32(b2).double()
    dl = torch.softmax(logits, 1)
    dl[torch.arange(n), y] -= 1
    dl = bf((dl / n).float())
    parts = []      # (gradient, sum of its terms' magnitudes)
    if hidden:
        gate = (z > 0).double()
        w2r = bf(f32(w2))
        dhd = bf(((dl @ w2r.T) * gate).float())
        mag = (dl.abs() @ w2r.abs().T) * gate + dhd.abs()
        parts += [(x.T @ dhd, x.abs().T @ mag), (dhd.sum(0), mag.sum(0)), (hd.T @ dl, hd.abs().T @ dl.abs()), (dl.sum(0), dl.abs().sum(0))]
    else:
        parts += [(x.T @ dl, x.abs().T @ dl.abs()), (dl.sum(0), dl.abs().sum(0))]
    at = 0
    for ref, mag in parts:
        got = gg[at:at + ref.numel()].view_as(ref)
        at += ref.numel()
        err = (got - ref).abs()
        # fp32 logits within ~2^-20 of the fp64 ones move a dL, Hd or dHd over a rounding boundary now and then: by a bf16 step,
        # 2^-8 of that term, in each of two rounded factors
        assert (err <= 2.0 ** -7 * mag + 1e-12).all(), (err / mag.clamp(min=1e-30)).max()
        # such a term is one in ~2^10, so the typical entry's error is that of its fp32 sums: 2^-24 of the running sum per addition
        # of up to 2^8 ones in a row (16 rows an MMA, a range's rows, then the ranges)
        assert err.median() <= 2.0 ** -16 * mag.median() + 1e-12, (err.median(), mag.median())
    assert at == gg.numel() and int(gpu.status.item()) == 0
