"""retexo_pack_rows at the edges of its streaming kernel (16-byte pieces, 1 .. 32 lanes per row) and of the layouts it leaves to
the other kernel: rounding to bf16 is exact, so every value has to match."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("dim,pad", [(1, 7), (7, 1), (8, 0), (9, 7), (63, 1), (64, 0), (65, 3), (253, 3), (602, 6), (1031, 9)])
def test_pack_rows(dim, pad, bf16):
    """pad: the source's row stride is dim + pad elements (not a multiple of 4 or 8 in the later ones: the plain kernel)."""
    from paper_2302_13053_b200 import binding as B
    n = 77
    src = torch.randn((n, dim + pad), generator=torch.Generator().manual_seed(dim)).cuda()
    src = src.to(torch.bfloat16) if bf16 else src
    idx = torch.from_numpy(np.random.default_rng(dim).permutation(n)[:41].astype(np.int32)).cuda()
    for rows in (None, idx):
        for ones in (False, True):
            for multiple in (8, 64):
                got, _ = B.retexo_pack_rows(src, rows, dim=dim, ones=ones, ld_multiple=multiple)
                want = torch.zeros_like(got)
                want[:, :dim] = (src if rows is None else src[rows.long()])[:, :dim].to(torch.bfloat16)
                if ones:
                    want[:, dim] = 1.0
                assert torch.equal(got, want)
