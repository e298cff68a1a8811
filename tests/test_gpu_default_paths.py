"""The kernels that run when a call names no program parameters, at the sizes where
each can go wrong: edges of tiles, remainders, strides and bases that rule wide accesses
out, the smallest and largest of a rule's range."""
import numpy as np
import pytest
import torch

from paper_1801_04348_gb300 import pgk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    import __graft_entry__
    __graft_entry__.build()
    d = torch.device("cuda:0")
    torch.cuda.set_device(d)
    return d


@pytest.mark.parametrize("rows,cols", [(1, 1), (64, 64), (65, 63), (3, 200), (200, 3), (130, 66), (1000, 777)])
@pytest.mark.parametrize("pad_s,pad_d,shift", [(0, 0, 0), (4, 4, 0), (3, 0, 0), (0, 5, 0), (4, 4, 1)])
def test_transpose_without_parameters(dev, rows, cols, pad_s, pad_d, shift):
    """Row strides rounded up to 16 bytes plus a pad (0 and 4 keep 128-bit accesses, 3, 5
    and a base moved by one word rule them out): exact, and nothing outside is written."""
    lds, ldd = (cols + 3) // 4 * 4 + pad_s, (rows + 3) // 4 * 4 + pad_d
    s = torch.randint(-2 ** 31, 2 ** 31 - 1, (rows * lds + shift,), device=dev, dtype=torch.int32)
    d = torch.full((cols * ldd + shift,), -7, device=dev, dtype=torch.int32)
    src, dst = s[shift:].view(rows, lds)[:, :cols], d[shift:].view(cols, ldd)
    pgk.transpose(src, dst[:, :rows])
    assert torch.equal(dst[:, :rows], src.t())
    assert (dst[:, rows:] == -7).all() and (d[:shift] == -7).all()
