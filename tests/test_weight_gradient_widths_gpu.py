"""The weight gradient on both sides of the widths that its own kernel takes,
which depend on the size of dA: the oracle's bits either way."""
import numpy as np
import pytest
import torch

import oracle
from paper_cs_0603115_gb300 import inputs

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_cs_0603115_gb300 as ff


# below 4e6 values, from there, from 6.5e7; few columns; even and odd rows
@pytest.mark.parametrize("m,n", [(1999, 2000), (2001, 2000), (2003, 1999), (8125, 8000), (8127, 8001), (66000, 1023),
                                 (66001, 1025)])
@pytest.mark.parametrize("k", [20, 21, 24, 25, 26, 27])
def test_bits(m, n, k):
    gen = torch.Generator(device="cuda").manual_seed(m + k)
    dY = inputs.to_ff(inputs.loguniform_f64(k * m, gen, "cuda")).view(k, m, 2)
    X = inputs.to_ff(inputs.loguniform_f64(k * n, gen, "cuda")).view(k, n, 2)
    dA = ff.gemv_dA(dY, X)
    rows = torch.tensor(sorted({0, 1, 3, m // 3, m // 2, m - 2, m - 1}))
    want = oracle.gemv_dA(np.ascontiguousarray(dY[:, rows.cuda()].cpu().numpy()), X.cpu().numpy())
    assert (dA[rows.cuda()].cpu().numpy().view("u4") == want.view("u4")).all()
    assert torch.isfinite(dA).all()
