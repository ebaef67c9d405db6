"""ff_gemv on matrices of many rows, whose kernel is chosen by the length of the
rows, the number of rows and the access width: rows at both ends and between,
bit for bit against the replay of the documented order, and next to one another
on either side of each line."""
import pytest
import torch

import replay
from paper_cs_0603115_gb300 import inputs

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_cs_0603115_gb300 as ff

QUARTERS = 4 * (torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152)


def check(m, n, k, law, offset=0):
    if law == "any pairs":
        g = torch.Generator(device="cuda").manual_seed(m + n + k)
        A0, X = torch.randn(m, n, 2, generator=g, device="cuda"), torch.randn(k, n, 2, generator=g, device="cuda")
    else:
        gen = torch.Generator(device="cuda").manual_seed(m + n + k)
        A0 = inputs.to_ff(inputs.loguniform_f64(m * n, gen, "cuda")).view(m, n, 2)
        X = inputs.to_ff(inputs.loguniform_f64(k * n, gen, "cuda")).view(k, n, 2)
    buf = torch.empty(m * n + 1, 2, device="cuda")
    A = buf[offset:offset + m * n].view(m, n, 2)
    A.copy_(A0)
    Y = ff.gemv(A, X)
    rows = torch.cat([torch.arange(0, min(m, 40)), torch.arange(m // 2, m // 2 + 9), torch.arange(max(m - 40, 0), m)]).unique()
    got = Y[:, rows.cuda()].cpu().numpy()
    want = replay.gemv_warp_replay(A0[rows.cuda()].cpu().numpy(), X.cpu().numpy(), vec=n % 2 == 0 and offset == 0)
    assert (got.view("u4") == want.view("u4")).all()
    assert torch.isfinite(Y).all() and (Y[:, :, 0] != 0).any(dim=1).all()


@pytest.mark.parametrize("law", ["float-float", "any pairs"])
@pytest.mark.parametrize("k", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 65, 127, 128, 129, 130])
def test_short_rows(n, k, law):
    check(16 * QUARTERS + 3, n, k, law)


@pytest.mark.parametrize("law", ["float-float", "any pairs"])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 7])
@pytest.mark.parametrize("n", [129, 255, 256, 257])
def test_short_rows_of_very_many(n, k, law):
    check(64 * QUARTERS + 5, n, k, law)


@pytest.mark.parametrize("m", [8 * QUARTERS, 8 * QUARTERS + 1, 12 * QUARTERS, 12 * QUARTERS + 1, 16 * QUARTERS - 1, 24 * QUARTERS])
@pytest.mark.parametrize("n", [128, 130, 400, 402, 2048, 2050])
def test_one_vector(m, n):
    check(m, n, 1, "float-float")


@pytest.mark.parametrize("n,k", [(128, 1), (64, 3), (256, 2)])
def test_eight_byte_access(n, k):
    check(64 * QUARTERS, n, k, "float-float", offset=1)
