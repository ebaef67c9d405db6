"""The GEMV adjoint where its row blocks go through the workspace and a second
launch adds them: every access width with every width of right-hand-side tile
(narrow, one wide tile, several, mixed), operands that are normalised and not,
and calls in a row that reuse the workspace."""
import ctypes

import pytest
import torch

import replay
from paper_cs_0603115_gb300 import inputs

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_cs_0603115_gb300 as ff
    from paper_cs_0603115_gb300 import _lib

# 16-byte access; single columns; two columns apart: k = 1, many narrow tiles, one tile of two, three and
# two, twice three, fours and threes, fours
SHAPES = [(2828, 4882, 1), (5419, 490, 10), (6000, 3672, 2), (6251, 2034, 5), (6265, 2012, 6), (5822, 742, 18), (6574, 736, 20),
          (689, 19831, 1), (9309, 125, 20), (9516, 1915, 2), (13088, 635, 5), (12889, 609, 6), (6563, 377, 18), (9029, 251, 20),
          (17316, 3697, 1), (1382, 3713, 13), (3373, 9489, 2), (7020, 1833, 5), (6629, 1893, 6), (2370, 1531, 19), (4986, 1263, 12)]


def two_launches(A, dY, out):
    """True when this call cannot run without a workspace."""
    k, m = dY.shape[:2]
    n = A.shape[1]
    st = _lib.load().ff_gemv_t(A.data_ptr(), m, n, n, dY.data_ptr(), m, k, out.data_ptr(), n, None, 0,
                               torch.cuda.current_stream().cuda_stream)
    assert st in (0, 2)
    return st == 2


def operands(m, n, k, law):
    gen = torch.Generator(device="cuda").manual_seed(m + n + k)
    if law == "any pairs":
        return torch.randn(m, n, 2, generator=gen, device="cuda"), torch.randn(k, m, 2, generator=gen, device="cuda")
    return (inputs.to_ff(inputs.loguniform_f64(m * n, gen, "cuda")).view(m, n, 2),
            inputs.to_ff(inputs.loguniform_f64(k * m, gen, "cuda")).view(k, m, 2))


@pytest.mark.parametrize("law", ["float-float", "any pairs"])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_sums(m, n, k, law):
    A, dY = operands(m, n, k, law)
    nrb, vec = ctypes.c_int64(), ctypes.c_int()
    _lib.call("ff_gemv_t_launch_shape", A.data_ptr(), m, n, n, k, ctypes.byref(nrb), ctypes.byref(vec))
    assert bool(vec.value) == (n % 2 == 0)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:   # the sizes were picked for this many
        assert two_launches(A, dY, torch.empty(k, n, 2, device="cuda"))
    dX = ff.gemv_t(A, dY)
    cols = torch.tensor(sorted({0, 1, n // 2, n - 130, n - 2, n - 1}))
    got = dX[:, cols.cuda()].cpu().numpy()
    want = replay.gemv_t_replay(A[:, cols.cuda()].cpu().numpy(), dY.cpu().numpy(), nrb.value)
    assert (got.view("u4") == want.view("u4")).all()
    assert torch.isfinite(dX).all()


@pytest.mark.parametrize("m,n,k", [(5419, 490, 10), (6563, 377, 18), (1382, 3713, 13)])
def test_calls_in_a_row(m, n, k):
    """Each adjoint reads what the product before it made of the last one; one workspace serves them all."""
    A, dY = operands(m, n, k, "float-float")
    scale = lambda t: t * torch.exp2(-torch.ceil(torch.log2(t.abs().amax())))   # noqa: E731
    A = scale(A)

    def chain(step):
        d, out = scale(dY).clone(), []
        dX, Y = torch.empty(k, n, 2, device="cuda"), torch.empty(k, m, 2, device="cuda")
        for _ in range(4):
            step()
            ff.gemv_t(A, d, dX)
            step()
            ff.gemv_t(A, d, dX)          # the same again, over the first one's partial sums
            step()
            out.append(dX.clone())
            ff.gemv(A, dX, Y)
            step()
            d = scale(Y).clone()
        return torch.stack(out)

    want = chain(torch.cuda.synchronize)
    for s in (torch.cuda.current_stream(), torch.cuda.Stream()):
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            got = [chain(lambda: None) for _ in range(3)]
        torch.cuda.synchronize()
        for g in got:
            assert torch.equal(g.view(torch.int32), want.view(torch.int32))
