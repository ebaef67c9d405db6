"""Products that underflow, whose low parts come out as -0 in the Fast2Sum form
and as +0 in the theorem's: no stored result shows it, for sums of one term and
of several, by any kernel that uses the form."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import replay

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_cs_0603115_gb300 as ff
    from paper_cs_0603115_gb300 import _lib, batch

U = 2.0 ** -12
VALUES = np.array([(s * h, t * l) for h, l in ((2.0 ** -100, 2.0 ** -130), (2.0 ** -80, 2.0 ** -106), (2.0 ** -100, 0.0), (0.0, 0.0),
                                               ((1 + U) * 2.0 ** -60, 0.0), ((1 + U) * 2.0 ** -75, 0.0), (2.0 ** -149, 0.0), (1.0, 2.0 ** -30))
                   for s in (1, -1) for t in (1, -1)], np.float32)


def operand(*shape, seed):
    rng = np.random.default_rng(seed)
    return VALUES[rng.integers(0, len(VALUES), shape)]


def same(got, want):
    assert (np.ascontiguousarray(got).view("u4") == np.ascontiguousarray(want).view("u4")).all()


@pytest.mark.parametrize("k", [1, 2, 3, 13, 21])
@pytest.mark.parametrize("m,n", [(64, 64), (65, 67), (300, 130)])
def test_weight_gradient_and_product(m, n, k):
    dY, X = operand(k, m, seed=k), operand(k, n, seed=k + 1)
    want = oracle.gemv_dA(dY, X)
    d, x = torch.from_numpy(dY).cuda(), torch.from_numpy(X).cuda()
    same(ff.gemv_dA(d, x).cpu().numpy(), want)
    same(ff.gemm(d, x, transa=True).cpu().numpy(), want)


@pytest.mark.parametrize("k", [1, 2, 5])
@pytest.mark.parametrize("m,n", [(33, 1), (40, 2), (12, 65), (1, 300), (2, 301), (70, 128)])
def test_gemv_and_adjoint(m, n, k):
    A, X, dY = operand(m, n, seed=m), operand(k, n, seed=n + 1), operand(k, m, seed=m + 2)
    a = torch.from_numpy(A).cuda()
    same(ff.gemv(a, torch.from_numpy(X).cuda()).cpu().numpy(), replay.gemv_warp_replay(A, X, vec=n % 2 == 0))
    nrb, vec = ctypes.c_int64(), ctypes.c_int()
    _lib.call("ff_gemv_t_launch_shape", a.data_ptr(), m, n, n, k, ctypes.byref(nrb), ctypes.byref(vec))
    same(ff.gemv_t(a, torch.from_numpy(dY).cuda()).cpu().numpy(), replay.gemv_t_replay(A, dY, nrb.value))


@pytest.mark.parametrize("m,n", [(9, 1), (40, 2), (33, 64), (7, 129)])
def test_batched_rows(m, n):
    A, x = operand(m, n, seed=m), operand(n, seed=n + 1)
    y = torch.full((m, 2), float("nan"), device="cuda")
    a, xd = torch.from_numpy(A).cuda(), torch.from_numpy(x).cuda()
    plan = batch.BatchPlan(batch.make_instances([(batch.GEMV, a, xd, y, None)]))
    plan.run()
    same(y.cpu().numpy(), replay.gemv_rows8_replay(A, x, n % 2 == 0))
    plan.close()
