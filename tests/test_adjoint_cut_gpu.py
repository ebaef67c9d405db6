"""The row blocks that the GEMV adjoint is cut into: the chain of additions
behind one result (rows of a block plus blocks) stays within its limit, and the
sums follow the cut bit for bit."""
import ctypes
import math

import pytest
import torch

import replay
from paper_cs_0603115_gb300 import inputs

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_cs_0603115_gb300 as ff
    from paper_cs_0603115_gb300 import _lib


def cut(m, n, k, offset=0):
    """(row blocks, rows of a block, 16-byte access) for a matrix `offset` values past a 16-byte boundary."""
    nrb, vec = ctypes.c_int64(), ctypes.c_int()
    _lib.call("ff_gemv_t_launch_shape", 4096 + 8 * offset, m, n, n, k, ctypes.byref(nrb), ctypes.byref(vec))
    return nrb.value, -(-m // nrb.value), bool(vec.value)


def longest_chain(m):
    """A tenth above the chain with row blocks of at least 32 rows, at most 64 of them."""
    blocks = min(max(m // 32, 1), 64)
    return 1.1 * (blocks + -(-m // blocks))


# tall, wide, square and ragged; the first two were cut into a quarter of these blocks by time alone
SHAPES = [(1035, 4196, 13), (4096, 16384, 64), (64, 16384, 1), (100, 9001, 5), (700, 9001, 2), (2001, 3001, 5),
          (12001, 12001, 1), (16384, 64, 7), (8191, 300, 16), (65600, 2048, 3), (33, 1000, 64), (1, 5000, 2)]


@pytest.mark.parametrize("m,n,k", SHAPES)
@pytest.mark.parametrize("offset", [0, 1])
def test_chain_stays_short(m, n, k, offset):
    nrb, rows, _ = cut(m, n, k, offset)
    assert (nrb - 1) * rows < m <= nrb * rows
    assert nrb + rows <= longest_chain(m)


def test_chain_stays_short_over_the_range():
    import random
    rng = random.Random(5)
    for _ in range(2000):
        m, n, k = (round(math.exp(rng.uniform(math.log(a), math.log(b)))) for a, b in ((1, 70000), (1, 40000), (1, 64)))
        nrb, rows, _ = cut(m, n, k)
        assert nrb + rows <= longest_chain(m), (m, n, k)


@pytest.mark.parametrize("m,n,k", [(1035, 196, 13), (1035, 4196, 2), (700, 901, 2)])
def test_sums_follow_the_cut(m, n, k):
    gi = inputs.gemv(m, n, k, inputs.seed_for(4, 200 + k))
    nrb, _, vec = cut(m, n, k)
    assert vec == (n % 2 == 0)
    dX = ff.gemv_t(gi.A.cuda(), gi.dY.cuda()).cpu().numpy()
    want = replay.gemv_t_replay(gi.A.numpy(), gi.dY.numpy(), nrb)
    assert (dX.view("u4") == want.view("u4")).all()


@pytest.mark.parametrize("m,n,k", [(8, 1000000, 5), (12, 100001, 5), (16, 1000001, 2), (24, 200000, 16), (32, 200001, 5)])
def test_wide_matrices_are_cut_into_few_row_blocks(m, n, k):
    """The columns alone fill the device: one row block (4 to 16 before, at half the rate and less)."""
    assert cut(m, n, k)[0] == 1


@pytest.mark.parametrize("m,n,k", [(12, 100001, 3), (5, 70001, 4), (48, 16001, 5), (100, 20000, 2), (2, 200001, 1)])
@pytest.mark.parametrize("offset", [0, 1])
def test_sums_of_wide_matrices(m, n, k, offset):
    gi = inputs.gemv(m, n, k, inputs.seed_for(4, 300 + k))
    buf = torch.empty(m * n + 2, 2, device="cuda")
    A = buf[offset:offset + m * n].view(m, n, 2)
    A.copy_(gi.A)
    nrb, _, vec = cut(m, n, k, offset)
    assert vec == (n % 2 == 0 and offset == 0)
    dX = ff.gemv_t(A, gi.dY.cuda()).cpu().numpy()
    want = replay.gemv_t_replay(gi.A.numpy(), gi.dY.numpy(), nrb)
    assert (dX.view("u4") == want.view("u4")).all()


def test_host_time_does_not_depend_on_recent_sizes():
    """Forty sizes in turn cost a call no more host time than one size again and again (4 us more when a
    thread's plans held eight sizes)."""
    import time
    lib = _lib.load()
    shapes = [(1000 + 211 * i, 3001 + 97 * i, 1 + i % 16) for i in range(40)]

    def per_call(turn):
        best = 1.0
        for _ in range(7):
            t = time.perf_counter()
            for _ in range(10):
                for m, n, k in turn:
                    lib.ff_gemv_t_workspace_bytes(m, n, k)
            best = min(best, (time.perf_counter() - t) / (10 * len(turn)))
        return best

    assert per_call(shapes) < per_call(shapes[:1] * 40) + 1e-6


@pytest.mark.parametrize("m,n", [(1, 1), (1, 2), (1, 513), (2, 1000), (3, 257), (3, 10001), (2, 60002), (3, 2), (1, 200001)])
@pytest.mark.parametrize("k", [1, 2, 3, 5, 9])
@pytest.mark.parametrize("law", ["float-float", "any pairs"])
def test_sums_of_few_rows(m, n, k, law):
    """Row blocks of one to three rows, with operands that are normalised and that are not."""
    if law == "any pairs":
        g = torch.Generator().manual_seed(m + n + k)
        A, dY = torch.randn(m, n, 2, generator=g), torch.randn(k, m, 2, generator=g)
    else:
        gi = inputs.gemv(m, n, k, inputs.seed_for(4, 400 + k))
        A, dY = gi.A, gi.dY
    nrb, rows, _ = cut(m, n, k)
    assert rows <= 3
    dX = ff.gemv_t(A.cuda(), dY.cuda()).cpu().numpy()
    want = replay.gemv_t_replay(A.numpy(), dY.numpy(), nrb)
    assert (dX.view("u4") == want.view("u4")).all()
