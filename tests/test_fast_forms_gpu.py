"""The Fast2Sum forms of the products and the paths around them: every result
has the bits of the full Mul22 / Add22 sequence (the oracle's, in the
documented order), for normalised operands, for pairs whose sum does not round
to the high part (they leave the fast path), for sums that overflow to an
infinity at any point, and for infinities, NaN, signed zeros and subnormals;
at the edges of every tile shape."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import replay
from paper_cs_0603115_gb300 import inputs

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_cs_0603115_gb300 as ff
    from paper_cs_0603115_gb300 import _lib

DEV = "cuda"


def same_bits(got, want):
    got = np.ascontiguousarray(got, np.float32)
    want = np.ascontiguousarray(want, np.float32)
    assert got.shape == want.shape
    nan = np.isnan(got) & np.isnan(want)
    eq = (got.view(np.uint32) == want.view(np.uint32)) | nan
    if not eq.all():
        bad = np.argwhere(~eq)[:5]
        raise AssertionError(f"{(~eq).sum()} mismatches, first at {bad.tolist()}: "
                             f"got {got[tuple(bad[0])]} want {want[tuple(bad[0])]}")


def plant(v, kind, seed):
    """Special pairs at random places of a (..., 2) array (a copy)."""
    v = v.clone()
    f = v.reshape(-1, 2)
    g = torch.Generator().manual_seed(seed)
    at = torch.randperm(f.shape[0], generator=g)[:max(1, f.shape[0] // 50)]
    if kind == "unnormalised":
        f[at, 1] = f[at, 0] * 0.75
    elif kind == "swapped":          # |lo| > |hi|
        f[at] = f[at].flip(1)
    elif kind == "overflow":         # products and sums around the largest binary32
        f[at, 0] = torch.sign(f[at, 0]) * 1.8446744e19
        f[at, 1] = f[at, 0] * 2.0 ** -25
    elif kind == "specials":
        vals = torch.tensor([[float("inf"), 0.0], [float("nan"), 0.0], [-0.0, 0.0], [0.0, -0.0], [1e-40, 0.0],
                             [-3e-39, 1e-45], [float("-inf"), 1.0], [0.0, 1e-45]])
        f[at] = vals[torch.arange(at.numel()) % vals.shape[0]]
    return f.reshape(v.shape)


KINDS = ["plain", "unnormalised", "swapped", "overflow", "specials"]


# one shape for each tile shape of the dispatch (8x16, 16x16, 32x32, 64x64
# outputs), each ragged in both directions and in the inner index
@pytest.mark.parametrize("m,n,k", [(33, 65, 70), (250, 255, 49), (1020, 1023, 33), (1209, 1021, 19)])
@pytest.mark.parametrize("kind", KINDS)
def test_gemm_tiles(m, n, k, kind):
    g = inputs.gemm(m, n, k, inputs.seed_for(6, 60))
    A, B = plant(g.A, kind, 1), plant(g.B, kind, 2)
    At, Bt = A.permute(1, 0, 2).contiguous(), B.permute(1, 0, 2).contiguous()
    want = oracle.gemm(A.numpy(), B.numpy())
    for ta in (False, True):
        for tb in (False, True):
            got = ff.gemm((At if ta else A).to(DEV), (Bt if tb else B).to(DEV), transa=ta, transb=tb)
            same_bits(got.cpu().numpy(), want)


# inner lengths around a whole slice of the two small tiles and of a group of
# its steps, for each operand layout; one value off the fast forms in the first
# slice only, so that later slices switch back
@pytest.mark.parametrize("m,n", [(33, 65), (250, 255)])
@pytest.mark.parametrize("k", [1, 7, 63, 64, 65, 72, 127, 129, 200])
def test_gemm_slices(m, n, k):
    g = inputs.gemm(m, n, k, inputs.seed_for(6, 61))
    A, B = g.A.clone(), g.B
    A[m // 2, 0, 1] = A[m // 2, 0, 0]
    At, Bt = A.permute(1, 0, 2).contiguous(), B.permute(1, 0, 2).contiguous()
    want = oracle.gemm(A.numpy(), B.numpy())
    for ta in (False, True):
        for tb in (False, True):
            got = ff.gemm((At if ta else A).to(DEV), (Bt if tb else B).to(DEV), transa=ta, transb=tb)
            same_bits(got.cpu().numpy(), want)


# one warp per row and right-hand side (few rows), pairs, and tiles of 2, 3 + 2,
# 3, 4 and 4 + 3; row lengths around the loads in flight, even and odd
FORWARD = [(40, 1100, 1), (40, 515, 3), (700, 130, 4), (700, 67, 3), (650, 70, 9), (1300, 66, 2), (1300, 33, 3), (1230, 131, 5),
           (1230, 34, 6), (700, 260, 7), (620, 36, 8)]


@pytest.mark.parametrize("m,n,k", FORWARD)
@pytest.mark.parametrize("kind", KINDS)
def test_gemv_tiles(m, n, k, kind):
    g = inputs.gemv(m, n, k, inputs.seed_for(4, 200))
    A, X = plant(g.A, kind, 3), plant(g.X, kind, 4)
    Y = ff.gemv(A.to(DEV), X.to(DEV)).cpu().numpy()
    rows = np.unique(np.r_[0:8, m // 2:m // 2 + 8, m - 8:m])
    want = replay.gemv_warp_replay(A.numpy()[rows], X.numpy(), vec=n % 2 == 0)
    same_bits(Y[:, rows], want)


# one to a few rows, blocks of 2 to 128 column groups with their row blocks
# combined in shared memory, and two launches; narrow and wide tiles
ADJOINT = [(1, 9, 2), (2, 300, 1), (7, 64, 5), (33, 2050, 3), (300, 1000, 1), (300, 1001, 4), (1001, 128, 7), (3000, 40, 9),
           (5003, 37, 2), (4001, 4999, 1), (2100, 4096, 16)]


@pytest.mark.parametrize("m,n,k", ADJOINT)
@pytest.mark.parametrize("kind", KINDS)
def test_gemv_t_cuts(m, n, k, kind):
    g = inputs.gemv(m, n, k, inputs.seed_for(4, 201))
    A, dY = plant(g.A, kind, 5), plant(g.dY, kind, 6)
    Ad, dYd = A.to(DEV), dY.to(DEV)
    nrb, vec = ctypes.c_int64(), ctypes.c_int()
    _lib.call("ff_gemv_t_launch_shape", Ad.data_ptr(), m, n, n, k, ctypes.byref(nrb), ctypes.byref(vec))
    dX = ff.gemv_t(Ad, dYd).cpu().numpy()
    cols = np.unique(np.r_[0:min(4, n), n // 2, max(n - 4, 0):n])
    want = replay.gemv_t_replay(A.numpy()[:, cols], dY.numpy(), nrb.value)
    same_bits(dX[:, cols], want)


# two columns per thread, `apart` from one another: odd rows, an even row length
# on an 8-byte address (shift 1), every width of right-hand-side tile, the last
# columns without a partner
@pytest.mark.parametrize("m,n,k,shift", [(1009, 2003, 33, 0), (300, 214001, 1, 0), (640, 50001, 2, 0), (701, 18301, 5, 0),
                                         (702, 18300, 5, 1), (2401, 1027, 27, 0), (60, 270001, 4, 0)])
@pytest.mark.parametrize("kind", ["plain", "unnormalised", "specials"])
def test_gemv_t_columns_apart(m, n, k, shift, kind):
    gen = torch.Generator(device=DEV).manual_seed(11)
    store = torch.zeros(m * n + shift, 2, device=DEV)
    A = store[shift:].view(m, n, 2)
    A.copy_(inputs.to_ff(inputs.loguniform_f64(m * n, gen, DEV)).view(m, n, 2))
    dY = inputs.to_ff(inputs.loguniform_f64(k * m, gen, DEV)).view(k, m, 2)
    dY = plant(dY.cpu(), "plain" if kind == "specials" else kind, 6).to(DEV)
    cols = np.unique(np.r_[0:4, 127:131, 255:259, n // 2:n // 2 + 3, n - 260:n - 254, n - 4:n])
    if kind != "plain":
        A[m // 3, cols[::2], 1] = A[m // 3, cols[::2], 0] * 0.75
    if kind == "specials":
        A[m // 2, int(cols[1]), 0] = float("inf")
        A[m - 1, int(cols[3]), 0] = float("nan")
        A[0, int(cols[5])] = torch.tensor([-0.0, 0.0], device=DEV)
    nrb, vec = ctypes.c_int64(), ctypes.c_int()
    _lib.call("ff_gemv_t_launch_shape", A.data_ptr(), m, n, n, k, ctypes.byref(nrb), ctypes.byref(vec))
    assert vec.value == 0
    dX = ff.gemv_t(A, dY).cpu().numpy()
    want = replay.gemv_t_replay(A[:, cols].cpu().numpy(), dY.cpu().numpy(), nrb.value)
    same_bits(dX[:, cols], want)


# one pass, the widest single pass, two passes, the matrix-product route; even
# and odd rows of dA; rows around the steps and the staged chunks
@pytest.mark.parametrize("m,n,k", [(5, 6, 1), (131, 7, 1), (261, 514, 2), (129, 515, 5), (66, 36, 12), (67, 35, 13), (133, 130, 20),
                                   (130, 131, 21), (40, 41, 25)])
@pytest.mark.parametrize("kind", KINDS)
def test_gemv_dA_passes(m, n, k, kind):
    g = inputs.gemv(m, n, k, inputs.seed_for(4, 202))
    X, dY = plant(g.X, kind, 7), plant(g.dY, kind, 8)
    dA = ff.gemv_dA(dY.to(DEV), X.to(DEV)).cpu().numpy()
    same_bits(dA, oracle.gemv_dA(dY.numpy(), X.numpy()))


# rows around the chunks in flight (16- and 8-byte access), few and many tiles
@pytest.mark.parametrize("shapes", [[(9, 5)], [(40, 70), (33, 131), (5, 600), (7, 1025)], [(3000, 66), (2500, 67), (900, 258)]])
@pytest.mark.parametrize("kind", KINDS)
def test_batch_gemv_rows(shapes, kind):
    from paper_cs_0603115_gb300 import batch
    specs, want = [], []
    for i, (m, n) in enumerate(shapes):
        g = inputs.gemv(m, n, 1, inputs.seed_for(4, 203 + i))
        A, x = plant(g.A, kind, 9 + i), plant(g.X[0], kind, 19 + i)
        out = torch.full((m, 2), float("nan"), device=DEV)
        specs.append((batch.GEMV, A.to(DEV), x.to(DEV), out, None))
        rows = np.unique(np.r_[0:min(m, 40), m // 2, max(m - 9, 0):m])
        want.append((rows, replay.gemv_rows8_replay(A.numpy()[rows], x.numpy(), n % 2 == 0)))
    plan = batch.BatchPlan(batch.make_instances(specs))
    for _ in range(2):
        plan.run()
        for (_, _, _, out, _), (rows, w) in zip(specs, want):
            same_bits(out.cpu().numpy()[rows], w)
            out.fill_(float("nan"))
    plan.close()


# weight gradients whose grid takes several waves of blocks, ragged in rows and
# columns, pairs of columns and single ones; chunks of few rows; and either side
# of the widest k that a large matrix takes without the matrix product
@pytest.mark.parametrize("m,n,k", [(9, 200000, 2), (1003, 130001, 1), (301, 70000, 13), (77, 131072, 3),
                                   (1, 33, 20), (5, 300, 6), (9, 515, 12), (131, 40, 7), (129, 6000, 20),
                                   (2049, 131077, 21), (2049, 131078, 28), (2049, 131072, 29)])
def test_weight_gradient_waves(m, n, k):
    dY, X = inputs.to_ff(inputs.loguniform_f64(k * m, torch.Generator().manual_seed(3), "cpu")).reshape(k, m, 2), \
        inputs.to_ff(inputs.loguniform_f64(k * n, torch.Generator().manual_seed(4), "cpu")).reshape(k, n, 2)
    got = ff.gemv_dA(dY.to(DEV), X.to(DEV)).cpu().numpy()
    rows = sorted({r for r in (0, 1, 4, m // 3, m // 2, m - 2, m - 1) if 0 <= r < m})
    want = oracle.gemv_dA(np.ascontiguousarray(dY[:, rows].numpy()), X.numpy())
    same_bits(got[rows], want)
    assert np.isfinite(got).all()
