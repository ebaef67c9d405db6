"""The reductions' two kernels for vectors on common 16-byte offsets (one group
of chunks per thread, and the loop), and the one for mixed offsets: around the
longest one-group grid and the grid cap, with first and last values outside the
chunks, part groups, and pairs that are not normalised.  Every result has the
bits of the replay of the documented order, so no tolerance."""
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
    np.testing.assert_array_equal(np.ascontiguousarray(got, np.float32).view(np.uint32),
                                  np.ascontiguousarray(want, np.float32).view(np.uint32))


def shape(name, x, y):
    g, h, v = ctypes.c_uint(), ctypes.c_int(), ctypes.c_int()
    _lib.call(name, x.data_ptr(), None if y is None else y.data_ptr(), x.shape[0],
              ctypes.byref(g), ctypes.byref(h), ctypes.byref(v))
    return g.value, h.value, bool(v.value)


def sizes():
    """Chunks: whole and part groups of one block, and of the grids around 5 and
    6 blocks per SM (152 SMs; another count only moves the edges)."""
    for blocks in (1, 2, 760, 912):
        for chunks in (blocks * 1024 - 1025, blocks * 1024 - 257, blocks * 1024, blocks * 1024 + 3):
            if chunks > 0:
                yield chunks


@pytest.mark.parametrize("chunks", list(sizes()))
@pytest.mark.parametrize("kind", ["aligned", "head", "mixed"])
def test_float_float(chunks, kind):
    n = 2 * chunks + 1
    g = inputs.ill_dot(n + 1, 1e9, inputs.seed_for(8, 70))
    x, y = g.x.clone(), g.y.clone()
    x[::97, 1] = x[::97, 0] * 0.75                     # sums that do not round to the high part
    xd, yd = x.to(DEV), y.to(DEV)
    a, b = {"aligned": (0, 0), "head": (1, 1), "mixed": (1, 0)}[kind]
    xd, yd = xd[a:a + n], yd[b:b + n]
    xn, yn = x[a:a + n].numpy(), y[b:b + n].numpy()
    same_bits(ff.dot(xd, yd).cpu().numpy(),
              replay.reduce_replay(oracle.mul22(xn, yn), *shape("ff_reduce_launch_shape", xd, yd)))
    if kind != "mixed":
        same_bits(ff.sum(xd).cpu().numpy(), replay.reduce_replay(xn, *shape("ff_reduce_launch_shape", xd, None)))


@pytest.mark.parametrize("chunks", list(sizes()))
@pytest.mark.parametrize("kind", ["aligned", "head", "mixed"])
def test_binary32(chunks, kind):
    n = 4 * chunks + 3
    g = inputs.ill_dot_f32(n + 3, 1e9, inputs.seed_for(8, 71))
    a, b = {"aligned": (0, 0), "head": (3, 3), "mixed": (2, 1)}[kind]
    xd, yd = g.x.to(DEV)[a:a + n], g.y.to(DEV)[b:b + n]
    xn, yn = g.x[a:a + n].numpy(), g.y[b:b + n].numpy()
    pol = replay.Dot2Policy()
    same_bits(ff.dot2(xd, yd).cpu().numpy(),
              replay.reduce_replay(oracle.mul12(np.stack([xn, yn], 1)),
                                   *shape("ff_reduce2_launch_shape", xd, yd), pol))
    if kind != "mixed":
        same_bits(ff.sum2(xd).cpu().numpy(),
                  replay.reduce_replay(np.stack([xn, np.zeros_like(xn)], 1),
                                       *shape("ff_reduce2_launch_shape", xd, None), pol))
