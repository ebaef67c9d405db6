"""Kernels launched back to back: each reads what the one before it wrote, on
one stream, across two streams joined by events, between other libraries'
kernels and copies, and inside a captured graph.  Every chain gives the bits of
the same chain with the device idle before each call."""
import pytest
import torch

from paper_cs_0603115_gb300 import inputs

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_cs_0603115_gb300 as ff
    from paper_cs_0603115_gb300 import batch

DEV = "cuda"


def rnd(seed, *shape):
    n = 1
    for q in shape:
        n *= q
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return inputs.to_ff(inputs.loguniform_f64(n, g, DEV)).reshape(*shape, 2)


def unit(t):
    """Scaled by a power of two so that the largest value is near 1 (no value of the chain overflows)."""
    return t * torch.exp2(-torch.ceil(torch.log2(t.abs().amax())))


class Chain:
    """Every kind of kernel, each call reading an earlier call's output that a
    later call overwrites."""

    def __init__(self, m, n):
        k = 3
        self.A, self.B = rnd(1, m, n), rnd(2, n, k)
        self.X, self.dY = rnd(3, k, n), rnd(4, k, m)
        self.v, self.w = rnd(5, n), rnd(6, n)
        self.d = torch.zeros(2, device=DEV)
        self.z = torch.zeros(n, 2, device=DEV)
        self.C = torch.zeros(m, k, 2, device=DEV)
        self.Y = torch.zeros(k, m, 2, device=DEV)
        self.dX = torch.zeros(k, n, 2, device=DEV)
        self.s = torch.zeros(2, device=DEV)
        self.u = torch.zeros(n, 2, device=DEV)
        self.plan = batch.BatchPlan(batch.make_instances([(batch.DOT, self.w, self.z, self.s, None),
                                                          (batch.AXPY, self.v, self.z, self.u, (1.5, 2.0 ** -26))]))
        for t in (self.A, self.B, self.X, self.dY, self.v, self.w):
            t.copy_(unit(t))

    def steps(self):
        yield lambda: ff.mul(self.v, self.w, out=self.z)
        yield lambda: ff.dot(self.z, self.w, self.d)
        yield lambda: ff.dot_backward(self.d, self.z, self.w, self.v, self.u)
        yield lambda: ff.add(self.u, self.w, out=self.z)
        yield lambda: self.plan.run()
        yield lambda: ff.add(self.u, self.v, out=self.w)
        yield lambda: self.w.copy_(unit(self.w))            # other kernels in between
        yield lambda: ff.gemv(self.A, self.X, self.Y)
        yield lambda: ff.gemv_t(self.A, self.Y, self.dX)
        yield lambda: self.X.copy_(unit(self.dX))
        yield lambda: self.Y.copy_(unit(self.Y))
        yield lambda: ff.gemv_dA(self.Y, self.X, self.A)
        yield lambda: ff.gemm(self.A, self.B, out=self.C)
        yield lambda: self.dY.copy_(self.C.permute(1, 0, 2))
        yield lambda: ff.gemv_t(self.A, self.dY, self.dX)
        yield lambda: ff.sum(self.dX.reshape(-1, 2), self.s)
        yield lambda: self.X.copy_(unit(self.dX))
        yield lambda: ff.add(self.w, self.z, out=self.v)
        yield lambda: self.v.copy_(unit(self.v))

    def state(self):
        return [t.clone() for t in (self.v, self.w, self.z, self.d, self.A, self.X, self.Y, self.dX, self.C, self.s, self.u)]


def same(a, b):
    for x, y in zip(a, b):
        assert torch.equal(x.view(torch.int32), y.view(torch.int32))


SHAPES = [(33, 70), (300, 1001), (700, 1500)]


def alone(m, n, rounds):
    c = Chain(m, n)
    for _ in range(rounds):
        for f in c.steps():
            torch.cuda.synchronize()
            f()
    torch.cuda.synchronize()
    got = c.state()
    assert all(torch.isfinite(t).all() for t in got)
    return got


@pytest.mark.parametrize("m,n", SHAPES)
def test_one_stream(m, n):
    want = alone(m, n, 4)
    for s in (torch.cuda.current_stream(), torch.cuda.Stream()):
        for _ in range(5):
            c = Chain(m, n)
            torch.cuda.synchronize()
            with torch.cuda.stream(s):
                for _ in range(4):
                    for f in c.steps():
                        f()
            torch.cuda.synchronize()
            same(c.state(), want)


@pytest.mark.parametrize("m,n", SHAPES)
def test_two_streams(m, n):
    want = alone(m, n, 3)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(5):
        c = Chain(m, n)
        torch.cuda.synchronize()
        i = 0
        for _ in range(3):
            for f in c.steps():
                s, t = streams[i % 2], streams[(i + 1) % 2]
                with torch.cuda.stream(s):
                    f()
                t.wait_stream(s)
                i += 1
        torch.cuda.synchronize()
        same(c.state(), want)


@pytest.mark.parametrize("m,n", SHAPES)
def test_captured(m, n):
    want = alone(m, n, 3)
    c = Chain(m, n)
    start = [t.clone() for t in (c.A, c.X, c.dY, c.v, c.w)]
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        for f in c.steps():      # workspaces and allocations
            f()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        for f in c.steps():
            f()
    for t, v in zip((c.A, c.X, c.dY, c.v, c.w), start):
        t.copy_(v)
    for t in (c.z, c.d, c.C, c.Y, c.dX, c.s, c.u):
        t.zero_()
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    same(c.state(), want)
