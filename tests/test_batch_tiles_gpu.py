"""The batched kernel's tile walk: blocks that meet several multi-tile dots one
after another (each arrival is looked at one dot tile later), partial groups of
a tile, and records whose arrays start at different offsets modulo 16 bytes."""
import numpy as np
import pytest
import torch

import oracle
from paper_cs_0603115_gb300 import inputs

pytestmark = pytest.mark.gpu

DEV = "cuda"


def same_bits(got, want):
    got = np.ascontiguousarray(got, np.float32)
    want = np.ascontiguousarray(want, np.float32)
    nan = np.isnan(got) & np.isnan(want)
    assert ((got.view(np.uint32) == want.view(np.uint32)) | nan).all()


@pytest.mark.parametrize("tune", [(128, 8 * 2, 2, 4), (256, 8, 2, 2), (128, 16, 0, 4)])
def test_many_multi_tile_dots_per_block(tune):
    """700 dots of two to five tiles with AXPYs between them: every block
    takes several, ends some, and combines each of them once."""
    from paper_cs_0603115_gb300 import batch
    import replay
    tile = tune[0] * tune[1]
    rng = np.random.default_rng(5)
    lengths = [int(v) for v in rng.integers(tile + 1, 5 * tile, 700)]
    e = inputs.elementwise(5 * tile, 41)
    x, y = e.a.to(DEV), e.b.to(DEV)
    d = torch.full((700, 2), float("nan"), device=DEV)
    z = torch.full((350, 33, 2), float("nan"), device=DEV)
    specs = []
    for i, n in enumerate(lengths):
        specs.append((batch.DOT, x[:n], y[:n], d[i], None))
        if i % 2:
            specs.append((batch.AXPY, x[:33], y[:33], z[i // 2], (1.5, 2.0 ** -26)))
    plan = batch.BatchPlan(batch.make_instances(specs), tune=tune)
    want = {}
    for _ in range(3):
        d.fill_(float("nan"))
        z.fill_(float("nan"))
        plan.run()
        got = d.cpu().numpy()
        for i in list(range(0, 700, 53)) + [699]:
            if i not in want:
                n = lengths[i]
                want[i] = replay.batch_dot_replay(e.a.numpy()[:n], e.b.numpy()[:n], tune[0], tune[1], 1)
            same_bits(got[i], want[i])
        assert np.isfinite(got).all()
        same_bits(z.cpu().numpy(), np.broadcast_to(
            oracle.axpy(np.array([1.5, 2.0 ** -26], np.float32), e.a.numpy()[:33], e.b.numpy()[:33]), (350, 33, 2)))
    plan.close()


@pytest.mark.parametrize("tune", [None, (128, 16, 0, 2), (512, 64, 2, 4)])
def test_offsets_and_partial_groups(tune):
    """AXPY and DOT_GRAD with every combination of array offsets modulo 16
    bytes, lengths around the groups of a tile; nothing beside the outputs is
    written."""
    from paper_cs_0603115_gb300 import batch
    lengths = [1, 2, 127, 256, 257, 511, 1023, 2047, 2049, 8191, 8193]
    e = inputs.elementwise(max(lengths), 43)
    a, b = e.a.numpy(), e.b.numpy()
    alpha = np.array([-0.75, 2.0 ** -27], np.float32)
    dout = torch.from_numpy(alpha).to(DEV)

    def place(src, off):
        t = torch.full((src.shape[0] + 2, 2), 7.0, device=DEV)
        t[off:off + src.shape[0]] = torch.from_numpy(src).to(DEV)
        return t, t[off:off + src.shape[0]]

    specs, keep = [], []
    for n in lengths:
        for offs in range(8):
            ox, oy, oz = offs & 1, offs >> 1 & 1, offs >> 2
            _, x = place(a[:n], ox)
            _, y = place(b[:n], oy)
            zb, z = place(np.zeros((n, 2), np.float32), oz)
            specs.append((batch.AXPY, x, y, z, tuple(float(v) for v in alpha)))
            ub, u = place(np.zeros((n, 2), np.float32), oz)
            vb, v = place(np.zeros((n, 2), np.float32), oy)
            specs.append((batch.DOT_GRAD, x, y, u, None, v, dout))
            keep.append((n, oz, oy, zb, ub, vb))
    plan = batch.BatchPlan(batch.make_instances(specs), tune=tune)
    plan.run()
    for n, oz, oy, zb, ub, vb in keep:
        dx, dy = oracle.dot_backward(alpha, a[:n], b[:n])
        for buf, off, want in ((zb, oz, oracle.axpy(alpha, a[:n], b[:n])), (ub, oz, dx), (vb, oy, dy)):
            full = np.full((n + 2, 2), 7.0, np.float32)
            full[off:off + n] = want
            same_bits(buf.cpu().numpy(), full)
    plan.close()
