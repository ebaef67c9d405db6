"""Batched GEMV plans of many small matrices: a block per tile, a matrix's rows
spread over the tile's warps, every row bit for bit the documented eight-lane
sum; and plans of large tiles, walked by resident blocks."""
import random

import pytest
import torch

import replay
from paper_cs_0603115_gb300 import inputs

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_cs_0603115_gb300 import batch


def plan_of(shapes, tune=None, pad=True):
    rng = torch.Generator(device="cuda").manual_seed(len(shapes))
    up = (lambda v: v + (v & 1)) if pad else (lambda v: v)
    A = inputs.to_ff(inputs.loguniform_f64(sum(up(m * n) for m, n in shapes), rng, "cuda"))
    x = inputs.to_ff(inputs.loguniform_f64(sum(up(n) for _, n in shapes), rng, "cuda"))
    y = torch.full((sum(m for m, _ in shapes), 2), float("nan"), device="cuda")
    specs, a, b, c = [], 0, 0, 0
    for m, n in shapes:
        specs.append((batch.GEMV, A[a:a + m * n].view(m, n, 2), x[b:b + n], y[c:c + m], None))
        a, b, c = a + up(m * n), b + up(n), c + m
    return batch.BatchPlan(batch.make_instances(specs), tune=tune), specs, y


def check(specs, picks):
    for i in picks:
        _, A, x, y, _ = specs[i]
        vec = A.data_ptr() % 16 == 0 and x.data_ptr() % 16 == 0 and A.shape[1] % 2 == 0
        want = replay.gemv_rows8_replay(A.cpu().numpy(), x.cpu().numpy(), vec)
        assert (y.cpu().numpy().view("u4") == want.view("u4")).all(), tuple(A.shape)


@pytest.mark.parametrize("pad", [True, False])
@pytest.mark.parametrize("tune", [None, (128, 16, 0, 2), (512, 8, 0, 4), (256, 32, 2, 4)])
@pytest.mark.parametrize("lo,hi,count", [(1, 9, 6000), (8, 8, 6000), (17, 70, 5000)])
def test_small_matrices(lo, hi, count, tune, pad):
    rng = random.Random(count + hi)
    shapes = [(rng.randint(lo, hi), rng.randint(lo, hi)) for _ in range(count)]
    plan, specs, y = plan_of(shapes, tune, pad)
    if tune is None or tune[2] == 0:
        assert plan.grid == plan.ntiles     # a block per tile
    for _ in range(2):
        y.fill_(float("nan"))
        plan.run()
        torch.cuda.synchronize()
        assert torch.isfinite(y).all()
        check(specs, list(range(0, count, count // 60)) + [count - 1])
    plan.close()


def test_large_tiles_stay_with_resident_blocks():
    plan, specs, y = plan_of([(9000, 400)] * 10)
    assert plan.grid < plan.ntiles
    plan.run()
    torch.cuda.synchronize()
    assert torch.isfinite(y).all()
    sub = [(k, A[:5], x, out[:5], al) for k, A, x, out, al in specs]
    check(sub, [0, 9])
    plan.close()
