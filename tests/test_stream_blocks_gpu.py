"""The elementwise kernels' blocks: sizes around one block's run, around the
line between one and two vectors per thread (and one and four values on mixed
offsets), with first and last values outside the 16-byte vectors.  Every value
has the oracle's bits; values beside the output stay untouched."""
import numpy as np
import pytest
import torch

import oracle
from paper_cs_0603115_gb300 import inputs

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_cs_0603115_gb300 as ff

DEV = "cuda"
LINE = 152 * 2048          # resident threads (152 SMs; another count only moves the edge)


def same_bits(got, want):
    np.testing.assert_array_equal(np.ascontiguousarray(got, np.float32).view(np.uint32),
                                  np.ascontiguousarray(want, np.float32).view(np.uint32))


@pytest.mark.parametrize("n", [1, 2, 3, 255, 256, 257, 511, 513, LINE - 1, LINE, LINE + 1, LINE + 511, 2 * LINE - 1, 2 * LINE,
                               2 * LINE + 1, 2 * LINE + 255, 2 * LINE + 513])
@pytest.mark.parametrize("offsets", [(0, 0, 0), (1, 1, 1), (0, 1, 0), (1, 0, 1), (0, 0, 1)])
def test_blocks(n, offsets):
    e = inputs.elementwise(n + 1, 17)
    i, j, k = offsets
    a, b = e.a[i:i + n], e.b[j:j + n]
    ad, bd = e.a.to(DEV)[i:i + n], e.b.to(DEV)[j:j + n]
    d = torch.tensor([1.5, 2.0 ** -26], device=DEV)

    def run(f, want):
        whole = torch.full((n + 2, 2), 7.0, device=DEV)
        f(whole[k:k + n])
        got = whole.cpu().numpy()
        same_bits(got[k:k + n], want)
        assert (got[:k] == 7.0).all() and (got[k + n:] == 7.0).all()

    run(lambda o: ff.mul(ad, bd, o), oracle.mul22(a.numpy(), b.numpy()))
    run(lambda o: ff.div(ad, bd, o), oracle.div22(a.numpy(), b.numpy()))
    s = e.a_sqrt.to(DEV)[i:i + n]
    run(lambda o: ff.sqrt(s, o), oracle.sqrt22(e.a_sqrt[i:i + n].numpy()))
    dx = torch.full((n + 2, 2), 7.0, device=DEV)
    dy = torch.full((n + 2, 2), 7.0, device=DEV)
    ff.dot_backward(d, ad, bd, dx[k:k + n], dy[j:j + n])
    dn = np.broadcast_to(d.cpu().numpy(), (n, 2))
    same_bits(dx.cpu().numpy()[k:k + n], oracle.mul22(dn, b.numpy()))
    same_bits(dy.cpu().numpy()[j:j + n], oracle.mul22(dn, a.numpy()))
    assert (dx[k + n:] == 7.0).all() and (dy[j + n:] == 7.0).all()
