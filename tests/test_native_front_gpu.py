"""The native front of the wrappers (csrc/ff_torch.cpp): it takes the calls the
wrappers accept and leaves every other one, untouched, to the Python path."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_cs_0603115_gb300 as ff
    from paper_cs_0603115_gb300 import _lib


class Sub(torch.Tensor):
    pass


def operands():
    g = torch.Generator(device="cuda").manual_seed(1)
    return (torch.rand((37, 2), generator=g, device="cuda"), torch.rand((37, 2), generator=g, device="cuda"))


def test_valid_calls_are_taken_and_agree():
    a, b = operands()
    out = torch.empty_like(a)
    _lib.call("ff_mul", a.data_ptr(), b.data_ptr(), out.data_ptr(), 37, torch.cuda.current_stream().cuda_stream)
    got = ff._native("binary", "ff_mul", a, b, None)
    assert got is not None and torch.equal(got, out)
    given = torch.empty_like(a)
    assert ff._native("binary", "ff_mul", a, b, given) is given and torch.equal(given, out)
    w = torch.nn.Parameter(a)
    got = ff._native("binary", "ff_mul", w, b, None)
    assert torch.equal(got, out) and not got.requires_grad


@pytest.mark.parametrize("case", ["cpu", "dtype", "shape", "last", "strided", "subclass", "out shape", "out strided",
                                  "mode", "vmap", "number"])
def test_other_calls_are_left_alone(case):
    a, b = operands()
    out = None
    if case == "cpu":
        a, b = a.cpu(), b.cpu()
    elif case == "dtype":
        a = a.double()
    elif case == "shape":
        b = b[1:].contiguous()
    elif case == "last":
        a, b = a.reshape(2, 37), b.reshape(2, 37)
    elif case == "strided":
        a = a.t().contiguous().t()
    elif case == "subclass":
        a = a.as_subclass(Sub)
    elif case == "out shape":
        out = torch.empty(38, 2, device="cuda")
    elif case == "out strided":
        out = torch.empty(2, 37, device="cuda").t()
    elif case == "number":
        a = 1.0
    if case == "mode":
        class Mode(torch.overrides.TorchFunctionMode):
            def __torch_function__(self, func, types, args=(), kwargs=None):
                return func(*args, **(kwargs or {}))
        with Mode():
            assert ff._native("binary", "ff_add", a, b, out) is None
        return
    if case == "vmap":
        seen = []

        def f(x):
            seen.append(ff._native("binary", "ff_add", x, x, None))
            return x
        torch.vmap(f)(a.reshape(37, 1, 2))
        assert seen == [None]
        return
    assert ff._native("binary", "ff_add", a, b, out) is None
    if case == "subclass":     # the Python path serves it
        assert torch.equal(ff.add(a, b).as_subclass(torch.Tensor), ff.add(a.as_subclass(torch.Tensor), b))
    else:
        with pytest.raises((ValueError, AttributeError)):
            ff.add(a, b, out)


def test_workspace_missing_then_cached():
    a, b = operands()
    ff.clear_workspaces()
    size = _lib.address["ff_reduce_workspace_bytes"]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        assert ff._native("reduce2", "ff_dot", a, b, None, True, size, ff._ws_cache, "reduce") is None
        want = ff.dot(a, b)    # the Python path allocates this stream's workspace
        got = ff._native("reduce2", "ff_dot", a, b, None, True, size, ff._ws_cache, "reduce")
    torch.cuda.synchronize()
    assert got is not None and torch.equal(got, want)


def test_library_errors_are_raised():
    A = torch.rand((8, 4, 2), device="cuda")
    X = torch.rand((65, 4, 2), device="cuda")       # at most 64 right-hand sides
    with pytest.raises(ff.FFError) as e:
        ff.gemv(A, X)
    assert e.value.status == 1
