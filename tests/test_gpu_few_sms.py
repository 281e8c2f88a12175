"""Calls on a stream that owns a few SMs (a green context of the driver): the launches whose blocks
must all run at once are refused there or fit, and the results are the same."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

I32_MIN, I32_MAX = -(1 << 31), (1 << 31) - 1
SM_RESOURCE, DEFAULT_STREAM, NON_BLOCKING = 1, 1, 1


class DevResource(C.Structure):
    _fields_ = [("type", C.c_uint32), ("padding", C.c_ubyte * 92), ("body", C.c_ubyte * 48)]


@pytest.fixture(scope="module")
def crys():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2003_01178_gb300 import _build
    _build.build()
    import paper_2003_01178_gb300 as crys
    crys.crys_device_errors(clear=True)
    yield crys
    assert crys.crys_device_errors(clear=True) == 0


@pytest.fixture(scope="module")
def few_sms():
    """Handle of a stream on 8 SMs."""
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    if not hasattr(cu, "cuGreenCtxStreamCreate"):
        pytest.skip("the driver has no green contexts")
    whole, part, rest = DevResource(), DevResource(), DevResource()
    groups, desc, ctx, stream = C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
    steps = [lambda: cu.cuDeviceGetDevResource(0, C.byref(whole), SM_RESOURCE),
             lambda: cu.cuDevSmResourceSplitByCount(C.byref(part), C.byref(groups), C.byref(whole), C.byref(rest), 0, 8),
             lambda: cu.cuDevResourceGenerateDesc(C.byref(desc), C.byref(part), 1),
             lambda: cu.cuGreenCtxCreate(C.byref(ctx), desc, 0, DEFAULT_STREAM),
             lambda: cu.cuGreenCtxStreamCreate(C.byref(stream), ctx, NON_BLOCKING, 0)]
    for i, step in enumerate(steps):
        if step() != 0:
            pytest.skip(f"no green context here (step {i})")
    yield stream.value
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


def _bits(n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    return torch.randint(I32_MIN, I32_MAX, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)


@pytest.mark.parametrize("n", [1000, 65_536, 131_072, 3_000_017])
@pytest.mark.parametrize("ordered", [0, 1])
def test_selections(crys, few_sms, n, ordered):
    x = _bits(n)
    out, count = torch.empty_like(x), torch.zeros(1, dtype=torch.int64, device="cuda")
    tb = crys.crys_select(None, n, 0, 0, None, None, ordered, None, -1)
    temp = crys.scratch(tb, "cuda") if tb else None
    torch.cuda.synchronize()
    crys.crys_select(x, n, 0, I32_MAX, out, count, ordered, temp, tb, stream=few_sms)
    torch.cuda.synchronize()
    got, ref = out[:int(count)], x[x >= 0]
    assert torch.equal(got, ref) if ordered else torch.equal(got.sort().values, ref.sort().values)


@pytest.mark.parametrize("n", [4000, 5000, 100_003, 1 << 20, 3_000_017])
@pytest.mark.parametrize("op", ["sort", "sort_msb"])
def test_sorts(crys, few_sms, n, op):
    keys, vals = _bits(n), torch.arange(n, dtype=torch.int32, device="cuda")
    ko, vo = torch.empty_like(keys), torch.empty_like(vals)
    f = getattr(crys, "crys_" + op)
    tb = f(None, None, None, None, n, None, -1)
    temp = crys.scratch(tb, "cuda")
    torch.cuda.synchronize()
    f(keys, vals, ko, vo, n, temp, tb, stream=few_sms)
    torch.cuda.synchronize()
    rk, order = torch.sort(keys, stable=True)
    assert torch.equal(ko, rk) and torch.equal(keys[vo.long()], rk) and torch.equal(vo.sort().values, vals)
    if op == "sort":
        assert torch.equal(vo, order.to(torch.int32))
