"""Tensors and modes that the native half of the Python binding must not look
into: each gives the result, or the refusal, of the binding's own checks."""
import importlib
import threading

import pytest
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
from torch.overrides import TorchFunctionMode
from torch.utils._python_dispatch import TorchDispatchMode

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mw():
    m = importlib.import_module("paper_2608_01127_gb300")
    m.library()
    assert m._native is not None
    return m


class Sub(torch.Tensor):
    pass


class FunctionMode(TorchFunctionMode):
    def __torch_function__(self, func, types, args=(), kwargs=None):
        return func(*args, **(kwargs or {}))


class DispatchMode(TorchDispatchMode):
    def __torch_dispatch__(self, func, types, args=(), kwargs=None):
        return func(*args, **(kwargs or {}))


def fake(mw, q, do):
    with FakeTensorMode(allow_non_fake_inputs=True) as mode:
        f = mode.from_tensor(q)
        return mw.mw_bca_fwd(f, f, f, 64)


def fake_outputs(mw, q, do):
    with FakeTensorMode(allow_non_fake_inputs=True):
        return mw.mw_bca_fwd(q, q, q, 64)


def with_mode(mode):
    def run(mw, q, do):
        with mode:
            o, lse = mw.mw_bca_fwd(q, q, q, 64)
            return o, lse, *mw.mw_bca_bwd(q, q, q, o, lse, do, 64)
    return run


def subclass(mw, q, do):
    s = q.as_subclass(Sub)
    return mw.mw_bca_fwd(s, s, s, 64)


def parameter(mw, q, do):
    p = torch.nn.Parameter(q)
    return mw.mw_bca_fwd(p, p, p, 64)


def vmap(mw, q, do):
    return torch.func.vmap(lambda x: mw.mw_bca_fwd(x, x, x, 64)[0])(torch.stack([q, q]))


def grad(mw, q, do):
    return torch.func.grad(lambda x: mw.mw_bca_fwd(x, x, x, 64)[0].float().sum())(q)


def grad_inside(mw, q, do):  # plain inputs, but outputs allocated at a grad level
    return torch.func.grad(lambda x: x.sum() + mw.mw_bca_fwd(q, q, q, 64)[0].sum())(q)


def functionalize(mw, q, do):
    return torch.func.functionalize(lambda x: mw.mw_bca_fwd(x, x, x, 64)[0])(q)


def dual(mw, q, do):
    with torch.autograd.forward_ad.dual_level():
        return mw.mw_bca_fwd(torch.autograd.forward_ad.make_dual(q, q), q, q, 64)


def dual_function(mw, q, do):
    with torch.autograd.forward_ad.dual_level():
        return mw.BlockCausalAttention.apply(torch.autograd.forward_ad.make_dual(q, q), q, q, 64, None)


def lazy_ring(mw, q, do):  # the commit writes the clone, not what it shares
    ring = torch.zeros_like(q)
    kc, vc = torch._lazy_clone(ring), torch._lazy_clone(ring)
    out = mw.mw_bca_cache_step(q, q, q, kc, vc, 0, 0, 0, 64, 64)
    return *out, kc, vc, ring


def freed(mw, q, do):
    t = q.clone()
    t.untyped_storage().resize_(0)
    return mw.mw_bca_fwd(t, q, q, 64)


def negated(mw, q, do):
    n = torch._neg_view(q)
    return mw.mw_bca_fwd(n, q, q, 64)


def inference(mw, q, do):
    with torch.inference_mode():
        return mw.mw_bca_fwd(q, q, q, 64)


def saved_hooks(mw, q, do):
    x = [q.clone().requires_grad_() for _ in range(3)]
    with torch.autograd.graph.saved_tensors_hooks(lambda t: t.cpu(), lambda t: t.cuda()):
        o = mw.BlockCausalAttention.apply(*x, 64, None)
    o.backward(do)
    return o.detach(), *(t.grad for t in x)


def second_thread(mw, q, do):
    out = []
    t = threading.Thread(target=lambda: out.extend(mw.mw_bca_fwd(q, q, q, 64)))
    t.start()
    t.join()
    return out


def own_stream(mw, q, do):
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        x = q * 1.0  # on that stream: the forward has to follow it there
        out = mw.mw_bca_fwd(x, x, x, 64)
    torch.cuda.current_stream().wait_stream(s)
    return out


FORMS = [fake, fake_outputs, subclass, parameter, vmap, grad, grad_inside, functionalize, dual, dual_function,
         lazy_ring, freed, negated, inference, saved_hooks, second_thread, own_stream]


REFUSED = {fake, fake_outputs, vmap, grad, grad_inside, functionalize, dual_function, freed}


def outcome(run, mw, q, do):
    try:
        out = run(mw, q, do)
    except Exception as e:  # noqa: BLE001
        return type(e), str(e)
    return [out] if isinstance(out, torch.Tensor) else list(out)


@pytest.mark.parametrize("run", FORMS + [with_mode(FunctionMode()), with_mode(DispatchMode())],
                         ids=[f.__name__ for f in FORMS] + ["function_mode", "dispatch_mode"])
def test_same_as_the_checked_way(mw, run, monkeypatch):
    g = torch.Generator("cuda").manual_seed(3)
    # one query tile against one key tile: the backward's bits do not depend on an order
    q, do = (torch.randn(1, 2, 128, 64, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    native = outcome(run, mw, q, do)
    monkeypatch.setattr(mw, "_native", None)
    checked = outcome(run, mw, q, do)
    torch.cuda.synchronize()
    assert type(native) is type(checked) is (tuple if run in REFUSED else list), (native, checked)
    if isinstance(native, tuple):
        assert native == checked
        return
    for a, b in zip(native, checked, strict=True):
        assert type(a) is type(b) and a.shape == b.shape and a.dtype == b.dtype
        assert a.requires_grad == b.requires_grad and a.is_inference() == b.is_inference()
        assert torch.equal(a, b)
