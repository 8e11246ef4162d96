"""The native form of the binding's marshalling against its Python form: the same results, the same refusals."""
import numpy as np
import pytest
import torch

from paper_2603_06738_b200 import binding, synthetic
from paper_2603_06738_b200.synthetic import Workload

pytestmark = pytest.mark.gpu


def both(monkeypatch, call):
    """What `call` returns or raises with the native marshaller and without it."""
    results = []
    for native in (True, False):
        with monkeypatch.context() as m:
            if not native:
                m.setattr(binding, "_marshal", None)
            try:
                results.append(call())
            except Exception as e:          # noqa: BLE001 - whatever it is has to be the same
                results.append((type(e), str(e)))
    return results


def same(a, b):
    if torch.is_tensor(a):
        return torch.is_tensor(b) and a.dtype == b.dtype and a.shape == b.shape and a.device == b.device and not a.requires_grad and bool(torch.equal(a, b))
    if isinstance(a, (tuple, list)):
        return type(a) is type(b) and len(a) == len(b) and all(same(x, y) for x, y in zip(a, b))
    return a == b


def inputs(headwise):
    wl = Workload("marshal", 1, 32, 32, 2, 32, 16, 16, 8, seed=41, headwise=headwise)
    g = {k: v.cuda() for k, v in synthetic.make_inputs(wl, True).items()}
    return [g[k] for k in ("q", "k", "v", "pq", "pk")], g["dout"]


def test_the_library_was_built_with_it():
    assert binding._marshal is not None


@pytest.mark.parametrize("name,headwise", [("", False), ("_headwise", True), ("_padded", False), ("_padded", True), ("_masked", False), ("_masked", True)])
def test_same_results(monkeypatch, name, headwise):
    args, dout = inputs(headwise)
    fwd, bwd = getattr(binding, "rib_window_attn_fwd" + name), getattr(binding, "rib_window_attn_bwd" + name)
    for options in ({}, {"want_lse": False}, {"stream": torch.cuda.Stream()}):
        a, b = both(monkeypatch, lambda: fwd(*args, 16, 8, **options))
        torch.cuda.synchronize()
        assert same(a, b)
    out, lse = fwd(*args, 16, 8)
    workspace = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
    a, b = both(monkeypatch, lambda: bwd(*args, out, lse, dout, 16, 8, workspace=workspace))
    assert same(a[:3], b[:3])           # dpq, dpk are sums in an order that may differ
    for x, y in zip(a[3:], b[3:]):
        assert x.shape == y.shape and x.dtype == y.dtype and float((x - y).norm()) <= 1e-5 * float(y.norm())


def test_same_generator_results(monkeypatch):
    gen = torch.Generator(device="cuda").manual_seed(3)
    w = [torch.nn.Parameter(torch.randn(s, generator=gen, device="cuda") * 0.2) for s in ((42, 32), (32,), (32, 16), (32, 16))]
    a, b = both(monkeypatch, lambda: binding.rib_generate_features(*w, 16))
    assert same(a, b)
    d = [torch.randn((256, 16), generator=gen, device="cuda") for _ in range(2)]
    a, b = both(monkeypatch, lambda: binding.rib_generate_features_bwd(*w, *d, 16))
    for x, y in zip(a, b):
        assert x.shape == y.shape and not x.requires_grad and float((x - y).norm()) <= 1e-5 * float(y.norm())


def test_same_refusals(monkeypatch):
    args, dout = inputs(False)
    q, k, v, pq, pk = args
    fwd, bwd = binding.rib_window_attn_fwd, binding.rib_window_attn_bwd
    out, lse = fwd(*args, 16, 8)
    ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
    strided = q.permute(0, 2, 1, 3, 4)
    for call in (lambda: fwd(strided, k, v, pq, pk, 16, 8), lambda: fwd(q.cpu(), k, v, pq, pk, 16, 8), lambda: fwd(q.float(), k, v, pq, pk, 16, 8),
                 lambda: fwd(q, k[:, :16].contiguous(), v, pq, pk, 16, 8), lambda: fwd(q, k, v, pq[:64], pk[:64], 16, 8), lambda: fwd(q, k, v, pq[None], pk[None], 16, 8),
                 lambda: fwd(*args, 0, 0), lambda: fwd(*args, 12, 0), lambda: fwd(*args, 16, 99), lambda: fwd(*args, 16, -8), lambda: fwd(*args, "16", 8),
                 lambda: fwd(None, k, v, pq, pk, 16, 8), lambda: fwd(q[0], k, v, pq, pk, 16, 8), lambda: bwd(*args, out, lse[..., :16], dout, 16, 8, workspace=ws),
                 lambda: bwd(*args, out, lse.half(), dout, 16, 8, workspace=ws), lambda: bwd(*args, out, lse, dout.float(), 16, 8, workspace=ws),
                 lambda: bwd(*args, out, lse, dout, 16, 8, workspace=ws[:64]), lambda: fwd(q[:0], k[:0], v[:0], pq, pk, 16, 8)):
        a, b = both(monkeypatch, call)
        torch.cuda.synchronize()
        assert same(a, b) if torch.is_tensor(a[0]) else a == b, (a, b)      # (a pair of type and text where it was refused)
    # and what is taken although it is not quite plain: a subclass, a NumPy integer, a flag that is no bool
    class Sub(torch.Tensor):
        pass
    for call in (lambda: fwd(q.as_subclass(Sub), k, v, pq, pk, 16, 8), lambda: fwd(*args, np.int64(16), np.int32(8)), lambda: fwd(*args, 16, 8, want_lse=0)):
        a, b = both(monkeypatch, call)
        assert torch.is_tensor(a[0]) and torch.equal(a[0], b[0]) and type(a[0]) is type(b[0]) and (a[1] is None) == (b[1] is None)


def test_under_capture():
    args, _ = inputs(False)
    want = binding.rib_window_attn_fwd(*args, 16, 8)[0].clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out, _ = binding.rib_window_attn_fwd(*args, 16, 8)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


def test_tensors_that_have_no_plain_memory(monkeypatch):
    """A nested tensor is strided, dense and five-dimensional, and throws when it is asked for its sizes; what is allocated inside a
    gradient transform is a wrapper without storage.  Either is an exception of the Python form, not the end of the process."""
    args, dout = inputs(False)
    q, k, v, pq, pk = args
    fwd, bwd = binding.rib_window_attn_fwd, binding.rib_window_attn_bwd
    out, lse = fwd(*args, 16, 8)
    ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(3)
    w = [torch.randn(s, generator=gen, device="cuda") * 0.2 for s in ((42, 32), (32,), (32, 16), (32, 16))]
    d = [torch.randn((256, 16), generator=gen, device="cuda") for _ in range(2)]
    nest = lambda t: torch.nested.nested_tensor(list(t), dtype=t.dtype, device="cuda")
    x = torch.ones(3, device="cuda")

    def inside(transform, call):
        def f(x):
            call()
            return x.sum()
        return transform(f)

    calls = (lambda: fwd(*args, 16, 8), lambda: bwd(*args, out, lse, dout, 16, 8, workspace=ws), lambda: binding.rib_generate_features(*w, 16),
             lambda: binding.rib_generate_features_bwd(*w, *d, 16))
    for call in (lambda: fwd(nest(q), k, v, pq, pk, 16, 8), lambda: fwd(q, k, v, nest(pq), pk, 16, 8), lambda: bwd(q, k, nest(v), pq, pk, out, lse, dout, 16, 8, workspace=ws),
                 lambda: bwd(*args, out, nest(lse), dout, 16, 8, workspace=ws), lambda: binding.rib_generate_features(nest(w[0]), *w[1:], 16),
                 lambda: binding.rib_generate_features_bwd(*w, nest(d[0]), d[1], 16),
                 *(lambda c=c: inside(torch.func.grad, c)(x) for c in calls), *(lambda c=c: inside(lambda f: lambda x: torch.func.jvp(f, (x,), (x,)), c)(x) for c in calls)):
        a, b = both(monkeypatch, call)
        torch.cuda.synchronize()
        assert a == b and issubclass(a[0], Exception), (a, b)
    for call in calls:                          # (no wrapper is made under a batched map of something else)
        a, b = both(monkeypatch, lambda: inside(torch.vmap, call)(torch.ones(2, 3, device="cuda")))
        assert torch.equal(a, b)
