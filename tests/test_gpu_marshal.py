"""The native form of the binding's marshalling against its Python form: the same results, the same refusals."""
import os
import subprocess
import sys
import sysconfig
from pathlib import Path

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


# an allocator that counts its calls and those in which this thread held the interpreter's lock
COUNTING_ALLOCATOR = r"""
#include <Python.h>
#include <cuda_runtime_api.h>
static int calls, locked;
extern "C" int count_calls() { return calls; }
extern "C" int count_locked() { return locked; }
extern "C" void* counting_alloc(ssize_t size, int, cudaStream_t)
{
    void* p = nullptr;
    ++calls;
    locked += PyGILState_Check();
    return cudaMalloc(&p, size) == cudaSuccess ? p : nullptr;
}
extern "C" void counting_free(void* p, ssize_t, int, cudaStream_t) { cudaFree(p); }
"""
COUNTING_PROGRAM = r"""
import ctypes, sys
import torch
torch.cuda.memory.change_current_allocator(torch.cuda.memory.CUDAPluggableAllocator(sys.argv[1], "counting_alloc", "counting_free"))
from paper_2603_06738_b200 import binding
assert binding._marshal is not None
count = ctypes.CDLL(sys.argv[1])
q = torch.randn((1, 16, 16, 1, 32), device="cuda").bfloat16()
pq = torch.randn((256, 16), device="cuda").bfloat16()
w = [torch.randn(s, device="cuda") for s in ((6, 8), (8,), (8, 16), (8, 16))]
d = torch.randn((256, 16), device="cuda")
ws = torch.empty(1 << 22, dtype=torch.uint8, device="cuda")
before, held = count.count_calls(), count.count_locked()
out, lse = binding.rib_window_attn_fwd(q, q, q, pq, pq, 16)
grads = binding.rib_window_attn_bwd(q, q, q, pq, pq, out, lse, q, 16, workspace=ws)
features = binding.rib_generate_features(*w, 16)
generator = binding.rib_generate_features_bwd(*w, d, d, 16)
torch.cuda.synchronize()
print(count.count_calls() - before, count.count_locked() - held)
"""


def test_results_are_allocated_without_the_interpreters_lock(tmp_path):
    source, lib = tmp_path / "alloc.cpp", tmp_path / "alloc.so"
    source.write_text(COUNTING_ALLOCATOR)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-shared", "-fPIC", f"-I{sysconfig.get_path('include')}", f"-I{cuda}/include", str(source), f"-L{cuda}/lib64", "-lcudart", "-o", str(lib)], check=True)
    run = subprocess.run([sys.executable, "-c", COUNTING_PROGRAM, str(lib)], cwd=Path(__file__).resolve().parent.parent, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr
    calls, locked = map(int, run.stdout.split()[-2:])
    assert calls >= 13 and locked == 0, run.stdout      # 2 + 5 + 2 + 4 results
