"""The native half of the binding: what it does not take goes to the Python half, and what it takes gives the same results."""
import numpy as np
import pytest

from workloads import configs as C


@pytest.fixture(scope="module")
def P(_built_library):
    import paper_2505_00232_b200 as P
    return P


def test_anything_but_plain_cuda_tensors_is_left_to_python(P):
    import torch
    native = P.binding._bind_torch()
    x, ids = torch.zeros((2, 64), dtype=torch.float16), torch.zeros((3,), dtype=torch.int32)

    class Sub(torch.Tensor):
        pass
    layer, heads = (1, 64, 8), (2, 32, 64, 1, 1, 1)
    for a in (x, x.as_subclass(Sub), x.numpy(), None, 3):
        assert native.forward(layer, a, None, None) is None and native.forward_a8(layer, a, None, None) is None
        assert native.forward_gated(layer, layer, a, 1, None, None) is None and native.embed(layer, a, None, None) is None
        assert native.residual_rmsnorm(a, None, a, 1e-5, 0.0, None, None, True, None) is None
        assert native.rope_qkv(a, a, a, ids, x, x, 1, 2, 1, 1, 64, None) is None
        assert native.kv_append(heads, 0, a, a, None) is None and native.kv_scores(heads, a, None) is None and native.kv_output_heads(heads, a, None) is None
        assert native.kv_output(layer, 1, a, None) is None and native.kv_scores_one(layer, a, None, None) is None
        assert native.forward_group([], a, None) is None and native.forward_group([object()], a, None) is None
    assert native.forward(None, x, None, None) is None                   # (a closed layer)
    with pytest.raises(P.QLinearError):
        P.qlinear_residual_rmsnorm(x, None, x[0], 1e-5)


def test_value_product_is_given_the_scales_that_the_cache_has_now(P, monkeypatch):
    """`v_scale` may be replaced (a restored cache): every call gets the tensor that is there."""
    import torch
    seen = []

    class Native:
        def kv_output(self, *a):
            seen.append(a)
            return a[2]
    monkeypatch.setattr(P.binding, "_native", Native())
    kv, prob = P.KVCache.__new__(P.KVCache), torch.zeros((1, 64), dtype=torch.float16)
    kv.v = type("V", (), {"_native": (1, 64, 32), "_h": None})()
    for _ in range(3):
        kv.v_scale = torch.ones((64,), dtype=torch.float16)
        assert kv.output(prob) is prob and seen[-1][1] is kv.v_scale


@pytest.mark.gpu
@pytest.mark.parametrize("R", [4, 64])
def test_value_product_after_the_scales_were_replaced(P, R):
    import torch
    f16 = lambda *s: torch.randn(s, device="cuda").half()
    d, T, k, prob = 64, 256, f16(5, 64), f16(R, 256)
    kv, fresh = P.KVCache(T, d, "cuda:0"), P.KVCache(T, d, "cuda:0")
    prob[:, 10:] = 0
    old = kv.v_scale
    for v in (f16(5, d), 30 * f16(5, d)):
        kv.append(k, v)
        fresh.append(k, v)
        kv.output(prob)
        kv.v_scale = kv.v_scale.clone()                                  # (the append writes to the new one from here on)
    old.fill_(float("nan"))
    assert torch.equal(kv.output(prob), fresh.output(prob))


ALLOCATOR = """
#include <cuda_runtime.h>
#include <sys/types.h>
extern "C" {
int PyGILState_Check(void);
int calls = 0, locked = 0;
void* take(ssize_t size, int, cudaStream_t) { void* p = nullptr; ++calls; locked += PyGILState_Check(); return cudaMalloc(&p, size ? size : 1) == cudaSuccess ? p : nullptr; }
void give(void* p, ssize_t, int, cudaStream_t) { cudaFree(p); }
}
"""
LOCK_CHILD = """
import ctypes, sys
sys.path.insert(0, {root!r})
import torch
torch.cuda.memory.change_current_allocator(torch.cuda.memory.CUDAPluggableAllocator({lib!r}, "take", "give"))
import paper_2505_00232_b200 as P
from tests.test_native_binding import tensor_calls
count = [ctypes.c_int.in_dll(ctypes.CDLL({lib!r}), n) for n in ("calls", "locked")]
for name, call in tensor_calls(P).items():
    before = [c.value for c in count]
    kept = call()
    after = [c.value for c in count]
    assert after[0] > before[0] and after[1] == before[1], (name, before, after)
torch.cuda.synchronize()
"""


def tensor_calls(P):
    """One call of every kind that allocates its outputs."""
    import torch
    rng = np.random.default_rng(1)
    f16 = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float16)).cuda()
    mk = lambda N, K, bits, group: P.QLinear.from_weights(*C.layer_weights(5, C.LayerSpec("t", N, K, bits, group, *((-8, 7) if bits == 4 else (-128, 127)))), bits, group, device="cuda:0")
    a, b, table, kv, wide = mk(256, 512, 8, 0), mk(256, 512, 8, 0), mk(1000, 128, 4, 32), P.KVHeads(2, 1280, 64), P.KVCache(4096, 1024)
    kv.append(f16(2, 9, 64), f16(2, 9, 64))
    x, g, ids, pos, ang = f16(5, 512), f16(512), torch.tensor([3, 999], device="cuda", dtype=torch.int32), torch.arange(6, device="cuda", dtype=torch.int32), torch.rand((16, 32), device="cuda")
    q, k, v, rows, prob, many = f16(6, 256), f16(6, 128), f16(6, 128), f16(2, 4, 64), f16(2, 4, 1280), f16(1024, 4096)
    return {"forward": lambda: a.forward(x), "forward_a8": lambda: a.forward_a8(x), "forward_group": lambda: P.qlinear_forward_group([a, b], x),
            "forward_gated": lambda: P.qlinear_forward_gated(a, b, x), "residual_rmsnorm": lambda: P.qlinear_residual_rmsnorm(x, x, g, 1e-5),
            "rope_qkv": lambda: P.qlinear_rope_qkv(q, k, v, pos, ang, ang, 1, 6, 4, 2, 64), "embed": lambda: table.embed(ids), "kv_scores": lambda: kv.scores(rows),
            "kv_scores_one": lambda: kv.heads[1].scores(rows[1]), "kv_output_heads": lambda: kv.output(prob), "kv_output": lambda: kv.heads[0].output(prob[0]),
            "kv_output, rows scaled by a pass of their own": lambda: wide.output(many)}


@pytest.mark.gpu
def test_outputs_are_allocated_without_the_interpreter_lock(P, tmp_path):
    """An allocation may have to go to the driver; other Python threads run meanwhile."""
    import os
    import subprocess
    import sys
    root, src, lib = os.path.dirname(os.path.dirname(os.path.abspath(__file__))), tmp_path / "alloc.cpp", str(tmp_path / "alloc.so")
    src.write_text(ALLOCATOR)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-shared", "-fPIC", f"-I{cuda}/include", str(src), "-o", lib, f"-L{cuda}/lib64", "-lcudart"], check=True)
    subprocess.run([sys.executable, "-c", LOCK_CHILD.format(root=root, lib=lib)], check=True, cwd=root, timeout=600)


def _modes(torch, fn):
    """Calls of fn(x) that an operator-level observer would see, by name."""
    from torch._subclasses.fake_tensor import FakeTensorMode
    from torch.overrides import TorchFunctionMode
    from torch.utils._python_dispatch import TorchDispatchMode

    class Dispatch(TorchDispatchMode):
        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            seen.append(str(func))
            return func(*args, **(kwargs or {}))

    class Function(TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            seen.append(getattr(func, "__name__", str(func)))
            return func(*args, **(kwargs or {}))

    def under(mode):
        def call(x):
            with mode():
                return fn(x)
        return call
    seen = []
    return seen, {"dispatch mode": under(Dispatch), "function mode": under(Function), "fake tensors": under(lambda: FakeTensorMode(allow_non_fake_inputs=True)), "vmap": lambda x: torch.vmap(lambda r: fn(r[None])[0])(x),
                  "jvp": lambda x: torch.func.jvp(fn, (x,), (x,)), "vjp": lambda x: torch.func.vjp(fn, x)[0], "functionalize": lambda x: torch.func.functionalize(fn)(x),
                  "trace": lambda x: torch.jit.trace(fn, (x,), check_trace=False).inlined_graph.findNode("aten::new_empty") is not None}


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["dispatch mode", "function mode", "fake tensors", "vmap", "jvp", "vjp", "functionalize", "trace"])
def test_calls_that_something_observes_are_left_to_python(P, monkeypatch, mode):
    """Modes, transforms and tracing see the allocations of the Python half (or its error): the native half takes none of these calls."""
    import torch
    lin = P.QLinear.from_weights(*C.layer_weights(5, C.LayerSpec("t", 64, 512, 8, 0, -128, 127)), 8, 0, device="cuda:0")
    x, native, answers = torch.ones((3, 512), device="cuda").half(), P.binding._bind_torch(), []

    class Recorded:
        def __getattr__(self, name):
            def call(*a):
                answers.append(getattr(native, name)(*a) if real else None)
                return answers[-1]
            return call
    monkeypatch.setattr(P.binding, "_native", Recorded())

    def outcome():
        seen, calls = _modes(torch, lin.forward)
        try:
            y = calls[mode](x)
        except Exception as e:
            return type(e), str(e), seen
        return [t.shape if isinstance(t, torch.Tensor) else t for t in (y if isinstance(y, tuple) else (y,))], seen
    real = True
    lin.forward(x)
    assert answers.pop() is not None                                     # (the same call without an observer)
    with_native = outcome()
    assert answers and all(a is None for a in answers)
    real = False
    assert outcome() == with_native


@pytest.mark.gpu
def test_common_calls_are_taken_by_the_native_half(P, monkeypatch):
    """None means "Python's": without this check a native half that takes nothing would go unnoticed.  Same bits from both, the product over
    more than 256 channels (whose scaled rows need a buffer) and single caches between appends among them."""
    import torch
    native, taken = P.binding._bind_torch(), []

    class Recorded:
        def __getattr__(self, name):
            def call(*a):
                taken.append((name, getattr(native, name)(*a) if real else None))
                return taken[-1][1]
            return call
    monkeypatch.setattr(P.binding, "_native", Recorded())
    real = True
    calls = tensor_calls(P)
    out = []
    for name, call in calls.items():
        taken.clear()
        out.append(call())
        assert len(taken) == 1 and taken[0][1] is not None, name
    assert {n for n in dir(native) if not n.startswith("_")} - {"init", "built_for", "kv_append"} == {n.split(",")[0] for n in calls}

    def cache():
        g = torch.Generator(device="cuda").manual_seed(3)
        f16 = lambda *s: torch.randn(s, generator=g, device="cuda").half()
        kv, heads, y = P.KVCache(256, 64), P.KVHeads(2, 256, 64), []
        for n in (5, 1, 70):
            kv.append(f16(n, 64), f16(n, 64))
            heads.append(f16(2, n, 64), f16(2, n, 64))
            for R in (2, 40):
                prob = f16(2, R, 256)
                prob[:, :, kv.length:] = 0
                y += [kv.scores(f16(R, 64)), kv.output(prob[0]), heads.scores(f16(2, R, 64))] + ([heads.output(prob)] if R <= 8 else [])
        return y
    fast = cache()
    assert taken and all(r is not None for _, r in taken) and {"kv_append", "kv_output", "kv_output_heads", "kv_scores_one"} <= {n for n, _ in taken}
    real = False
    slow = cache() + [call() for call in calls.values()]
    flat = lambda ys: [t for y in ys for t in (y if isinstance(y, (list, tuple)) else [y])]
    fast, slow = flat(fast + out), flat(slow)
    assert len(fast) == len(slow) and all(torch.equal(a, b) for a, b in zip(fast, slow))


@pytest.mark.gpu
def test_both_halves_agree(P, monkeypatch):
    import torch
    native = P.binding._bind_torch()

    class Python:                                                        # leaves every call to the Python half
        def __getattr__(self, name):
            return lambda *a: None
    rng = np.random.default_rng(5)
    f16 = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float16)).cuda()
    mk = lambda N, K, bits, group: P.QLinear.from_weights(*C.layer_weights(5, C.LayerSpec("t", N, K, bits, group, *((-8, 7) if bits == 4 else (-128, 127)))), bits, group, device="cuda:0")
    lins, gate, up, table = [mk(N, 512, 8, 0) for N in (256, 64, 64)], mk(256, 512, 4, 32), mk(256, 512, 4, 32), mk(1000, 128, 4, 32)
    pos, ang = torch.arange(6, device="cuda", dtype=torch.int32), torch.rand((16, 32), device="cuda")

    def calls():
        out, kv = [], P.KVHeads(2, 1280, 64)
        for M in (1, 5, 40, 300):
            x = inputs[M]
            out += [lins[0].forward(x), *P.qlinear_forward_group(lins, x), P.qlinear_forward_gated(gate, up, x, "silu"), *P.qlinear_residual_rmsnorm(x, x, x[0].contiguous(), 1e-5)]
            o = torch.empty((M, 256), device="cuda", dtype=torch.float16)
            assert lins[0].forward(x, out=o, stream=torch.cuda.current_stream()) is o and P.qlinear_forward_gated(gate, up, x, "gelu_tanh", out=o) is o
            h, y = P.qlinear_residual_rmsnorm(x, None, x[0].contiguous(), 1e-5, 1, y_out=o2(M), want_h=False)
            assert h is None
            out += [o, y]
            if M <= 8 or M > 128:
                out.append(lins[0].forward_a8(x))
        q, k, v = P.qlinear_rope_qkv(inputs["q"], inputs["k"], inputs["v"], pos, ang, ang, 1, 6, 4, 2, 64)
        kv.append(k, v)
        kv.append(k, v)
        assert kv.length == 12 == kv.heads[1].length
        for R in (4, 64):
            prob = inputs["prob"][:, :R].contiguous()
            out += [kv.scores(inputs["rows"][:, :R].contiguous()), kv.heads[1].scores(inputs["rows"][1, :R]), kv.heads[0].output(prob[0])] + ([kv.output(prob)] if R <= 8 else [])
        return out + [q, k, v, table.embed(inputs["ids"])]

    o2 = lambda M: torch.empty((M, 512), device="cuda", dtype=torch.float16)
    inputs = {M: f16(M, 512) for M in (1, 5, 40, 300)}
    inputs.update(q=f16(6, 256), k=f16(6, 128), v=f16(6, 128), rows=f16(2, 64, 64), prob=f16(2, 64, 1280), ids=torch.tensor([3, 999, -1, 1000], device="cuda", dtype=torch.int32))
    fast = calls()
    monkeypatch.setattr(P.binding, "_native", Python())
    slow = calls()
    monkeypatch.setattr(P.binding, "_native", native)
    assert len(fast) == len(slow) and all(a.dtype == b.dtype and a.shape == b.shape and torch.equal(a, b) for a, b in zip(fast, slow))
    for bad in (f16(3, 511), f16(3, 512).t(), f16(3, 512).float()):
        with pytest.raises(P.QLinearError) as e:
            lins[0].forward(bad)
        assert e.value.status == P.QL_ERR_INVALID_ARG
    with pytest.raises(P.QLinearError):
        lins[0].forward(inputs[1], out=torch.empty((2, 256), device="cuda", dtype=torch.float16))
    gate.close()
    with pytest.raises(P.QLinearError):
        gate.forward(inputs[1])
