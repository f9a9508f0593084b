"""The native call path of Plan's methods (_native.so) against the functions it stands in for: the regular call gives the
same bytes, and every other call (views, strides, wrong buffers, CPU tensors) is handed on to the Python path."""
import pytest
import torch

from paper_2504_13989_b200 import Plan, binding, synth
from paper_2504_13989_b200 import build as gbs_build

DEV = "cuda:0"


def test_irregular_calls_are_handed_on():
    gbs_build.build()
    nat = binding.native()
    x = torch.zeros(2, 128)
    assert nat.rotate_quantize(None, x, False, None, None) is None          # no plan
    assert nat.rotate_quantize(0, x, False, None, None) is None             # null plan
    assert nat.dequantize(0, x, x, False, torch.float32, None, None) is None
    assert nat.quantized_matmul(0, x, x, 0, x, x, torch.float32, None, None) is None
    assert nat.clip_error(0, x, [0.5], None) is None
    with pytest.raises(ValueError):
        nat.Calls(0, None)


@pytest.mark.gpu
def test_native_and_python_paths_agree():
    gbs_build.build()
    w = synth.WORKLOADS["llama4096"]
    x = synth.make_host("llama4096", 8).to(DEV)
    wide = torch.zeros(8, 2 * w.d, dtype=torch.bfloat16, device=DEV)
    wide[:, :w.d] = x
    with Plan(w.d, w.d_pad, w.m, 4, 0, w.alpha) as plan:
        ref = plan.alloc_outputs(8, DEV, True)
        binding.gbs_rotate_quantize(plan.handle, x, *ref)
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        for args in (dict(x=x), dict(x=x.view(2, 4, w.d)), dict(x=wide[:, :w.d]), dict(x=x, want_y=True), dict(x=x, stream=s),
                     dict(x=x, out=plan.alloc_outputs(8, DEV)), dict(x=wide.view(2, 4, -1)[..., :w.d]), dict(x=x[0])):
            codes, scales, y = plan.rotate_quantize(**args)
            torch.cuda.synchronize()
            n = codes.shape[0]
            assert torch.equal(codes, ref[0][:n]) and torch.equal(scales, ref[1][:n])
            assert (y is None) == (not args.get("want_y", False)) and (y is None or torch.equal(y, ref[2]))
        want = torch.empty((8, w.d), dtype=torch.bfloat16, device=DEV)
        binding.gbs_dequantize(plan.handle, ref[0], ref[1], 8, want, binding.GBS_INVERSE_ROTATE)
        assert torch.equal(plan.dequantize(ref[0], ref[1], inverse=True, dtype=torch.bfloat16), want)
        mm = torch.empty((8, 8), device=DEV)
        binding.gbs_quantized_matmul(plan.handle, ref[0], ref[1], plan.handle, ref[0], ref[1], mm)
        assert torch.equal(plan.quantized_matmul(ref[0], ref[1], plan, ref[0], ref[1]), mm)
        padded = torch.empty((8, 12), device=DEV)
        assert torch.equal(plan.quantized_matmul(ref[0], ref[1], plan, ref[0], ref[1], out=padded[:, :8]), mm)
        err = torch.zeros(3, dtype=torch.float64, device=DEV)
        plan.clip_error(x, [0.5, 0.75, 1.0], err_sum=err)
        # per-CTA fp64 totals are added in any order
        assert torch.allclose(plan.clip_error(x, torch.tensor([0.5, 0.75, 1.0])), err, rtol=1e-12)
        # errors are the Python path's
        for bad, exc in ((dict(x=x.cpu()), ValueError), (dict(x=x.half()), TypeError), (dict(x=x[:, :64]), ValueError),
                         (dict(x=x, out=plan.alloc_outputs(7, DEV)), ValueError)):
            with pytest.raises(exc):
                plan.rotate_quantize(**bad)
        with pytest.raises(TypeError):
            plan.dequantize(ref[0], ref[1], dtype=torch.float16)
        with pytest.raises(binding.GbsError):
            plan.clip_error(x, [1.5])


@pytest.mark.gpu
def test_methods_take_arguments_as_plan_declares_them():
    """The per-plan C methods parse like the Python methods they stand for, share their errors, and end with the plan."""
    gbs_build.build()
    x = synth.make_host("llama4096", 3).to(DEV)
    big = synth.make_host("llama4096", 700).to(DEV)
    with Plan(4096, bits=4, alpha=0.9) as plan:
        for rows in (x, big):
            codes, scales, y = plan.rotate_quantize(rows, True, None, None)
            c2, s2, y2 = plan.rotate_quantize(x=rows, want_y=True, stream=torch.cuda.current_stream())
            c3, s3, y3 = Plan.rotate_quantize(plan, rows)                  # the class's own method
            assert torch.equal(codes, c2) and torch.equal(scales, s2) and torch.equal(y, y2) and y3 is None
            assert torch.equal(codes, c3) and torch.equal(scales, s3)
            for t, shape, dtype in ((codes, (len(rows), 2048), torch.uint8), (scales, (len(rows), 1), torch.float32)):
                assert t.shape == shape and t.dtype == dtype and t.is_contiguous() and t.data_ptr() % 16 == 0
            a = plan.dequantize(codes, scales, True, torch.bfloat16)
            b = plan.dequantize(scales=scales, codes=codes, dtype=torch.bfloat16, inverse=True)
            assert torch.equal(a, b) and plan.dequantize(codes, scales).dtype == torch.float32
            out = torch.empty_like(a)
            assert plan.dequantize(codes, scales, inverse=True, out=out) is out and torch.equal(out, a)
            mm = plan.quantized_matmul(codes, scales, plan, codes, scales)
            assert torch.equal(mm, plan.quantized_matmul(codes, scales, plan_w=plan, codes_w=codes, scales_w=scales, dtype=torch.float32))
        assert plan.clip_error(x, alphas=[0.5, 1.0]).shape == (2,)
        err, per_row = plan.clip_error(x, [0.5, 1.0], want_rows=True)
        assert per_row.shape == (3, 2)
        for call in (lambda: plan.rotate_quantize(), lambda: plan.rotate_quantize(x, x=x), lambda: plan.rotate_quantize(x, wanty=1),
                     lambda: plan.rotate_quantize(x, False, None, None, 1), lambda: plan.dequantize(codes)):
            with pytest.raises(TypeError):
                call()
        kept = plan.rotate_quantize
    with pytest.raises(binding.GbsError):
        kept(x)

    class Mine(Plan):
        def rotate_quantize(self, x, **kw):
            return "mine"
    with Mine(4096) as plan:
        assert plan.rotate_quantize(x) == "mine" and plan.dequantize(codes, scales).shape == (700, 4096)


def test_native_methods_bind_like_functions():
    """The method objects over Plan's functions: they bind to whatever object they are looked up on, keep it alive, show the
    function's name and signature, and hand on what is not a regular call -- here on a stand-in without a plan."""
    import functools
    import gc
    import inspect
    import weakref
    gbs_build.build()
    nat = binding.native()
    for name, f in binding._PYTHON_METHODS.items():
        m = Plan.__dict__[name]
        assert type(m).__name__ == "Method" and m.__wrapped__ is f and m.__name__ == name
        assert inspect.signature(getattr(Plan, name)) == inspect.signature(f) and m.__doc__ == f.__doc__

    class Other:
        clip_error = nat.method("clip_error", lambda self, x, alphas, want_rows=False: (self, x, alphas, want_rows), None)

    class Derived(Other):
        def clip_error(self, x, alphas):
            return super().clip_error(x, alphas=alphas, want_rows=True)

    o, d = Other(), Derived()
    assert o.clip_error(1, 2) == (o, 1, 2, False) and d.clip_error(1, 2) == (d, 1, 2, True) and Other.clip_error(o, 1, 2)[0] is o
    with pytest.raises(TypeError):
        o.clip_error(1)
    kept, ref = functools.partial(o.clip_error, 1), weakref.ref(o)
    del o
    gc.collect()
    assert ref() is not None and kept(2)[0] is ref()                          # a bound method owns its object
    del kept
    gc.collect()
    assert ref() is None
    with pytest.raises(ValueError):
        nat.method("close", None, None)


@pytest.mark.gpu
def test_a_method_outlives_the_name_of_its_plan():
    import functools
    import gc
    gbs_build.build()
    x = synth.make_host("llama4096", 3).to(DEV)
    with Plan(4096, bits=4, alpha=0.9) as plan:
        codes, scales, _ = plan.rotate_quantize(x)
        rows = plan.dequantize(codes, scales, inverse=True)
        mm = plan.quantized_matmul(codes, scales, plan, codes, scales)
        err = plan.clip_error(x, [0.5, 1.0])
    assert torch.equal(Plan(4096, bits=4, alpha=0.9).rotate_quantize(x)[0], codes)
    quantize, restore = Plan(4096, bits=4, alpha=0.9).rotate_quantize, functools.partial(Plan(4096, bits=4).dequantize, inverse=True)
    multiply, score = Plan(4096, bits=4).quantized_matmul, Plan(4096, bits=4).clip_error
    gc.collect()
    assert torch.equal(quantize(x)[0], codes) and torch.equal(restore(codes, scales), rows)
    assert torch.equal(multiply(codes, scales, Plan(4096, bits=4), codes, scales), mm)
    assert torch.allclose(score(x, [0.5, 1.0]), err, rtol=1e-12)


@pytest.mark.gpu
def test_a_method_replaced_on_the_class_reaches_plans_that_exist(monkeypatch):
    gbs_build.build()
    x = synth.make_host("llama4096", 3).to(DEV)
    with Plan(4096) as plan:
        original = Plan.rotate_quantize
        calls = []
        monkeypatch.setattr(Plan, "rotate_quantize", lambda self, *a, **k: calls.append(self) or original(self, *a, **k))
        codes, scales, _ = plan.rotate_quantize(x)
        assert calls == [plan] and codes.shape == (3, 2048)
        monkeypatch.undo()
        plan.rotate_quantize(x)
        assert calls == [plan]
        # outputs come from the plan's alloc_outputs, whoever replaced it
        pool = plan.alloc_outputs(3, DEV)
        plan.alloc_outputs = lambda n_rows, device, want_y=False: pool
        got = plan.rotate_quantize(x)
        assert got[0] is pool[0] and got[1] is pool[1] and torch.equal(got[0], codes)

    class Pooled(Plan):
        def alloc_outputs(self, n_rows, device, want_y=False):
            return pool
    with Pooled(4096) as plan:
        assert plan.rotate_quantize(x)[0] is pool[0]


@pytest.mark.gpu
def test_tensors_without_memory_are_refused():
    """A batched tensor's data pointer throws in C++, a fake tensor's is null: the call is handed to the Python path, which raises,
    and the process lives."""
    from torch._subclasses.fake_tensor import FakeTensorMode
    gbs_build.build()
    x = synth.make_host("llama4096", 2).to(DEV)
    with Plan(4096) as plan:
        codes, scales, _ = plan.rotate_quantize(x)
        out, rows, mm = plan.alloc_outputs(1, DEV), torch.empty(1, 4096, device=DEV), torch.empty(1, 1, device=DEV)
        for call in (lambda r, c, s: plan.rotate_quantize(r)[0], lambda r, c, s: plan.rotate_quantize(r, out=out)[0],
                     lambda r, c, s: plan.clip_error(r, [0.5]), lambda r, c, s: plan.dequantize(c[None], s[None]),
                     lambda r, c, s: plan.quantized_matmul(c[None], s[None], plan, c[None], s[None], out=mm)):
            with pytest.raises(RuntimeError):
                torch.vmap(call)(x, codes, scales)
        mode = FakeTensorMode()
        fx, fc, fs = (mode.from_tensor(t) for t in (x, codes, scales))
        for call in (lambda: plan.rotate_quantize(fx, out=plan.alloc_outputs(2, DEV)), lambda: plan.dequantize(fc, fs)):
            with pytest.raises(Exception):
                call()
        torch.cuda.synchronize()
        assert torch.equal(plan.rotate_quantize(x)[0], codes)


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [1, 3, 700])
def test_outputs_have_storages_of_their_own(rows):
    """Codes and scales are saved, kept, resized and freed each by itself."""
    gbs_build.build()
    x = synth.make_host("llama4096", rows).to(DEV)
    with Plan(4096, bits=4) as plan:
        codes, scales, y = plan.rotate_quantize(x, want_y=True)
        outs = (codes, scales, y, plan.dequantize(codes, scales), plan.quantized_matmul(codes, scales, plan, codes, scales))
        assert len({t.untyped_storage().data_ptr() for t in outs}) == len(outs)
        for t in outs:
            assert t.storage_offset() == 0 and t.untyped_storage().nbytes() == t.numel() * t.element_size()
        want = scales.clone()
        codes.untyped_storage().resize_(0)
        assert torch.equal(scales, want)
