"""What the binding refuses before any launch: tensors that do not match the
shape, type or device that the kernels will read or write.  No GPU needed: the
checks come before the one for a CUDA device, or are called on their own."""
import pytest
import torch

from paper_2607_13500_gb300 import api


def _bound(seqlens=(3, 4), d=16, dtype=torch.bfloat16):
    b = object.__new__(api._Bound)
    b.seqlens, b._total, b.d, b.dtype = list(seqlens), sum(seqlens), d, dtype
    b.d_k = torch.zeros(len(seqlens), dtype=torch.int32)
    b.stride, b._cu, b._tok = "alg1", None, None
    return b


@pytest.mark.parametrize("shape,dtype", [
    ((7, 32), torch.bfloat16), ((7, 8), torch.bfloat16), ((7, 16), torch.float32), ((7, 16), torch.float16),
    ((6, 16), torch.bfloat16), ((8, 16), torch.bfloat16), ((1, 6, 16), torch.bfloat16), ((2, 4, 16), torch.bfloat16),
    ((1, 7, 32), torch.bfloat16), ((1, 7, 16), torch.float32), ((16,), torch.bfloat16), ((), torch.bfloat16)])
def test_bound_tokens_of_another_shape_or_type(shape, dtype):
    # outputs and scratch were allocated for [7, 16] bf16
    x = torch.zeros(shape, dtype=dtype)
    with pytest.raises(ValueError, match=r"sum to|\[7, 16\]|\[B, N, D\]"):
        _bound()._bind(x, None, x)


@pytest.mark.gpu
@pytest.mark.parametrize("cls", ["Reducer", "Pipeline"])
def test_refused_before_any_launch(cls):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2607_13500_gb300 as altr
    obj = getattr(altr, cls)([40, 24], 64, torch.bfloat16, "cuda", k=4)
    call = obj.run if cls == "Reducer" else obj.submit
    mk = lambda *s, dt=torch.bfloat16: torch.randn(*s, device="cuda").to(dt)
    for bad in (mk(64, 128), mk(64, 32), mk(64, 64, dt=torch.float32), mk(1, 60, 64), mk(2, 32, 128)):
        with pytest.raises(ValueError):
            call(bad, bad, bad)
    good = mk(64, 64)
    r = call(good, good, good)
    torch.cuda.synchronize()
    assert r.status.tolist()[3] == 0 and r.y.shape == (8, 64)


def test_bound_tokens_on_another_device():
    x = torch.zeros(7, 16, dtype=torch.bfloat16, device="meta")
    with pytest.raises(ValueError, match=r"\[7, 16\]"):
        _bound()._bind(x, None, x)


def test_bound_tokens_that_match():
    x = torch.zeros(7, 16, dtype=torch.bfloat16)
    with pytest.raises(ValueError, match="CUDA device"):  # the next check
        _bound()._bind(x, None, x)


def _kept(**over):
    a = dict(idx=torch.arange(9, dtype=torch.int32), cu_k=[0, 4, 9], w=torch.zeros(48, 32, dtype=torch.bfloat16),
             bias=torch.zeros(48), error=torch.zeros(1, dtype=torch.int32))
    a.update(over)
    return a


KEPT_REFUSED = {
    "narrow_w": dict(w=torch.zeros(48, 16, dtype=torch.bfloat16)),
    "wide_w": dict(w=torch.zeros(48, 64, dtype=torch.bfloat16)),
    "flat_w": dict(w=torch.zeros(48 * 32, dtype=torch.bfloat16)),
    "int64_idx": dict(idx=torch.arange(9)),
    "short_idx": dict(idx=torch.arange(8, dtype=torch.int32)),
    "strided_idx": dict(idx=torch.arange(18, dtype=torch.int32)[::2]),
    "short_bias": dict(bias=torch.zeros(47)),
    "short_offsets": dict(cu_k=[0, 9]),
    "long_offsets": dict(cu_k=[0, 4, 9, 9]),
    "float_error": dict(error=torch.zeros(1)),
    "empty_error": dict(error=torch.zeros(0, dtype=torch.int32)),
}


@pytest.mark.parametrize("name", KEPT_REFUSED)
def test_project_kept_operands(name):
    api._check_kept(2, 32, torch.device("cpu"), **_kept())
    api._check_kept(2, 32, torch.device("cpu"), **_kept(bias=None, error=None))
    with pytest.raises(ValueError):
        api._check_kept(2, 32, torch.device("cpu"), **_kept(**KEPT_REFUSED[name]))


@pytest.mark.gpu
@pytest.mark.parametrize("k", [9, 4000], ids=["few_rows", "many_rows"])
def test_project_kept_refuses_before_any_launch(k):
    # on either side of the number of rows from which they are copied first
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2607_13500_gb300 as altr
    n = 2500
    x = torch.randn(2 * n, 32, device="cuda").to(torch.bfloat16)
    good = _kept(idx=torch.arange(k, dtype=torch.int32) % n, cu_k=[0, k // 2, k], w=torch.zeros(1024, 32, dtype=torch.bfloat16),
                 bias=torch.zeros(1024))
    on = lambda a: {n: v.cuda() if isinstance(v, torch.Tensor) else v for n, v in a.items()}
    call = lambda a: altr.project_kept(x, a["idx"], a["cu_k"], a["w"], a["bias"], seqlens=[n, n], error=a["error"])
    for bad in (dict(w=torch.zeros(1024, 16, dtype=torch.bfloat16)), dict(idx=good["idx"].long()), dict(idx=good["idx"][1:]),
                dict(bias=torch.zeros(1000)), dict(cu_k=[0, k]), dict(error=torch.zeros(1))):
        with pytest.raises(ValueError):
            call(on({**good, **bad}))
    z, err = call(on(good))
    torch.cuda.synchronize()
    assert z.shape == (k, 1024) and err.item() == 0 and not bool(z.any())


def test_bias_length():
    api._check_bias(None, 8, "b")
    api._check_bias(torch.zeros(8), 8, "b")
    with pytest.raises(ValueError, match="b must hold 8"):
        api._check_bias(torch.zeros(7), 8, "b")


@pytest.mark.gpu
def test_dense_layers_refuse_short_biases_and_other_error_buffers():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2607_13500_gb300 as altr
    w = torch.randn(64, 32, device="cuda").to(torch.bfloat16)
    b64, b32, y = torch.zeros(64, device="cuda"), torch.zeros(32, device="cuda"), torch.ones_like(w)
    for b1, b2 in ((b32, b32), (b64, b32[1:])):
        with pytest.raises(ValueError):
            altr.Mlp(64, w, w.t(), b1, b2)
    for kw in (dict(bias=b32), dict(error=torch.zeros(1, device="cuda")), dict(error=torch.zeros(1, dtype=torch.int32))):
        with pytest.raises(ValueError):
            altr.project(y, w, **kw)
    assert altr.Mlp(64, w, w.t(), b64, b32).run(y).error.item() == 0
    assert altr.project(y, w, b64)[1].item() == 0


@pytest.mark.parametrize("budget", [
    ([2], [0, 1], [0, 2, 5]), ([2, 3], [0], [0, 2, 5]), ([2, 3], [0, 1], [0, 5]), ([2, 3], [0, 1], [0, 2, 5, 5]),
    ([2, 4], [0, 1], [0, 2, 5]), ([2, 3], [0, 1], [-1, 2, 5]), ([6, 0], [0, 0], [0, 0, 5])])
def test_explicit_budgets_keep_to_the_outputs(budget):
    with pytest.raises(ValueError, match="budget"):
        api._budget_of(budget, [7, 7], None, None, (1, 3))


def test_explicit_budgets_that_fit():
    for budget in (([2, 3], [0, 1], [0, 2, 5]), ([0, 5], [0, 5], [0, 0, 5]), ([2, 3], [0, 1], [0, 4, 9])):
        assert api._budget_of(budget, [7, 7], None, None, (1, 3)) == budget
