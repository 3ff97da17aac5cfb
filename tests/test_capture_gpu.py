"""Calls captured into a CUDA graph behind a join: the work before the call's
first kernel (which carries the programmatic launch attribute) is a copy on a
second stream, alone or beside a kernel of the capturing stream.  A replay on
refilled inputs gives what the call gives outside a capture, bit for bit.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2607_13500_gb300 import _build
    _build.build()


def _bf16(g, *shape):
    return torch.randn(*shape, generator=g).to(torch.bfloat16)


def _call(kind):
    """(device inputs, two sets of host inputs, the call as inputs -> outputs)."""
    import paper_2607_13500_gb300 as altr
    g = torch.Generator().manual_seed(len(kind))
    if kind in ("mlp", "project", "kept"):
        t, d, dh = 576, 256, 1024
        host = [(_bf16(g, t, d).pin_memory(),) for _ in range(2)]
        w1, w2 = (_bf16(g, dh, d) / 16).cuda(), (_bf16(g, d, dh) / 32).cuda()
        if kind == "mlp":
            m = altr.Mlp(t, w1, w2, act="quick_gelu", scores=True)

            def call(x):
                o = m.run(x, x)
                return [o.h, o.x_post, o.x, o.stats, o.h2, o.s, o.error]
        elif kind == "project":
            def call(x):
                return list(altr.project(x, w1))
        else:
            idx = torch.arange(0, t, 3, dtype=torch.int32, device="cuda")

            def call(x):
                return list(altr.project_kept(x, idx, [0, idx.numel()], w1))
    else:
        seqlens = {"one": [576], "clip": [5200], "ragged": [300, 17, 900], "reduce": [200, 200]}[kind]
        d = 128
        host = [tuple(_bf16(g, sum(seqlens), d).pin_memory() for _ in range(3)) for _ in range(2)]
        if kind == "reduce":  # the one-line call, which allocates and uploads its budgets
            def call(x, xp, xq):
                r = altr.reduce(x, xp, xq, seqlens=seqlens, ratio=(2, 9), scores=True)
                return [r.y, r.idx, r.h2, r.s]
        else:
            red = altr.Reducer(seqlens, d, torch.bfloat16, "cuda", ratio=(2, 9), scores=True)

            def call(x, xp, xq):
                r = red.run(x, xp, xq)
                return [r.y, r.idx, r.h2, r.s]
    dev = tuple(torch.empty_like(h, device="cuda") for h in host[0])
    return dev, host, call


@pytest.mark.parametrize("beside", [False, True], ids=["copy", "copy_and_kernel"])
@pytest.mark.parametrize("kind", ["one", "clip", "ragged", "reduce", "mlp", "project", "kept"])
def test_call_behind_a_join(kind, beside):
    dev, host, call = _call(kind)
    want = []
    for h in host:
        for a, b in zip(dev, h):
            a.copy_(b)
        want.append([v.clone() for v in call(*dev)])
    torch.cuda.synchronize()
    staged = [h.clone().pin_memory() for h in host[0]]
    other = torch.zeros(1 << 16, device="cuda")
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cap = torch.cuda.current_stream()
        side.wait_stream(cap)
        with torch.cuda.stream(side):
            for a, b in zip(dev, staged):
                a.copy_(b, non_blocking=True)
        if beside:
            other.add_(1.0)
        cap.wait_stream(side)
        out = call(*dev)
    for i in (1, 0, 1):
        for a, b in zip(staged, host[i]):
            a.copy_(b)
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(out, want[i]):
            assert torch.equal(a, b)
    assert not beside or bool((other == 3.0).all())
