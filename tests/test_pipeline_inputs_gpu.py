"""Pipeline.submit on inputs that the binding has to copy first (3-D tensors
that are not contiguous): each submission's copies outlive its kernels, which
run on the pipeline's own streams."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_copied_inputs_outlive_their_submission():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2607_13500_gb300 as altr
    from paper_2607_13500_gb300 import _build
    _build.build()
    b, n, d = 64, 576, 1024
    g = torch.Generator(device="cuda").manual_seed(3)
    sets = [[torch.randn(n, b, d, generator=g, device="cuda").to(torch.bfloat16).transpose(0, 1) for _ in range(3)]
            for _ in range(3)]
    red = altr.Reducer([n] * b, d, torch.bfloat16, "cuda", k=96)
    want = [(r.y.clone(), r.idx.clone()) for r in (red.run(*(t.contiguous() for t in s)) for s in sets)]
    torch.cuda.synchronize()
    pipe = altr.Pipeline([n] * b, d, torch.bfloat16, "cuda", k=96)
    got = []
    for i in range(12):
        with torch.cuda.stream(pipe.select_stream):
            torch.cuda._sleep(3000000)  # the selections and copies fall behind the submissions
        r = pipe.submit(*sets[i % 3])
        with torch.cuda.stream(pipe.select_stream):
            got.append((r.y.clone(), r.idx.clone()))
    pipe.synchronize()
    torch.cuda.synchronize()
    for i, (y, idx) in enumerate(got):
        assert torch.equal(idx, want[i % 3][1]), i
        assert torch.equal(y, want[i % 3][0]), i
    pipe.close()
