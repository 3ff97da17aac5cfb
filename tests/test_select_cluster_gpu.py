"""The selection's fast path, in one CTA and in a cluster of CTAs per image,
against the oracle: the edges of its rules (5120 and 8192 tokens; 12, 36 and
72 images), images much smaller than the batch's largest, near-ties at the
cut and at the picks, and the inputs it leaves to select_image (exact ties
in numbers, crowded keys, rows outside the fp32 model).  Kept indices and
rows are compared bit for bit.
"""
import pytest
import torch

from test_parity_gpu import _near_tie_triples, _rows, check_reduce

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2607_13500_gb300 import _build
    _build.build()


def _budget(ks, k1s):
    cu = [0]
    for k in ks:
        cu.append(cu[-1] + k)
    return list(ks), list(k1s), cu


@pytest.mark.parametrize("batch,n,d,dtype", [
    # one CTA per image, up to 8192 tokens
    (3, 1, 64, torch.bfloat16), (3, 2, 64, torch.float16), (2, 511, 64, torch.bfloat16), (5, 513, 64, torch.float32),
    (200, 1025, 32, torch.bfloat16), (1, 5119, 128, torch.bfloat16), (37, 8192, 32, torch.bfloat16),
    # clusters
    (1, 5120, 128, torch.bfloat16), (1, 5121, 64, torch.float32), (3, 7001, 64, torch.float16),
    (12, 5123, 64, torch.bfloat16), (13, 5200, 64, torch.bfloat16), (36, 5120, 32, torch.float32),
    (37, 8193, 32, torch.bfloat16), (72, 8200, 32, torch.bfloat16), (1, 16384, 64, torch.bfloat16),
    (2, 16383, 32, torch.float32),
    # neither
    (73, 8193, 32, torch.bfloat16),
])
def test_sizes(batch, n, d, dtype):
    x, xp, xq = _rows(batch * n, d, 7 * n + batch, dtype)
    images = sorted({0, batch // 2, batch - 1})
    for k, k1, stride in [(max(1, n // 9), n // 27, "alg1"), (min(n, n // 3 + 1), n // 10, "interval")]:
        check_reduce(x, xp, xq, [n] * batch, _budget([k] * batch, [k1] * batch), images=images, stride=stride)


def test_ragged_sizes():
    for seqlens in ([2560, 1, 16384, 255, 0, 7000, 16, 513], [600, 1, 4000, 0, 17]):
        _ragged(seqlens)


def _ragged(seqlens):
    x, xp, xq = _rows(sum(seqlens), 64, 5, torch.bfloat16)
    ks = [max(1, 2 * n // 9) if n else 0 for n in seqlens]
    check_reduce(x, xp, xq, seqlens, _budget(ks, [k // 3 for k in ks]))


@pytest.mark.parametrize("n", [700, 6000])
def test_budgets(n):
    x, xp, xq = _rows(n, 128, 11, torch.bfloat16)
    for k, k1 in [(1, 0), (1, 1), (2, 1), (n, n // 3), (n, 0), (n, n), (n - 1, n - 1), (n // 2, n // 2), (n - 1, 1),
                  (n // 4, 0)]:
        check_reduce(x, xp, xq, [n], _budget([k], [k1]))


@pytest.mark.parametrize("rows", [2500, 5500])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
def test_near_ties(dtype, rows):
    # triples that the fp32 keys leave uncertain and the double-float keys
    # separate, among ordinary rows: no exact sums are needed, wherever the cut
    # splits a triple and for dense and sparse picks
    d = 1024
    tx, tp, tq, *_ = _near_tie_triples(32, d, dtype, 3)
    x, xp, xq = (torch.cat([a, b]) for a, b in zip((tx, tp, tq), _rows(rows, d, 4, dtype)))
    perm = torch.randperm(x.shape[0], generator=torch.Generator().manual_seed(6))
    x, xp, xq = x[perm], xp[perm], xq[perm]
    n = x.shape[0]
    v = x.double()
    order = torch.argsort(v.abs().sum(1) ** 2 / (v * v).sum(1), descending=True)
    members = (perm[order] < 96).nonzero()[:, 0]  # places of the triples' rows by R
    for k1, k2, stride in [(int(members[31]), 400, "alg1"), (int(members[34]) + 1, 1200, "alg1"),
                           (int(members[60]), 701, "interval"), (0, 900, "interval")]:
        st = check_reduce(x, xp, xq, [n], _budget([k1 + k2], [k1]), stride=stride)
        assert st[2] == 0, st

    # exact ties: a few rows twice, one pair at the cut; their runs, and only
    # they, take exact sums
    pairs = [(int(order[members[20]]), 5)] + [(i, n - 1 - i) for i in range(40, 60)]
    for i, j in pairs:
        x[j], xp[j], xq[j] = x[i], xp[i], xq[i]
    v = x.double()
    r = v.abs().sum(1) ** 2 / (v * v).sum(1)
    place = int((r > r[5]).sum())  # the tied pair at the cut holds places `place` and `place` + 1 (in its run)
    for k1, k2 in [(place + 1, 1000), (0, n - 1)]:
        st = check_reduce(x, xp, xq, [n], _budget([k1 + k2], [k1]))
        assert 0 < st[2] <= 4 * len(pairs) + 8, st


@pytest.mark.parametrize("groups,rows,exact", [(40, 1900, True), (150, 1700, False), (150, 1700, True), (300, 1500, False),
                                               (300, 6000, True)],
                         ids=["40", "150", "150_exact", "300", "300_exact"])
def test_many_runs(groups, rows, exact):
    # every row a pick and hundreds of near-tie runs: in the small list, in the
    # large one (an eighth as many runs as rows) and more than it holds; some
    # with an exact tie, which alone take exact sums
    d = 1024
    t3 = _near_tie_triples(groups, d, torch.float32, 5)
    where = torch.argsort(t3[3])
    tx, tp, tq = t3[:3]
    ties = range(0, 3 * groups, 36) if exact else ()
    for i in ties:
        for t in (tx, tp, tq):
            t[where[i + 1]] = t[where[i]]
    x, xp, xq = (torch.cat([a, b]) for a, b in zip((tx, tp, tq), _rows(rows, d, 4, torch.float32)))
    perm = torch.randperm(x.shape[0], generator=torch.Generator().manual_seed(6))
    x, xp, xq = x[perm], xp[perm], xq[perm]
    n = x.shape[0]
    st = check_reduce(x, xp, xq, [n], _budget([n - 1], [0]))
    assert 2 * len(ties) <= st[2] <= 8 * len(ties), st


@pytest.mark.parametrize("n", [2600, 6000])
def test_left_to_select_image(n):
    d = 64
    base, bp, bq = _rows(n, d, 21, torch.bfloat16)

    def run(edit, k=600, k1=200, **kw):
        x, xp, xq = base.clone(), bp.clone(), bq.clone()
        edit(x, xp, xq)
        return check_reduce(x, xp, xq, [n], _budget([k], [k1]), **kw)

    def ties(x, xp, xq):  # every row four times, far apart
        for v in (x, xp, xq):
            v.copy_(v[:n // 4].repeat(4, 1))

    def equal(x, xp, xq):
        for v in (x, xp, xq):
            v.copy_(v[:1].expand(n, d).clone())

    def crowded(x, xp, xq):  # one far outlier: nearly all keys fall into one bucket
        x[7] = 0
        x[7, 0] = 1
        xq[9] = -xp[9]
        x[100:2400] = x[100:101] + 0.01 * torch.randn(2300, d, generator=torch.Generator().manual_seed(1)).to(x.dtype)

    def outside(x, xp, xq):
        x[3, 1] = float("nan")
        x[5] = 0
        xq[11, 0] = float("inf")
        xp[12] = 0
        x[13] = x[13] * 2.0 ** 70

    assert run(ties)[2] > 0
    run(equal)
    run(crowded)
    run(outside, expect_nonfinite=True)


@pytest.mark.parametrize("edge,exact", [(2.0 ** -50, False), (2.0 ** -51, True)], ids=["least", "below"])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16, torch.float32], ids=["bf16", "f16", "f32"])
def test_near_ties_at_the_value_range(dtype, edge, exact):
    # the double-float keys take rows of zeros and of values down to 2^-50,
    # and leave rows with a smaller one to exact sums; fp16's least value is
    # inside.  129 (bf16, fp16) or 258 chunks a row: partial rounds of a warp
    # group.
    if dtype == torch.float16:
        edge, exact = 2.0 ** -24, False
    x, xp, xq, *_ = _near_tie_triples(32, 1032, dtype, 8)
    for col, v in ((100, edge), (101, -edge), (102, 0.0), (103, -0.0), (1031, edge)):
        for t in (x, xp, xq):
            t[:, col] = v
    n = x.shape[0]
    for k, k1 in [(40, 31), (60, 0), (45, 16)]:
        st = check_reduce(x, xp, xq, [n], _budget([k], [k1]))
        assert (st[2] > 0) == exact, st


@pytest.mark.parametrize("rows", [1500, 5500])
def test_exact_sums_only_for_the_run_that_needs_them(rows):
    # every row a pick: a row outside the double-float keys' value range sends
    # its own near-tie run to exact sums, and no other
    d = 1024
    tx, tp, tq, shuffle, *_ = _near_tie_triples(32, d, torch.float32, 3)
    where = torch.argsort(shuffle)  # where[i]: the place of row i
    for t in (tp, tq):
        t[:, 7] = 0.0
        t[where[15:18], 7] = 2.0 ** -60  # below 2^-50, and far below what moves a key
    x, xp, xq = (torch.cat([a, b]) for a, b in zip((tx, tp, tq), _rows(rows, d, 4, torch.float32)))
    perm = torch.randperm(x.shape[0], generator=torch.Generator().manual_seed(6))
    x, xp, xq = x[perm], xp[perm], xq[perm]
    n = x.shape[0]
    st = check_reduce(x, xp, xq, [n], _budget([n - 1], [0]))
    assert 3 <= st[2] <= 8, st
