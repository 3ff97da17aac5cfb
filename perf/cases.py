"""The work that a program using this package has it do, as measurable cases.

Every case goes through the package's public entry points:

* ``reduce``   -- ``Reducer.run``: one batch of images reduced on the current
                  stream with the buffers the program keeps (an image, a batch,
                  tiles, a video clip, a ragged batch);
* ``stream``   -- ``Pipeline.submit``: one batch of a stream of batches;
* ``call``     -- ``reduce(...)``: the one-line call that allocates its outputs;
* ``mlp``      -- ``Mlp.run``: the encoder's last MLP with the scoring fused in;
* ``project``  -- ``project``: the projector's first layer on gathered rows;
* ``kept``     -- ``project_kept``: the same layer on rows read by kept index.

A case is a dict of plain values; ``listed()`` names twelve of them and
``draw(rng)`` gives others of the same ranges.  Inputs are drawn on the GPU
from the seed: clustered token features with a few activation outliers, the
MLP's output from a small random MLP, and x = x' + x''.
"""
import math

import torch

import paper_2607_13500_gb300 as altr

DEV = "cuda"
DTYPES = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}
LAM = (1, 3)


# ---------------------------------------------------------------- cases
def listed():
    return [
        # one image of a 336-pixel encoder in fp32, the smallest request of an
        # interactive program: latency and launches are what counts
        dict(name="image_f32", kind="reduce", n=576, images=1, d=1024, dtype="f32", k=64),
        # a served batch of ordinary images at the largest printed budget
        dict(name="batch_bf16", kind="reduce", n=576, images=64, d=4096, dtype="bf16", k=192),
        # five-tile images in half precision, with the real-valued stride and
        # the H2 and s outputs asked for
        dict(name="tiles_f16", kind="reduce", n=2880, images=4, d=4096, dtype="f16", k=320, stride="interval",
             scores=True),
        # one video clip of 32 frames x 196 tokens (similar frames: crowded keys)
        dict(name="clip_video", kind="reduce", n=6272, images=1, d=3584, dtype="bf16", num=1, den=8, frame=196),
        # dynamic-resolution images of 256 to 16384 tokens in one ragged batch
        dict(name="ragged_bf16", kind="reduce", n=16384, n_min=256, images=12, d=3584, dtype="bf16", num=2, den=9),
        # a stream of batches, each overlapping the next: the serving loop
        dict(name="stream_bf16", kind="stream", n=576, images=32, d=4096, dtype="bf16", k=192),
        # the one-line call on two odd-sized images, x' = x, nothing kept between calls
        dict(name="call_alias", kind="call", n=729, images=2, d=1152, dtype="bf16", k=81, alias=True),
        # the encoder's last MLP for one image: the latency of a single request
        dict(name="mlp_image", kind="mlp", t=576, d=1024, dh=4096, act="quick_gelu"),
        # the same for one five-tile image on an encoder of uneven widths, erf
        # GELU, no residual, with the scores
        dict(name="mlp_tiles", kind="mlp", t=2885, d=1152, dh=4304, act="gelu", resid=False, scores=True),
        # the same for a served batch of 64 images
        dict(name="mlp_batch", kind="mlp", t=36864, d=1024, dh=4096, act="quick_gelu"),
        # the projector's first layer on one image's kept tokens
        dict(name="project_image", kind="project", rows=192, d=1024, out=4096, act="gelu"),
        # the projector's first layer on a batch's kept tokens, read by index
        dict(name="kept_batch", kind="kept", n=576, images=64, d=1024, k=192, out=4096, act="gelu"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MAX_ELEMS = 64 * 576 * 4096   # elements of one token tensor of the largest reduction
MAX_MACS = 36864 * 1024 * 4096


def draw(rng):
    kind = rng.choice(["reduce", "reduce", "reduce", "stream", "call", "mlp", "mlp", "project", "kept"])
    if kind in ("reduce", "stream", "call"):
        dtype = rng.choice(["bf16", "bf16", "f16", "f32"])
        d = 8 * rng.randint(96, 512)
        n = _log_int(rng, 64, 16384 if kind == "reduce" else 4096)
        most = max(1, MAX_ELEMS // (n * d) // (2 if dtype == "f32" else 1))
        images = _log_int(rng, 1, min(most, 4 if kind == "call" else 128))
        c = dict(kind=kind, n=n, images=images, d=d, dtype=dtype)
        if rng.random() < 0.5:
            c["k"] = max(1, n // rng.randint(3, 12))
        else:
            c["num"], c["den"] = rng.choice([(1, 9), (2, 9), (1, 8), (1, 3)])
        if kind == "reduce" and images > 1 and "num" in c and rng.random() < 0.5:
            c["n_min"] = max(1, n // rng.randint(2, 64))
        if rng.random() < 0.25:
            c["stride"] = "interval"
        if rng.random() < 0.3:
            c["scores"] = True
        if rng.random() < 0.3:
            c["alias"] = True
        return c
    d = 16 * rng.randint(48, 80)
    act = rng.choice(["gelu", "quick_gelu", "none"])
    if kind == "mlp":
        dh = 16 * rng.randint(2 * d // 16, 4 * d // 16)
        t = _log_int(rng, 48, min(36864, MAX_MACS // (d * dh)))
        return dict(kind=kind, t=t, d=d, dh=dh, act=act, resid=rng.random() < 0.7, scores=rng.random() < 0.3)
    out = 16 * rng.randint(128, 256)
    if kind == "project":
        return dict(kind=kind, rows=_log_int(rng, 16, 12288), d=d, out=out, act=act)
    n = _log_int(rng, 64, 2880)
    k = max(1, n // rng.randint(3, 12))
    return dict(kind=kind, n=n, images=_log_int(rng, 1, max(1, 12288 // k)), d=d, k=k, out=out, act=act)


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _seqlens(case):
    """The images' token counts: equal, or spread unevenly over [n_min, n] with
    the largest present (the same for every seed: the sizes are the case's)."""
    n, b = case["n"], case["images"]
    lo = case.get("n_min")
    if not lo:
        return [n] * b
    g = torch.Generator().manual_seed(n * 131 + b)
    jit = torch.rand(b, generator=g).tolist()
    order = torch.randperm(b, generator=g).tolist()
    sizes = [min(n, max(lo, int(lo + (n - lo) * (i + 0.2 + 0.6 * j) / b))) for i, j in enumerate(jit)]
    sizes[b - 1] = n
    return [sizes[i] for i in order]


def _features(g, n, d, frame=0):
    """Clustered features of one image (a clip: one frame and its drift) with
    outlier channels on one token in a hundred."""
    m = max(1, min(64, -(-n // 48)))
    base = frame if frame else n
    centres = _randn(g, m, d)
    h = centres[torch.randint(0, m, (base,), generator=g, device=DEV)] + 0.1 * _randn(g, base, d)
    if frame:
        steps = 0.02 * _randn(g, n // frame, frame, d)
        steps[0] = 0.0
        h = (h + steps.cumsum(0)).reshape(n, d)
    hot = torch.randperm(n, generator=g, device=DEV)[:n // 100]
    if hot.numel():
        chans = torch.tensor(sorted({c % d for c in (7, 131, 509, 1021)}), device=DEV)
        h[hot[:, None], chans[None, :]] *= 20.0
    return h


def _token_tensors(case, seed, seqlens):
    g = _gen(seed)
    d, dt = case["d"], DTYPES[case["dtype"]]
    w1 = _randn(g, 64, d) / math.sqrt(d)
    w2 = _randn(g, d, 64) / 8.0
    t = sum(seqlens)
    x, xp, xq = (torch.empty(t, d, dtype=dt, device=DEV) for _ in range(3))
    off = 0
    for n in seqlens:
        h = _features(g, n, d, case.get("frame", 0))
        q = torch.nn.functional.gelu(h @ w1.T) @ w2.T
        x[off:off + n], xp[off:off + n], xq[off:off + n] = h + q, h, q
        off += n
    return x, (None if case.get("alias") else xp), xq


def _budget(case):
    return dict(k=case["k"]) if "k" in case else dict(ratio=(case["num"], case["den"]))


def _ks(case, seqlens):
    if "k" in case:
        return [case["k"]] * len(seqlens)
    return [max(1, n * case["num"] // case["den"]) for n in seqlens]


def _dense_weights(g, rows, cols):
    """nn.Linear weights [rows, cols] in bf16 and a small fp32 bias."""
    return (_randn(g, rows, cols) / math.sqrt(cols)).to(torch.bfloat16), 0.02 * _randn(g, rows)


def _mlp_inputs(case, seed):
    g = _gen(seed)
    t, d = case["t"], case["d"]
    xp = torch.cat([_features(g, min(576, t - o), d) for o in range(0, t, 576)]).to(torch.bfloat16)
    w1, b1 = _dense_weights(g, case["dh"], d)
    w2, b2 = _dense_weights(g, d, case["dh"])
    resid = xp.clone() if case.get("resid", True) else None
    return xp, resid, w1, b1, w2, b2


def _project_inputs(case, seed):
    g = _gen(seed)
    y = torch.cat([_features(g, min(576, case["rows"] - o), case["d"])
                   for o in range(0, case["rows"], 576)]).to(torch.bfloat16)
    w, b = _dense_weights(g, case["out"], case["d"])
    return y, w, b


def _kept_inputs(case, seed):
    g = _gen(seed)
    n, b, k = case["n"], case["images"], case["k"]
    x = torch.cat([_features(g, n, case["d"]) for _ in range(b)]).to(torch.bfloat16)
    keys = torch.rand(b, n, generator=g, device=DEV)
    idx = keys.argsort(1)[:, :k].sort(1).values.to(torch.int32).reshape(-1)  # ascending in each image
    w, bias = _dense_weights(g, case["out"], case["d"])
    return x, idx, [k * i for i in range(b + 1)], w, bias


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("reduce", "stream", "call"):
        seqlens = _seqlens(case)
        x, xp, xq = _token_tensors(case, seed, seqlens)
        opts = dict(lam=LAM, scores=bool(case.get("scores")), stride=case.get("stride", "alg1"), **_budget(case))
        if kind == "call":
            shape = (len(seqlens), case["n"], case["d"])
            x, xp, xq = (None if v is None else v.view(shape) for v in (x, xp, xq))
            return dict(kind=kind, x=x, xp=xp, xq=xq, opts=opts)
        cls = altr.Reducer if kind == "reduce" else altr.Pipeline
        obj = cls(seqlens, case["d"], x.dtype, x.device, alias_pre=xp is None, **opts)
        return dict(kind=kind, x=x, xp=xp, xq=xq, obj=obj)
    if kind == "mlp":
        xp, resid, w1, b1, w2, b2 = _mlp_inputs(case, seed)
        m = altr.Mlp(case["t"], w1, w2, b1, b2, act=case["act"], scores=bool(case.get("scores")))
        return dict(kind=kind, xp=xp, resid=resid, obj=m)
    err = torch.zeros(1, dtype=torch.int32, device=DEV)
    if kind == "project":
        y, w, b = _project_inputs(case, seed)
        out = torch.empty(case["rows"], case["out"], dtype=torch.bfloat16, device=DEV)
        return dict(kind=kind, y=y, w=w, b=b, out=out, err=err, act=case["act"])
    x, idx, cu_k, w, b = _kept_inputs(case, seed)
    return dict(kind=kind, x=x, idx=idx, cu_k=cu_k, w=w, b=b, err=err, act=case["act"],
                seqlens=[case["n"]] * case["images"])


# ---------------------------------------------------------------- one pass
def _reduced(r):
    out = dict(y=r.y, idx=r.idx)
    if r.h2 is not None:
        out.update(h2=r.h2, s=r.s)
    return out


def run(state):
    kind = state["kind"]
    if kind == "reduce":
        return _reduced(state["obj"].run(state["x"], state["xp"], state["xq"]))
    if kind == "stream":
        return _reduced(state["obj"].submit(state["x"], state["xp"], state["xq"]))
    if kind == "call":
        return _reduced(altr.reduce(state["x"], state["xp"], state["xq"], **state["opts"]))
    if kind == "mlp":
        o = state["obj"].run(state["xp"], state["resid"])
        out = dict(h=o.h, x_post=o.x_post, x=o.x, stats=o.stats, error=o.error)
        if o.h2 is not None:
            out.update(h2=o.h2, s=o.s)
        return out
    if kind == "project":
        z, err = altr.project(state["y"], state["w"], state["b"], act=state["act"], error=state["err"],
                              out=state["out"])
        return dict(z=z, error=err)
    z, err = altr.project_kept(state["x"], state["idx"], state["cu_k"], state["w"], state["b"], act=state["act"],
                               seqlens=state["seqlens"], error=state["err"])
    return dict(z=z, error=err)


# ---------------------------------------------------------------- what a pass needs
def work(case):
    """Each input read once, each output written once; multiply-adds as two."""
    kind = case["kind"]
    if kind in ("reduce", "stream", "call"):
        e = 4 if case["dtype"] == "f32" else 2
        seqlens = _seqlens(case)
        t, k, d = sum(seqlens), sum(_ks(case, seqlens)), case["d"]
        by = (2 if case.get("alias") else 3) * t * d * e + k * d * e + 4 * k
        if case.get("scores"):
            by += 8 * t
        return {"bytes": by, "flops": 10 * t * d}  # five sums of |x|, squares and products
    if kind == "mlp":
        t, d, dh = case["t"], case["d"], case["dh"]
        by = 2 * (t * d * (2 if case.get("resid", True) else 1) + 2 * d * dh) + 4 * (d + dh)
        by += 2 * (t * dh + 2 * t * d) + 32 * t + (8 * t if case.get("scores") else 0)
        return {"bytes": by, "flops": 4 * t * d * dh}
    rows = case["rows"] if kind == "project" else case["images"] * case["k"]
    d, out = case["d"], case["out"]
    return {"bytes": 2 * (rows * d + d * out + rows * out) + 4 * out + (4 * rows if kind == "kept" else 0),
            "flops": 2 * rows * d * out}


def tolerance(case):
    kind = case["kind"]
    if kind in ("reduce", "stream", "call"):
        # the selection and the copied rows are exact; H2 and s are fp32 values
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.0} if case.get("scores") else "exact"
    if kind == "mlp":
        # two chained bf16 GEMMs with a bf16 hidden layer: about 2.3e-3 from the
        # 64-bit result
        return {"rel": 1e-2, "max": 0.1, "differ": 0.0}
    return {"rel": 7e-3, "max": 0.05, "differ": 0.0}  # one bf16 layer: about 1.7e-3


# ---------------------------------------------------------------- 64-bit results
def _exact_reduce(case, seed):
    seqlens = _seqlens(case)
    x, xp, xq = _token_tensors(case, seed, seqlens)
    xp = x if xp is None else xp
    ys, ids, h2s, ss = [], [], [], []
    off = 0
    for n, k in zip(seqlens, _ks(case, seqlens)):
        h2, s = [], []
        for a in range(off, off + n, 4096):
            rows = slice(a, min(a + 4096, off + n))
            v, p, q = x[rows].double(), xp[rows].double(), xq[rows].double()
            h2.append(torch.log(v.abs().sum(1) ** 2 / (v * v).sum(1)))
            s.append((p * q).sum(1) / ((p * p).sum(1) * (q * q).sum(1)).sqrt())
        h2, s = torch.cat(h2), torch.cat(s)
        k1 = k * LAM[0] // LAM[1]
        k2 = k - k1
        kept = torch.zeros(n, dtype=torch.bool, device=DEV)
        kept[torch.sort(h2, descending=True, stable=True).indices[:k1]] = True
        if k2:
            rem = (~kept).nonzero()[:, 0]
            order = rem[torch.sort(s[rem], stable=True).indices]
            m = order.numel()
            j = torch.arange(k2, device=DEV)
            pos = j * m // k2 if case.get("stride") == "interval" else j * max(1, m // k2)
            kept[order[pos]] = True
        local = kept.nonzero()[:, 0]
        ids.append(local.to(torch.int32))
        ys.append(x[off + local])
        h2s.append(h2)
        ss.append(s)
        off += n
    out = dict(y=torch.cat(ys), idx=torch.cat(ids))
    if case.get("scores"):
        out.update(h2=torch.cat(h2s), s=torch.cat(ss))
    return out


def _act(v, act):
    if act == "gelu":
        return 0.5 * v * (1.0 + torch.erf(v / math.sqrt(2.0)))
    return v * torch.sigmoid(1.702 * v) if act == "quick_gelu" else v


def _exact_mlp(case, seed):
    xp, resid, w1, b1, w2, b2 = _mlp_inputs(case, seed)
    w1, b1, w2, b2 = (v.double() for v in (w1, b1, w2, b2))
    parts = []
    for a in range(0, case["t"], 4096):
        p = xp[a:a + 4096].double()
        h = _act(p @ w1.T + b1, case["act"])
        q = h @ w2.T + b2
        x = q if resid is None else resid[a:a + 4096].double() + q
        l1, s2 = x.abs().sum(1), (x * x).sum(1)
        pp, qq, pq = (p * p).sum(1), (q * q).sum(1), (p * q).sum(1)
        r, s = l1 * l1 / s2, pq / (pp * qq).sqrt()
        parts.append((h.float(), q, x, torch.stack([l1, s2, pp, qq, pq, torch.zeros_like(l1), r, s], 1), r.log(), s))
    h, q, x, stats, h2, s = (torch.cat(v) for v in zip(*parts))
    out = dict(h=h, x_post=q, x=x, stats=stats, error=None)
    if case.get("scores"):
        out.update(h2=h2, s=s)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("reduce", "stream", "call"):
        return _exact_reduce(case, seed)
    if kind == "mlp":
        return _exact_mlp(case, seed)
    if kind == "project":
        y, w, b = _project_inputs(case, seed)
    else:
        x, idx, cu_k, w, b = _kept_inputs(case, seed)
        first = torch.arange(case["images"], device=DEV).repeat_interleave(case["k"]) * case["n"]
        y = x[first + idx]
    w, b = w.double(), b.double()
    return dict(z=torch.cat([_act(y[a:a + 4096].double() @ w.T + b, case["act"]).float()
                             for a in range(0, y.shape[0], 4096)]), error=None)
