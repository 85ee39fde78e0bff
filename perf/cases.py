"""The reduce steps that users of this package run, as measurable cases.

Every case goes through the public Python entry points (``Context`` and
``ficoco_equivalent_token``).  Inputs are made on the GPU from a seed: spatially smooth patch
features on a grid, softmax attention, fp32 or bf16.  A step decides by comparing numbers (which
score wins a penalty window, where the discard boundary falls, which preserved tokens a discarded
one goes to); ``_separate`` moves inputs whose competing numbers are closer than fp32 rounding
noise, so that every correct implementation takes the same decisions and the indices can be
compared exactly.
"""
import math
import random

import torch

from paper_2411_17686_b200 import binding as B

EPS = 0.998                    # the package's default quantile level
WIDTHS = (768, 1024, 1152, 1280, 1408, 1664)    # ViT hidden sizes


def listed():
    return [
        # one image at the end of a schedule: the smallest call, all latency
        dict(name="v_one_small", kind="v", batch=1, gh=24, gw=24, alive=144, keep=64, dim=1024, heads=16,
             cls=True, dtype="bf16"),
        # one ViT-L/14-336 image in fp32, 64 of 576 patches discarded
        dict(name="v_one_fp32", kind="v", batch=1, gh=24, gw=24, alive=576, keep=512, dim=1024, heads=16,
             cls=True, dtype="fp32"),
        # the benchmark's batch: first step of 576 -> 288 -> 144 -> 64
        dict(name="v_batch", kind="v", batch=32, gh=24, gw=24, alive=576, keep=288, dim=1024, heads=16,
             cls=True, dtype="bf16"),
        # the same step on a throughput-serving batch that no cache holds
        dict(name="v_batch_large", kind="v", batch=256, gh=24, gw=24, alive=576, keep=288, dim=1024, heads=16,
             cls=True, dtype="bf16"),
        # multi-crop high resolution: 5 crops of 24 x 24 stacked into one grid
        dict(name="v_multicrop", kind="v", batch=8, gh=120, gw=24, alive=2880, keep=1440, dim=1024, heads=16,
             cls=True, dtype="bf16"),
        # a progressive schedule in one call
        dict(name="v_schedule", kind="schedule", batch=32, gh=24, gw=24, keep=288, keep2=144, keep3=64, dim=1024,
             heads=16, dtype="bf16"),
        # dynamic-resolution batch, no CLS, grids of 16..64 patches a side, 1/9 kept
        dict(name="v_ragged", kind="ragged", batch=16, lo=16, hi=64, grids=4000, divisor=9, dim=1280,
             heads=16, dtype="bf16"),
        # the step on a self-attention map that the encoder hands over
        dict(name="v_relation", kind="relation", batch=32, gh=24, gw=24, keep=288, dim=1024, heads=16,
             by_column=False, dtype="bf16"),
        # decoder layer of a 7B language model, 16 sequences, and a single request
        dict(name="l_batch", kind="l", batch=16, vision=576, text=64, keep=64, dim=4096, heads=32, dtype="bf16"),
        dict(name="l_one", kind="l", batch=1, vision=576, text=64, keep=64, dim=4096, heads=32, dtype="bf16"),
        # stand-in for the CLS attention of an encoder that has none
        dict(name="equivalent", kind="equivalent", batch=32, tokens=577, heads=16, head_dim=64, cls=True,
             dtype="bf16"),
        # the benchmark's batch in pinned host buffers, copies included
        dict(name="v_host", kind="host", batch=32, gh=24, gw=24, alive=576, keep=288, dim=1024, heads=16,
             cls=True, dtype="bf16"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: batch, grid, share kept and width over the ranges of the listed ones."""
    most = max(_cost(c) for c in listed())
    while True:
        case = _draw(rng)
        if _cost(case) <= most:
            return case


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def _draw(rng):
    most = 256 * 577 * 1024                       # token values of the largest listed case
    kind = rng.choice(("v", "v", "v", "v", "schedule", "ragged", "relation", "l", "equivalent", "host"))
    dim, heads = rng.choice(WIDTHS), rng.choice((12, 16))
    dtype = "fp32" if kind == "v" and rng.random() < 0.25 else "bf16"
    room = most // (2 if dtype == "fp32" else 1)

    def batch_of(values, hi):
        return _log_int(rng, 1, max(1, min(hi, room // values)))

    def kept(n):
        return max(1, min(n - 1, int(n * math.exp(rng.uniform(math.log(1 / 9), math.log(8 / 9))))))

    if kind in ("v", "host"):
        gh, gw = _log_int(rng, 8, 64), _log_int(rng, 8, 64)
        alive = gh * gw if rng.random() < 0.6 else max(33, int(gh * gw * rng.uniform(0.25, 1.0)))
        batch = batch_of((alive + 1) * dim, 256 if kind == "v" else 64)
        return dict(kind=kind, batch=batch, gh=gh, gw=gw, alive=alive, keep=kept(alive), dim=dim, heads=heads,
                    cls=rng.random() < 0.7, dtype=dtype)
    if kind == "schedule":
        g = rng.randint(14, 32)
        k1 = int(g * g * rng.uniform(0.4, 0.7))
        k2 = int(k1 * rng.uniform(0.4, 0.7))
        return dict(kind=kind, batch=batch_of(g * g * dim, 64), gh=g, gw=g, keep=k1, keep2=k2,
                    keep3=int(k2 * rng.uniform(0.4, 0.7)), dim=dim, heads=heads, dtype=dtype)
    if kind == "ragged":
        lo = rng.randint(8, 24)
        hi = rng.randint(lo + 4, 64)
        return dict(kind=kind, batch=batch_of(hi * hi * dim, 32), lo=lo, hi=hi, grids=rng.randrange(1 << 20),
                    divisor=rng.randint(2, 9), dim=dim, heads=heads, dtype=dtype)
    if kind == "relation":
        gh, gw = rng.randint(10, 32), rng.randint(10, 32)
        n = gh * gw
        return dict(kind=kind, batch=batch_of(n * max(dim, 2 * n), 64), gh=gh, gw=gw, keep=kept(n), dim=dim,
                    heads=heads, by_column=rng.random() < 0.5, dtype=dtype)
    if kind == "l":
        vision, text = rng.randint(144, 1024), _log_int(rng, 8, 100)
        wide = rng.choice((2048, 3072, 3584, 4096, 5120))
        return dict(kind=kind, batch=batch_of((vision + text) * wide, 32), vision=vision, text=text,
                    keep=kept(vision), dim=wide, heads=rng.choice((16, 28, 32, 40)), dtype=dtype)
    return dict(kind=kind, batch=_log_int(rng, 1, 64), tokens=_log_int(rng, 64, 2048), heads=heads,
                head_dim=rng.choice((64, 80, 88, 128)), cls=rng.random() < 0.5, dtype=dtype)


# ---- inputs -----------------------------------------------------------------------------------

def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _field(gen, batch, gh, gw, dim, corr):
    """[batch, gh * gw, dim] fp32: Gaussian fields, smooth over ``corr[b]`` patches, unit variance per
    channel, plus 0.1 of white noise (neighbouring patches of an image look alike)."""
    def blur(n):
        i = torch.arange(n, device="cuda", dtype=torch.float32)
        m = torch.exp(-0.5 * ((i[:, None] - i[None, :]) / corr[:, None, None]) ** 2)
        return m / m.sum(dim=2, keepdim=True)

    x = torch.randn((batch, gh, gw * dim), generator=gen, device="cuda")
    x = torch.bmm(blur(gh), x).reshape(batch * gh, gw, dim)
    x = torch.bmm(blur(gw).repeat_interleave(gh, dim=0), x).reshape(batch, gh * gw, dim)
    x = (x - x.mean(dim=1, keepdim=True)) / (x.std(dim=1, keepdim=True) + 1e-12)
    return x.add_(torch.randn(x.shape, generator=gen, device="cuda"), alpha=0.1)


def _images(gen, case, gh, gw, batch, alive):
    """tokens [batch, cls + alive, dim], grid positions of the alive patches [batch, alive]."""
    if gh % gw == 0 and gh > gw:                    # stacked crops, each with a correlation length of its own
        corr = torch.rand((batch * (gh // gw),), generator=gen, device="cuda") * 4 + 2
        x = _field(gen, batch * (gh // gw), gw, gw, case["dim"], corr).reshape(batch, gh * gw, case["dim"])
    else:
        x = _field(gen, batch, gh, gw, case["dim"], torch.full((batch,), 3.0, device="cuda"))
    pos = torch.arange(gh * gw, device="cuda").expand(batch, -1)
    if alive < gh * gw:                             # a later step: the other patches are gone already
        pos = torch.rand((batch, gh * gw), generator=gen, device="cuda").argsort(dim=1)[:, :alive].sort(dim=1)[0]
        x = x.gather(1, pos[:, :, None].expand(-1, -1, case["dim"]))
    if case.get("cls"):
        x = torch.cat([torch.randn((batch, 1, case["dim"]), generator=gen, device="cuda"), x], dim=1)
    return x.to(_dtype(case)).contiguous(), pos.contiguous()


def _sides(case):
    """Grid sides of a ragged batch: part of the case, as a program plans for the shapes that it meets."""
    r = random.Random(case["grids"])
    return [(r.randint(case["lo"], case["hi"]), r.randint(case["lo"], case["hi"])) for _ in range(case["batch"])]


def _attention(gen, shape, std=1.0):
    return torch.softmax(std * torch.randn(shape, generator=gen, device="cuda"), dim=-1)


def _raise_columns(gen, attn, which):
    """Attention of the tokens marked in ``which`` [B, N] up by 2 to 5 per cent (attn: [B, ..., N])."""
    f = 1.0 + which * (0.02 + 0.03 * torch.rand(which.shape, generator=gen, device="cuda"))
    attn.mul_(f.reshape([f.shape[0]] + [1] * (attn.dim() - 2) + [f.shape[1]]))


def _separate(gen, tokens, first, n, attns, keeps, *, pos=None, gw=0, relation=None, by_column=False, share=0.35):
    """Moves inputs, in place, until no decision of the step (or of any step of a schedule) hangs on rounding.

    tokens [B, rows, D], of which rows first .. first + n are scored; attns: per step [B, H, Np] (images) or
    [B, H, M, Np] (text to vision); keeps: per step.  Decisions are worked out in float64."""
    text = attns[0].dim() == 4
    for _ in range(12):
        x = tokens[:, first:first + n].double()
        origin = torch.arange(n, device="cuda").expand(x.shape[0], -1)
        p, moved = pos, torch.zeros((x.shape[0], n), dtype=torch.bool, device="cuda")
        raised = torch.zeros((), dtype=torch.bool, device="cuda")
        for step, (attn, keep) in enumerate(zip(attns, keeps)):
            near = 4e-6 if step == 0 else 1.2e-5    # later steps read rows rounded to the storage type
            t = attn.double().mean(dim=1)
            a = t.mean(dim=1) if text else t
            xh = x / x.norm(dim=2, keepdim=True)
            if relation is None:
                v = torch.bmm(xh, xh.mean(dim=1)[:, :, None])[:, :, 0]
            else:
                v = relation.mean(dim=1 if by_column else 2, dtype=torch.float64)
            s = share * v - (1 - share) * a
            close = near * s.abs().amax(dim=1, keepdim=True)
            bad = torch.zeros(s.shape, dtype=torch.bool, device="cuda")
            if p is not None:                       # winner and runner-up of every 2 x 2 window
                win = (p // gw // 2) * ((gw + 1) // 2) + p % gw // 2
                size = (s.shape[0], int(win.max()) + 1)
                low = torch.full(size, -math.inf, dtype=torch.float64, device="cuda")
                best = low.scatter_reduce(1, win, s, "amax").gather(1, win)
                rest = s.masked_fill(s == best, -math.inf)
                second = low.scatter_reduce(1, win, rest, "amax").gather(1, win)
                bad |= (rest == second) & (best - second < close) & (s < best)
                s = torch.where(s == best, 2 * s, s)
            order = s.argsort(dim=1, descending=True)
            n_src = s.shape[1] - keep
            edge = s.gather(1, order[:, n_src - 1:n_src + 1])
            tied = (edge[:, :1] - edge[:, 1:]) < close
            bad.scatter_(1, order[:, n_src:n_src + 1], tied | bad.gather(1, order[:, n_src:n_src + 1]))
            raised |= bad.any()
            _raise_columns(gen, attn, bad.float())
            src, tgt = order[:, :n_src], order[:, n_src:].sort(dim=1)[0]
            if relation is None:
                c = torch.bmm(_rows(xh, src), _rows(xh, tgt).transpose(1, 2))
                if text:
                    bridge = torch.bmm(_rows(t.transpose(1, 2), src), _rows(t.transpose(1, 2), tgt).transpose(1, 2))
                    c = 0.6 * c + 0.4 / t.shape[1] * bridge
                q = EPS * (keep - 1)
                frac = q - math.floor(q)
                taken = keep - math.floor(q) - (1 if frac > 1e-6 else 0)
                top = c.topk(min(taken + 1, keep), dim=2)
                if taken < keep:
                    gap = top[0][:, :, taken - 1] - top[0][:, :, taken]
                    slack = gap * (min(frac, 1 - frac) if frac > 1e-6 else 1.0)
                    doubt = (gap < near) | (slack < 1e-7)
                    moved.scatter_(1, _rows(origin, src), doubt | moved.gather(1, _rows(origin, src)))
            if step + 1 < len(keeps):               # merge, round, go on with the survivors
                w = top[0][:, :, :taken].clamp(min=0)
                w = (w / w.sum(dim=2, keepdim=True))[..., None]
                num, total = _rows(x, tgt), torch.zeros((x.shape[0], keep, 1), dtype=torch.float64, device="cuda")
                for k in range(taken):
                    at = top[1][:, :, k, None]
                    num.scatter_add_(1, at.expand(-1, -1, x.shape[2]), w[:, :, k] * _rows(x, src))
                    total.scatter_add_(1, at, w[:, :, k])
                x = (num / (1 + total)).to(tokens.dtype).double()
                origin, p = origin.gather(1, tgt), None if p is None else p.gather(1, tgt)
        doubtful = bool(moved.any())
        if not doubtful and not bool(raised):
            return
        if doubtful:
            b, i = moved.nonzero(as_tuple=True)
            row = tokens[b, first + i].float()
            row += 0.02 * row.square().mean(dim=1, keepdim=True).sqrt() * torch.randn(row.shape, generator=gen, device="cuda")
            tokens[b, first + i] = row.to(tokens.dtype)


def _rows(x, index):
    """x[b, index[b, i]] for [B, N] or [B, N, D] tensors."""
    return x.gather(1, index) if x.dim() == 2 else x.gather(1, index[:, :, None].expand(-1, -1, x.shape[2]))


# ---- what a program keeps, and one pass -------------------------------------------------------

def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "equivalent":
        shape = (case["batch"], case["tokens"], case["heads"], case["head_dim"])
        keys = torch.randn(shape, generator=gen, device="cuda")
        shared = torch.randn((shape[0], 1, 1, shape[3]), generator=gen, device="cuda")
        keys += shared * torch.rand((shape[0], shape[1], 1, 1), generator=gen, device="cuda")
        return dict(case=case, keys=keys.to(_dtype(case)).reshape(shape[0] * shape[1], -1))
    if kind == "l":
        n, m, batch = case["vision"], case["text"], case["batch"]
        x = (torch.randn((batch, n + m, case["dim"]), generator=gen, device="cuda") / 64).to(_dtype(case))
        logits = torch.randn((batch, case["heads"], m, n + m), generator=gen, device="cuda")
        logits[..., n:].masked_fill_(torch.ones((m, m), dtype=torch.bool, device="cuda").triu(1), -math.inf)
        attn = torch.softmax(logits, dim=-1)[..., :n].contiguous()
        _separate(gen, x, 0, n, [attn], [case["keep"]], share=0.6)
        ctx = B.Context(batch * (n + m), case["dim"], batch, m)
        return dict(case=case, ctx=ctx, params=B.make_params(), tokens=x.reshape(-1, case["dim"]), attn=attn)
    if kind == "ragged":
        sides = _sides(case)
        tokens, attns, keep = [], [], []
        for gh, gw in sides:
            x = _field(gen, 1, gh, gw, case["dim"], torch.full((1,), 3.0, device="cuda")).to(_dtype(case))
            attn = _attention(gen, (1, case["heads"], gh * gw))
            pos = torch.arange(gh * gw, device="cuda")[None]
            keep.append(-(-gh * gw // case["divisor"]))
            _separate(gen, x, 0, gh * gw, [attn], keep[-1:], pos=pos, gw=gw)
            tokens.append(x[0])
            attns.append(attn.reshape(-1))
        state = dict(case=case, tokens=torch.cat(tokens), attn=torch.cat(attns), pos=None, keep=keep,
                     gh=[g[0] for g in sides], gw=[g[1] for g in sides])
        sizes = dict(seqlens=[g[0] * g[1] for g in sides])
    else:
        gh, gw, batch = case["gh"], case["gw"], case["batch"]
        alive, cls = case.get("alive", gh * gw), int(case.get("cls", True))
        keeps = [case["keep"]] + ([case["keep2"], case["keep3"]] if kind == "schedule" else [])
        x, pos = _images(gen, dict(case, cls=cls), gh, gw, batch, alive)
        attns = [_attention(gen, (batch, case["heads"], k), 1.5) for k in [alive] + keeps[:-1]]
        relation = None
        if kind == "relation":                      # similar patches attend to each other
            xh = torch.nn.functional.normalize(x[:, cls:].float(), dim=2)
            logits = 8 * torch.bmm(xh, xh.transpose(1, 2))
            logits += torch.randn(logits.shape, generator=gen, device="cuda")
            relation = torch.softmax(logits, dim=2)
        _separate(gen, x, cls, alive, attns, keeps, pos=pos, gw=gw, relation=relation,
                  by_column=case.get("by_column", False))
        state = dict(case=case, tokens=x.reshape(-1, case["dim"]), attn=attns[0], attns=attns, relation=relation,
                     keep=case["keep"], keeps=keeps, gh=gh, gw=gw,
                     pos=None if alive == gh * gw else pos.to(torch.int32).reshape(-1))
        sizes = dict(n_tokens=cls + alive)
    rows = state["tokens"].shape[0]
    cls = kind != "ragged" and case.get("cls", True)
    state.update(sizes=sizes, params=B.make_params(has_cls=cls),
                 ctx=B.Context(rows, case["dim"], case["batch"]))
    if kind in ("v", "ragged"):                     # such a program plans its shapes at start-up
        state["ctx"].ficoco_v_reduce(state["tokens"], state["attn"], state["keep"], state["gh"], state["gw"],
                                     case["heads"], params=state["params"], plan_only=True, **sizes)
    if kind == "host":
        out = case["batch"] * (int(cls) + case["keep"])
        for key in ("tokens", "attn", "pos"):
            state[key] = None if state[key] is None else state[key].cpu().pin_memory()
        state["out"] = dict(
            out_tokens=torch.empty((out, case["dim"]), dtype=_dtype(case)).pin_memory(),
            kept_idx=torch.empty(out, dtype=torch.int32).pin_memory(),
            pos_out=torch.empty(case["batch"] * case["keep"], dtype=torch.int32).pin_memory())
    return state


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "equivalent":
        return B.ficoco_equivalent_token(state["keys"], case["heads"], case["head_dim"], n_tokens=case["tokens"],
                                         has_cls=case["cls"])
    ctx, p = state["ctx"], state["params"]
    if kind == "l":
        r = ctx.ficoco_l_reduce(state["tokens"], state["attn"], case["keep"], case["vision"], case["text"],
                                case["heads"], params=p)
        return r.out_tokens, r.kept_idx
    if kind == "schedule":
        r = ctx.ficoco_v_reduce_schedule(state["tokens"], state["attns"], state["keeps"], state["gh"], state["gw"],
                                         case["heads"], params=p, **state["sizes"])
    elif kind == "host":
        r = ctx.ficoco_v_reduce_host(state["tokens"], state["attn"], state["keep"], state["gh"], state["gw"],
                                     case["heads"], pos=state["pos"], params=p, **state["sizes"], **state["out"])
    elif kind == "relation":
        r = ctx.ficoco_v_reduce(state["tokens"], state["attn"], state["keep"], state["gh"], state["gw"], case["heads"],
                                params=p, relation=state["relation"], by_column=case["by_column"], **state["sizes"])
    else:
        r = ctx.ficoco_v_reduce(state["tokens"], state["attn"], state["keep"], state["gh"], state["gw"], case["heads"],
                                pos=state["pos"], params=p, **state["sizes"])
    return r.out_tokens, r.kept_idx, r.pos_out


def work(case):
    kind, size = case["kind"], 2 if case["dtype"] == "bf16" else 4
    if kind == "equivalent":
        rows, width = case["batch"] * case["tokens"], case["heads"] * case["head_dim"]
        return dict(bytes=rows * (width * size + 4), flops=rows * (width + 4 * case["head_dim"]))
    dim, batch, heads = case["dim"], case["batch"], case["heads"]
    if kind == "l":
        n, m, k = case["vision"], case["text"], case["keep"]
        token = batch * dim * size * (n + m + k + m)
        return dict(bytes=token + 4 * batch * (heads * m * n + k + m), flops=2 * batch * (n - k) * k * (dim + m))
    if kind == "ragged":
        ns = [gh * gw for gh, gw in _sides(case)]
        ks = [-(-n // case["divisor"]) for n in ns]
        return dict(bytes=dim * size * (sum(ns) + sum(ks)) + 4 * (heads * sum(ns) + 2 * sum(ks)),
                    flops=2 * dim * sum((n - k) * k for n, k in zip(ns, ks)))
    n, k, cls = case.get("alive", case["gh"] * case["gw"]), case["keep"], int(case.get("cls", True))
    n2k, maps = (n - k) * k, n * n if kind == "relation" else 0
    last, more_attn, products = k, 0, n2k
    if kind == "schedule":
        k2, last = case["keep2"], case["keep3"]
        more_attn = heads * (k + k2)
        products += (k - k2) * k2 + (k2 - last) * last
    if kind == "relation":                          # the correlations are read, not formed
        products = 0
    values = batch * (heads * n + more_attn + maps + 2 * last + cls)
    if case.get("alive", 0) and case["alive"] < case["gh"] * case["gw"]:
        values += batch * n
    return dict(bytes=batch * dim * size * (n + cls + last + cls) + 4 * values, flops=2 * batch * dim * products)


def tolerance(case):
    if case["kind"] == "equivalent":                # 32-bit sums of up to a few thousand terms
        return dict(rel=1e-5, max=1e-3)
    if case["dtype"] == "fp32":                     # weighted means with 32-bit weights
        return dict(rel=1e-5, max=1e-3)
    return dict(rel=4e-3, max=4e-2)                 # one rounding to bf16 per element (a schedule: per step)
