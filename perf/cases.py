"""The work that the library is timed on, through its Python entry points (`runner.Fusion`, `runner.Chain`).

A case is one call, or one captured schedule of calls, on a seeded synthetic batch: per image a few
cluster centres ~ N(0, I) with patches around them, a CLS row ~ N(0, I), CLS-attention scores that
are a softmax over the patches, per-image merge counts and keep ratios, random heads whose exit
threshold lies in a gap between two images' confidences.  Token arrays have room for the largest batch
of the case (`batch` x `tokens` rows), as a program that does not know the counts keeps them.  Kinds:

  stage      one fused merge -> exit -> prune -> compact stage (`Fusion.stage`)
  chain      a schedule of stages captured as one CUDA graph and replayed (`Chain.capture`)
  prune      top-k pruning alone on given scores (`fusion_prune` on buffers the program keeps)
  attention  the size-aware attention of the block that reads a compacted batch (`Fusion.attention`)
  scores     the linear pruning router over every token row (`Fusion.token_scores`)
  exit       the exit check alone with a linear or an MLP head (`Fusion.exit_check`, `exit_check_mlp`)
"""
import math

import numpy as np
import torch

from paper_2607_02612_gb300 import (FUSION_STAGE_EXIT, FUSION_STAGE_MERGE, FUSION_STAGE_PRUNE, check, fusion_prune,
                                    runner)

EPS = 1e-6   # LayerNorm epsilon (timm ViT)


def listed():
    return [
        # one image through one stage: an interactive request, all latency
        dict(name="stage_bf16_b1", kind="stage", dtype="bf16", batch=1, tokens=197, fewest=197, dim=384,
             classes=1000, sizes="ones", keys="tokens", r_lo=16, r_hi=16, rho_lo=0.7, rho_hi=0.7, exits=0.0),
        # DeiT-S, float32, a small batch with keys of its own: the reference setting of an accuracy study
        dict(name="stage_f32_b8", kind="stage", dtype="f32", batch=8, tokens=197, fewest=197, dim=384,
             classes=1000, sizes="ones", keys="own", r_lo=16, r_hi=16, rho_lo=0.7, rho_hi=0.7, exits=0.0),
        # DeiT-S, the 12-block schedule on a serving batch: merge at every block, exit and prune at four
        dict(name="chain12_bf16_b256", kind="chain", dtype="bf16", batch=256, tokens=197, fewest=197, dim=384,
             classes=1000, sizes="ones", r_lo=0, r_hi=24, rho_lo=0.5, rho_hi=1.0, exits=0.09, blocks=12,
             exit_blocks="4,6,8,10"),
        # DeiT-B, a full stage on a batch whose tokens were merged before (sizes 1..4), keys of its own
        dict(name="stage_bf16_b512_d768", kind="stage", dtype="bf16", batch=512, tokens=197, fewest=197, dim=768,
             classes=1000, sizes="mixed", keys="own", r_lo=8, r_hi=32, rho_lo=0.4, rho_hi=0.9, exits=0.1),
        # ViT-L/16 at 384 x 384: long samples, a 288 x 288 x 1024 similarity per image
        dict(name="stage_bf16_b128_n577", kind="stage", dtype="bf16", batch=128, tokens=577, fewest=577, dim=1024,
             classes=1000, sizes="ones", keys="tokens", r_lo=16, r_hi=64, rho_lo=0.5, rho_hi=0.9, exits=0.1),
        # many small images (32 x 32 in 4 x 4 patches), high exit rate, four chained full stages, float32
        dict(name="chain4_f32_b8192", kind="chain", dtype="f32", batch=8192, tokens=65, fewest=65, dim=384,
             classes=100, sizes="ones", r_lo=0, r_hi=16, rho_lo=0.3, rho_hi=1.0, exits=0.6, blocks=4,
             exit_blocks="1,2,3,4"),
        # the same in bf16 on ragged images, as after earlier stages
        dict(name="chain4_bf16_b8192", kind="chain", dtype="bf16", batch=8192, tokens=65, fewest=9, dim=384,
             classes=100, sizes="mixed", r_lo=0, r_hi=16, rho_lo=0.3, rho_hi=1.0, exits=0.6, blocks=4,
             exit_blocks="1,2,3,4"),
        # pruning alone (a schedule with P blocks only), float32, ragged, an odd batch
        dict(name="prune_f32_b77_d768", kind="prune", dtype="f32", batch=77, tokens=197, fewest=120, dim=768,
             sizes="mixed", rho_lo=0.5, rho_hi=1.0),
        # the attention of a DeiT-S block on a merged batch
        dict(name="attention_b256_n197", kind="attention", dtype="bf16", batch=256, tokens=197, fewest=100,
             heads=6, sizes="mixed"),
        # the attention of a ViT-L/16 block at 384 x 384
        dict(name="attention_b128_n577", kind="attention", dtype="bf16", batch=128, tokens=577, fewest=577,
             heads=16, sizes="ones"),
        # learned pruning scores of a DeiT-S batch
        dict(name="scores_bf16_b256", kind="scores", dtype="bf16", batch=256, tokens=197, fewest=197, dim=384),
        # the SpatialPool MLP exit head on a DeiT-S batch
        dict(name="exit_mlp_bf16_b256", kind="exit", dtype="bf16", batch=256, tokens=197, fewest=150, dim=384,
             classes=1000, hidden=768, pool="spatial", sizes="mixed", exits=0.2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stage", "stage", "stage", "chain", "prune", "attention", "attention", "scores", "exit"])
    dtype = rng.choice(["bf16", "bf16", "f32"])
    if kind == "attention":
        tokens = _log_int(rng, 16, 600)
        heads = rng.choice([3, 6, 12, 16])
        batch = _log_int(rng, 1, max(1, min(512, 16 * 128 * 577 * 577 // (heads * tokens * tokens))))
        return dict(kind=kind, dtype="bf16", batch=batch, tokens=tokens, fewest=rng.randint(1, tokens), heads=heads,
                    sizes=rng.choice(["ones", "mixed", "none"]))
    dim = rng.choice([192, 384, 384, 768, 1024])
    tokens = _log_int(rng, 10, 600)
    batch = _log_int(rng, 1, max(1, min(8192, 32_000_000 // (dim * tokens))))
    fewest = tokens if rng.random() < 0.4 else rng.randint(2, tokens)
    case = dict(kind=kind, dtype=dtype, batch=batch, tokens=tokens, fewest=fewest, dim=dim)
    if kind == "scores":
        return case
    case["sizes"] = rng.choice(["ones", "mixed"])
    if kind == "exit":
        case.update(classes=rng.choice([10, 100, 1000]), exits=rng.choice([0.0, 0.1, 0.3]),
                    pool=rng.choice(["linear", "spatial", "cls"]))
        case["hidden"] = 0 if case["pool"] == "linear" else rng.choice([dim // 2, dim, min(2 * dim, 1024)])
        return case
    case.update(rho_lo=round(rng.uniform(0.3, 0.7), 2), rho_hi=1.0)
    if kind == "prune":
        return case
    case.update(classes=rng.choice([10, 100, 1000]), r_lo=0, r_hi=max(1, tokens // rng.choice([4, 8, 12])),
                exits=rng.choice([0.0, 0.1, 0.5]))
    if kind == "chain":
        blocks = rng.randint(2, 8)
        case.update(blocks=blocks, exit_blocks=",".join(str(b) for b in range(2, blocks + 1, 2)))
    else:
        case["keys"] = rng.choice(["tokens", "own"])
    return case


# ---- inputs -------------------------------------------------------------------
def _gen(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(seed)


def _dtype(case):
    return runner.TORCH_DTYPE[case["dtype"]]


def _counts(case, seed):
    """Tokens per image (CLS included) and offsets, on the host."""
    rng = np.random.default_rng([seed, 7])
    n = rng.integers(case["fewest"], case["tokens"] + 1, size=case["batch"])
    return n, np.concatenate([[0], np.cumsum(n)]).astype(np.int32)


def _rows(case, seed):
    """The packed token rows in float32, before rounding (zeros beyond the last), and each row's image and
    position."""
    g = _gen(seed)
    n, offsets = _counts(case, seed)
    nt = torch.from_numpy(n).cuda()
    image = torch.repeat_interleave(torch.arange(len(n), device="cuda"), nt)
    pos = torch.arange(int(offsets[-1]), device="cuda") - torch.from_numpy(offsets[:-1].astype(np.int64)).cuda()[image]
    clusters = 32 if case["tokens"] > 256 else 12
    centres = torch.randn((case["batch"] * clusters, case["dim"]), generator=g, device="cuda")
    pick = torch.randint(0, clusters, (len(image),), generator=g, device="cuda")
    x = torch.randn((len(image), case["dim"]), generator=g, device="cuda")
    patch = pos > 0
    x = torch.where(patch[:, None], centres[image * clusters + pick] + 0.3 * x, x)
    return g, _room(case, x), image, pos, offsets


def _room(case, t):
    """The rows t, with zeros up to the largest batch."""
    out = torch.zeros((case["batch"] * case["tokens"],) + t.shape[1:], dtype=t.dtype, device="cuda")
    out[:len(t)] = t
    return out


def _sizes(case, g, pos):
    if case["sizes"] == "ones":
        return torch.ones(len(pos), device="cuda")
    s = torch.randint(1, 5, (len(pos),), generator=g, device="cuda").float()
    return torch.where(pos > 0, s, torch.ones_like(s))


def _scores(case, g, image, pos):
    z = torch.randn(len(pos), generator=g, device="cuda").exp() * (pos > 0)
    total = torch.zeros(case["batch"], device="cuda").index_add_(0, image, z)
    return z / total.clamp_min(1e-30)[image]


def _batch(case, seed, sizes=True, scores=True):
    g, x32, image, pos, offsets = _rows(case, seed)
    x = x32.to(_dtype(case))
    keys = x
    if case.get("keys") == "own":
        keys = (x32 + 0.1 * torch.randn(x32.shape, generator=g, device="cuda")).to(_dtype(case))
    del x32
    return runner.DeviceBatch(
        dtype=case["dtype"], dim=case["dim"], max_batch=case["batch"], max_tokens=case["tokens"],
        max_rows=len(x), x=x, keys=keys,
        sizes=_room(case, _sizes(case, g, pos) if sizes else torch.ones(len(pos), device="cuda")),
        scores=_room(case, _scores(case, g, image, pos)) if scores else None,
        offsets=torch.from_numpy(offsets).cuda())


def _affine(case, g):
    d = case["dim"]
    return ((1 + 0.1 * torch.randn(d, generator=g, device="cuda")).to(_dtype(case)),
            (0.1 * torch.randn(d, generator=g, device="cuda")).to(_dtype(case)))


def _linear_head(case, g):
    d, c = case["dim"], case["classes"]
    gamma, beta = _affine(case, g)
    w = (3.0 / math.sqrt(d) * torch.randn((c, d), generator=g, device="cuda")).to(_dtype(case))
    return runner.HeadTensors(gamma, beta, EPS, w, 0.1 * torch.randn(c, generator=g, device="cuda"), 2.0)


def _mlp_head(case, g):
    d, c, h = case["dim"], case["classes"], case["hidden"]
    gamma, beta = _affine(case, g)
    w1 = (torch.randn((h, d), generator=g, device="cuda") / math.sqrt(d)).to(_dtype(case))
    w2 = (3.0 / math.sqrt(h) * torch.randn((c, h), generator=g, device="cuda")).to(_dtype(case))
    b1, b2 = (0.1 * torch.randn(k, generator=g, device="cuda") for k in (h, c))
    pool = {"cls": 0, "spatial": 1}[case["pool"]]
    return runner.MlpHeadTensors(pool, gamma, beta, EPS, w1, b1, w2, b2, 2.0)


def _threshold(c, share):
    """A threshold in the widest gap near the upper `share` of the confidences c."""
    k = int(round(share * len(c)))
    if k == 0:
        return 2.0
    s = torch.sort(c, descending=True).values.cpu().numpy()
    if k >= len(s):
        return float(np.float32(0.5 * s[-1]))
    at = range(max(1, k - 4), min(len(s), k + 5))
    k = max(at, key=lambda j: s[j - 1] - s[j])
    return float(np.float32(0.5 * (s[k - 1] + s[k])))


def _schedule(case, g, cls):
    """The stages of a stage or chain case: flags, r, rho and head of each; thresholds are set from
    the images that are still there (CLS rows never change, so this needs no merging)."""
    exits = {int(b) for b in case["exit_blocks"].split(",") if b} if case["kind"] == "chain" else {1}
    alive = torch.arange(case["batch"], device="cuda")
    stages = []
    for blk in range(1, case.get("blocks", 1) + 1):
        r = torch.randint(case["r_lo"], case["r_hi"] + 1, (case["batch"],), generator=g, device="cuda",
                          dtype=torch.int32)
        if blk not in exits:
            stages.append(runner.ChainStage(FUSION_STAGE_MERGE, r))
            continue
        rho = case["rho_lo"] + (case["rho_hi"] - case["rho_lo"]) * torch.rand(case["batch"], generator=g, device="cuda")
        head = _linear_head(case, g)
        conf = _linear_exact(head, cls[alive], case)[1]
        head.tau = _threshold(conf, case["exits"])
        alive = alive[conf < head.tau]
        stages.append(runner.ChainStage(FUSION_STAGE_MERGE | FUSION_STAGE_EXIT | FUSION_STAGE_PRUNE, r, rho, head))
    return stages


def _zero(outs):
    for t in outs.values():
        if t is not None:
            t.zero_()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "attention":
        g = _gen(seed)
        _, offsets = _counts(case, seed)
        rows, width = case["batch"] * case["tokens"], case["heads"] * 64
        qkv = torch.randn((rows, 3 * width), generator=g, device="cuda").to(torch.bfloat16)
        sizes = None if case["sizes"] == "none" else _sizes(case, g, torch.arange(rows, device="cuda"))
        b = runner.DeviceBatch(dtype="bf16", dim=width, max_batch=case["batch"], max_tokens=case["tokens"],
                               max_rows=rows, x=qkv, keys=qkv, sizes=sizes, scores=None,
                               offsets=torch.from_numpy(offsets).cuda())
        out = torch.zeros((rows, width), dtype=torch.bfloat16, device="cuda")
        return dict(case=case, f=runner.Fusion(case["batch"]), b=b, qkv=qkv, sizes=sizes, out=out)
    b = _batch(case, seed, sizes="sizes" in case, scores=kind in ("stage", "chain", "prune"))
    g = _gen(seed + 1_000_003)
    f = runner.Fusion(case["batch"], case.get("classes", 1))
    st = dict(case=case, f=f, b=b)
    if kind == "scores":
        st["w"] = (torch.randn(case["dim"], generator=g, device="cuda") / math.sqrt(case["dim"])).to(_dtype(case))
        st["out"] = torch.zeros(b.max_rows, device="cuda")
    elif kind == "exit":
        st["head"] = head = _linear_head(case, g) if case["pool"] == "linear" else _mlp_head(case, g)
        head.tau = _threshold(_exit_exact(st)[1], case["exits"])
    elif kind == "prune":
        st["rho"] = case["rho_lo"] + (case["rho_hi"] - case["rho_lo"]) * torch.rand(
            case["batch"], generator=g, device="cuda")
        st["out"] = {"x": torch.zeros_like(b.x), "sizes": torch.zeros_like(b.sizes),
                     "scores": torch.zeros_like(b.scores), "offsets": torch.zeros_like(b.offsets),
                     "keep_idx": torch.zeros(b.max_rows, dtype=torch.int32, device="cuda")}
    else:
        stages = _schedule(case, g, b.x[b.offsets[:-1].long()])
        if kind == "stage":
            st["stage"], st["out"] = stages[0], f.stage_outputs(b, stages[0].flags, stages[0].head)
            _zero(st["out"])
        else:
            st["chain"] = runner.Chain(f, b, stages)
            for o in st["chain"].outs:
                _zero(o)
            st["chain"].run()
            torch.cuda.synchronize()
            st["graph"] = st["chain"].capture()
    return st


_STAGE_OUT = ("x", "sizes", "scores", "offsets", "keep_idx", "ids", "batch")
_EXIT_OUT = ("exit_mask", "logits", "max_prob")


def run(st):
    kind, f, b = st["case"]["kind"], st["f"], st["b"]
    if kind == "attention":
        return f.attention(b, st["qkv"], st["case"]["heads"], st["sizes"], out=st["out"])
    if kind == "scores":
        return f.token_scores(b, st["w"], 0.125, out=st["out"])
    if kind == "exit":
        return (f.exit_check if st["case"]["pool"] == "linear" else f.exit_check_mlp)(b, st["head"])
    if kind == "prune":
        o = st["out"]
        check(fusion_prune(runner.DTYPE_CODE[b.dtype], b.ragged(), b.x, b.dim, b.sizes, b.scores, st["rho"], o["x"],
                           o["sizes"], o["scores"], o["offsets"], o["keep_idx"], f.workspace, f.ws_bytes, f.status))
        return o
    if kind == "stage":
        s = st["stage"]
        o = f.stage(b, s.flags, s.r, s.rho, s.head, out=st["out"])
        return {k: o[k] for k in _STAGE_OUT + _EXIT_OUT}
    st["graph"].replay()
    outs = st["chain"].outs
    res = {k: outs[-1][k] for k in _STAGE_OUT}
    res["exits"] = [{k: o[k] for k in _EXIT_OUT} for o in outs if o["exit_mask"] is not None]
    return res


# ---- the work of a pass ----------------------------------------------------------
def work(case):
    """Each input read once and each output written once, at the mean counts of the case."""
    kind, B = case["kind"], case["batch"]
    n = 0.5 * (case["fewest"] + case["tokens"])
    n2 = n * n + (case["tokens"] - case["fewest"]) ** 2 / 12   # the mean of the square
    if kind == "attention":
        w = case["heads"] * 64
        return {"bytes": B * n * (8 * w + (4 if case["sizes"] != "none" else 0)) + 4 * B, "flops": 4 * B * n2 * w}
    d, eb = case["dim"], 2 if case["dtype"] == "bf16" else 4
    if kind == "scores":
        return {"bytes": B * n * (d * eb + 4) + d * eb + 4 * B, "flops": 2 * B * n * d}
    if kind == "exit":
        c, h = case["classes"], case["hidden"]
        rows = B * n if case["pool"] == "spatial" else B
        weights = (d * c if not h else d * h + h * c)
        return {"bytes": rows * (d * eb + 4) + weights * eb + B * (5 + 4 * c), "flops": 2 * B * weights + 2 * rows * d}
    rho = 0.5 * (case.get("rho_lo", 1.0) + case.get("rho_hi", 1.0))
    if kind == "prune":
        m = 1 + rho * (n - 1)
        return {"bytes": B * (m * (2 * d * eb + 20) + 4 * n + 12), "flops": 0.0}
    exits = {int(b) for b in case["exit_blocks"].split(",") if b} if kind == "chain" else {1}
    bytes_, flops = 0.0, 0.0
    for blk in range(1, case.get("blocks", 1) + 1):
        full = blk in exits
        half = n / 2
        r = sum(min(v, half) for v in range(case["r_lo"], case["r_hi"] + 1)) / (case["r_hi"] - case["r_lo"] + 1)
        left = B * (1 - case["exits"]) if full else B
        m = max(1.0, n - r)
        m = 1 + rho * (m - 1) if full else m
        if full:
            bytes_ += B * (d * eb + 9) + case["classes"] * (d * eb + 4) + (B - left) * 4 * case["classes"]
            flops += 2 * B * d * case["classes"]
        keys = n * d * eb if case.get("keys") == "own" else 0
        bytes_ += left * (n * (d * eb + 8) + keys + m * (d * eb + 12) + 24)
        flops += left * (2 * half * half * d + 2 * n * d)
        B, n = left, m
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Merged tokens, sizes, scores and indices are exact apart from their own rounding (measured against
    `exact`: 1.6e-3 for rounded bf16 tokens, 3e-8 for float32; logits and confidences 5e-7, with an
    MLP head 4e-6).  A decision may differ only where two candidates tie within the rounding of the
    similarities.  The attention's probabilities and outputs are rounded to bf16 (measured 3e-3)."""
    if case["kind"] == "attention":
        return {"rel": 1e-2, "max": 0.1}
    if case["kind"] == "scores":
        return {"rel": 1e-6, "max": 1e-5}
    if case["kind"] == "exit":
        return {"rel": 2e-5, "max": 2e-4, "differ": 0.002}
    return {"rel": 8e-3 if case["dtype"] == "bf16" else 4e-6, "max": 0.03 if case["dtype"] == "bf16" else 1e-4,
            "differ": 0.002}


# ---- the same in 64 bits ---------------------------------------------------------
def _stored(t, case):
    """A value as it is stored between two steps (one rounding to the token type)."""
    return t.to(_dtype(case)).double()


def _layer_norm(z, head):
    z = z.double()
    mean = z.mean(1, keepdim=True)
    var = ((z - mean) ** 2).mean(1, keepdim=True)
    return (z - mean) / torch.sqrt(var + head.eps) * head.gamma.double() + head.beta.double()


def _linear_exact(head, cls, case):
    u = _layer_norm(cls, head)
    u = _stored(u, case) if case["dtype"] == "bf16" else u
    logits = u @ head.weight.double().T + head.bias.double()
    return logits, torch.softmax(logits, 1).amax(1)


def _exit_exact(st):
    """Logits and confidences of an exit case."""
    case, b, head = st["case"], st["b"], st["head"]
    first = b.offsets[:-1].long()
    z = b.x[first].double()
    if case["pool"] == "linear":
        return _linear_exact(head, z, case)
    if case["pool"] == "spatial":
        n = torch.diff(b.offsets.long())
        image = torch.repeat_interleave(torch.arange(len(n), device="cuda"), n)
        s = b.sizes.double()
        s[first] = 0
        s = s[:len(image)]
        total = torch.zeros(len(n), dtype=torch.float64, device="cuda").index_add_(0, image, s)
        mean = torch.zeros_like(z).index_add_(0, image, b.x[:len(image)].double() * s[:, None])
        mean /= total.clamp_min(1e-300)[:, None]
        z = torch.where((n > 1)[:, None], mean, z)
    u = _layer_norm(z, head)
    u = _stored(u, case) if case["dtype"] == "bf16" else u
    h = torch.nn.functional.gelu(u @ head.w1.double().T + head.b1.double())
    h = _stored(h, case) if case["dtype"] == "bf16" else h
    logits = h @ head.w2.double().T + head.b2.double()
    return logits, torch.softmax(logits, 1).amax(1)


def _padded(t, n, width):
    """Packed rows -> [images, width, ...], zeros beyond each image's rows."""
    valid = torch.arange(width, device="cuda")[None] < n[:, None]
    out = torch.zeros((len(n), width) + t.shape[1:], dtype=t.dtype, device="cuda")
    out[valid] = t[:int(n.sum())]
    return out, valid


def _select(value, valid, k):
    """The k largest values of each row among the valid entries, the lower position first on a tie."""
    order = torch.sort(value.masked_fill(~valid, -math.inf), dim=1, descending=True, stable=True).indices
    rank = torch.empty_like(order).scatter_(1, order, torch.arange(value.shape[1], device="cuda").expand_as(order))
    return valid & (rank < k[:, None])


def _merge_exact(x, keys, sizes, scores, n, r):
    """Merged (x, sizes, scores, kept) on padded arrays [images, width]; x in float64 before rounding."""
    width = x.shape[1]
    valid = torch.arange(width, device="cuda")[None] < n[:, None]
    kept = valid.clone()
    if width < 3:
        return x, sizes, scores, kept
    kn = keys / torch.clamp(keys.norm(dim=2, keepdim=True), min=1e-12)
    sim = kn[:, 2::2] @ kn[:, 1::2].transpose(1, 2)
    sim.masked_fill_(~valid[:, None, 1::2], -math.inf)
    best, to = sim.max(2)
    del kn, sim
    va = valid[:, 2::2]
    gone = _select(best, va, torch.minimum(r.long().clamp_min(0), va.sum(1)))
    kept[:, 2::2] &= ~gone
    num, den, sc = x * sizes[..., None], sizes.clone(), scores.clone()
    at = torch.where(gone, 1 + 2 * to, 0)   # a token that stays adds nothing to position 0
    num.scatter_add_(1, at[..., None].expand(-1, -1, x.shape[2]), num[:, 2::2] * gone[..., None])
    den.scatter_add_(1, at, den[:, 2::2] * gone)
    sc.scatter_add_(1, at, sc[:, 2::2] * gone)
    merged = den != sizes
    x = torch.where(merged[..., None], num / den.clamp_min(1e-300)[..., None], x)
    return x, den, sc, kept


def _prune_exact(scores, kept, rho):
    patch = kept.clone()
    patch[:, 0] = False
    count = patch.sum(1)
    k = torch.minimum(torch.ceil(rho.double() * count).long().clamp_min(0), count)
    keep = _select(scores, patch, k)
    keep[:, 0] = kept[:, 0]
    return keep


def _into(t, like):
    out = torch.zeros(like.shape, dtype=torch.float64 if like.is_floating_point() else like.dtype, device="cuda")
    out[:len(t)] = t
    return out


def _stages_exact(st, stages, outs):
    case, b = st["case"], st["b"]
    offsets, ids = b.offsets.long(), torch.arange(case["batch"], device="cuda")
    x, keys, sizes, scores = b.x.double(), b.keys.double(), b.sizes.double(), b.scores.double()
    exits = []
    for s, o in zip(stages, outs):
        n = torch.diff(offsets)
        width = int(n.max()) if len(n) else 1
        xp, valid = _padded(x, n, width)
        kp = xp if keys is x else _padded(keys, n, width)[0]
        zp, cp = _padded(sizes, n, width)[0], _padded(scores, n, width)[0]
        rp = _padded(torch.arange(len(x), device="cuda"), n, width)[0]
        cls = x[offsets[:-1]]
        xp, zp, cp, kept = _merge_exact(xp, kp, zp, cp, n, s.r[ids])
        cp = cp.float().double()   # scores are stored in float32
        alive = torch.ones(len(n), dtype=torch.bool, device="cuda")
        if s.flags & FUSION_STAGE_EXIT:
            logits, conf = _linear_exact(s.head, cls, case)
            alive = conf < s.head.tau
            exits.append({"exit_mask": _into((~alive).to(torch.uint8), o["exit_mask"]),
                          "logits": _into(torch.where(alive[:, None], 0.0, logits), o["logits"]),
                          "max_prob": _into(conf, o["max_prob"])})
            kept = _prune_exact(cp, kept, s.rho[ids])
        kept &= alive[:, None]
        exact_x = xp[kept]
        x, sizes, scores, rows = _stored(exact_x, case), zp[kept], cp[kept], rp[kept]
        keys, ids = x, ids[alive]
        offsets = torch.cat([offsets.new_zeros(1), torch.cumsum(kept.sum(1)[alive], 0)])
        del xp, kp, zp, cp, rp
    o = outs[-1]
    res = {"x": _into(exact_x, o["x"]), "sizes": _into(sizes, o["sizes"]), "scores": _into(scores, o["scores"]),
           "offsets": _into(offsets.int(), o["offsets"]), "keep_idx": _into(rows.int(), o["keep_idx"]), "ids": _into(ids.int(), o["ids"]),
           "batch": torch.tensor([len(ids)], dtype=torch.int32, device="cuda")}
    return res, exits


def exact(case, seed):
    st, kind = prepare(case, seed), case["kind"]
    b = st["b"]
    if kind == "scores":
        rows = int(b.offsets[-1])
        return _into(b.x[:rows].double() @ st["w"].double() + 0.125, st["out"])
    if kind == "exit":
        logits, conf = _exit_exact(st)
        out = conf >= st["head"].tau
        return {"exit_mask": out.to(torch.uint8), "logits": torch.where(out[:, None], logits, 0.0), "max_prob": conf}
    if kind == "prune":
        n = torch.diff(b.offsets.long())
        cp, valid = _padded(b.scores.double(), n, int(n.max()))
        keep = _prune_exact(cp, valid, st["rho"])
        rows = keep[valid].nonzero()[:, 0]
        out = {"x": b.x.double()[rows], "sizes": b.sizes.double()[rows], "scores": b.scores.double()[rows],
               "offsets": torch.cat([n.new_zeros(1), torch.cumsum(keep.sum(1), 0)]).int(), "keep_idx": rows.int()}
        return {k: _into(t, st["out"][k]) for k, t in out.items()}
    if kind == "attention":
        h, off = case["heads"], b.offsets.tolist()
        out = torch.zeros(st["out"].shape, dtype=torch.float64, device="cuda")
        for lo, hi in zip(off[:-1], off[1:]):
            q, k, v = st["qkv"][lo:hi].double().view(hi - lo, 3, h, 64).permute(1, 2, 0, 3)
            z = q @ k.transpose(1, 2) / 8.0
            if st["sizes"] is not None:
                z += st["sizes"][lo:hi].double().log()
            out[lo:hi] = (torch.softmax(z, 2) @ v).permute(1, 0, 2).reshape(hi - lo, h * 64)
        return out
    if kind == "stage":
        res, exits = _stages_exact(st, [st["stage"]], [st["out"]])
        return {**res, **exits[0]}
    res, exits = _stages_exact(st, st["chain"].stages, st["chain"].outs)
    if case["batch"] < 1000:
        # every stage decides on the tokens that the one before it rounded, so near ties add up over a chain:
        # one of them, decided as float32 sums have it, moves a visible share of a small batch's rows
        res = {k: None for k in res}
    res["exits"] = exits
    return res
