"""The work a user of this library has it do, as measurable cases.

A video diffusion transformer calls the library once per attention layer and denoising step.  What it
holds by then are Q, K, V and a block mask; what it calls depends on the program around it:

  step    the mask is new (dynamic sparse attention): bitmap -> index lists, plan, attention.
  attend  the mask, its index lists and its row order are kept over several denoising steps:
          attention alone.
  plan    a program that drives its own attention backend asks for the row order only, from a
          bitmap or from index lists.
  deploy  such a program also has Q gathered into the order and O scattered back (the paper's two
          reorder operators).

Shapes and mask statistics are those of `paper_2609_34814_b200.inputs.CONFIGS`; the masks are drawn
here with the same recipe as `inputs.make_mask`, on the GPU (the sort of every row by priority takes
seconds per head in NumPy on the long sequences).
"""
import dataclasses
import math

import torch

from paper_2609_34814_b200 import binding as wb
from paper_2609_34814_b200 import inputs

DEFAULTS = dict(op="step", recipe="wan720p", heads=40, frames=21, cut=0, block=128, head_dim=128, density=0.0,
                mask="video", mode="auto", layout="hnd", lse=False, lists=False)


def _case(name=None, **kw):
    c = dict(DEFAULTS, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: two heads of 4096 tokens, 64x64 blocks; launches and host work count
        _case("tiny_step", recipe="tiny", heads=2, frames=4, block=64, head_dim=64),
        # one GPU's share of a 480p clip when its 40 heads are split over eight GPUs
        _case("480p_rank_step", recipe="wan480p", heads=5),
        # a whole 480p clip, 81 frames (21 latent ones)
        _case("480p_step", recipe="wan480p"),
        # a whole 720p clip, 81 frames: the workload of bench.py
        _case("720p_step"),
        # 64x64 blocks, densities of 5 to 30 % by head and rows that select everything
        _case("ltx_step", recipe="ltxmixed", heads=32, frames=64, block=64),
        # a 401-frame 720p clip, where the guard lets the plan run on every head: the largest call
        _case("long720p_step", recipe="long720p", frames=101),
        # a short clip of odd length straight out of a fused QKV projection ([tokens, 3, heads, D]),
        # kept mask, with the log-sum-exp for a later merge
        _case("clip_attend_qkv", recipe="wan480p", heads=12, frames=9, cut=83, op="attend", layout="qkv", lse=True),
        # head_dim 64 with 128x128 blocks, kept mask, ragged
        _case("d64_attend", recipe="wan480p", heads=24, frames=13, cut=41, head_dim=64, op="attend", lse=True),
        # the layers and first steps that a sparse method leaves dense go through the same call
        _case("dense_attend", recipe="wan480p", heads=8, op="attend", mask="dense"),
        # an engine that keeps index lists asks for the order of 64x64-block rows
        _case("ltx_plan_lists", recipe="ltxmixed", heads=32, frames=64, block=64, op="plan", mode="reorder", lists=True),
        # the order of a 401-frame clip on one of eight GPUs
        _case("long720p_rank_plan", recipe="long720p", heads=5, frames=101, op="plan", mode="reorder"),
        # another backend behind the plan: order, Q gathered, O scattered back
        _case("720p_deploy", op="deploy", mode="reorder"),
    ]


# head counts of whole models and of their shares on 2, 4 and 8 GPUs
_HEADS = [2, 3, 4, 5, 6, 8, 10, 12, 16, 20, 24, 32, 40]


def draw(rng):
    """One more case: any call, shape family, length, density, layout and option of the ranges above."""
    recipe = rng.choice(["tiny", "wan480p", "wan720p", "wan720p", "ltxmixed", "long720p"])
    base = inputs.CONFIGS[recipe]
    op = rng.choice(["step", "step", "step", "attend", "attend", "plan", "deploy"])
    frames = int(round(math.exp(rng.uniform(math.log(2 if recipe != "tiny" else 1), math.log(base.frames)))))
    cut = rng.choice([0, rng.randrange(1, base.frame_tokens // 2)])
    block = base.block if rng.random() < 0.8 else 192 - base.block
    head_dim = base.head_dim if rng.random() < 0.8 else 192 - base.head_dim
    mask = rng.choice(["video", "video", "video", "video", "random"])
    density = 0.0 if rng.random() < 0.5 else math.exp(rng.uniform(math.log(0.04), math.log(0.30)))
    if op == "deploy":
        cut = 0
    c = _case(op=op, recipe=recipe, frames=frames, cut=cut, block=block, head_dim=head_dim, mask=mask,
              density=round(density, 4), mode=rng.choice(["auto", "auto", "reorder"]), heads=rng.choice(_HEADS),
              layout=rng.choice(["hnd", "hnd", "qkv"]) if op in ("step", "attend") else "hnd",
              lse=op in ("step", "attend") and rng.random() < 0.3, lists=op == "plan" and rng.random() < 0.5)
    # no more work than half of the largest listed call (its matrix products, its rows of Q, its mask words)
    while c["heads"] > 2 and (_flops(dict(c, op="attend")) > 5e13 or _config(c).n_blocks ** 2 * c["heads"] > 1.7e8):
        c["heads"] = max(2, c["heads"] // 2)
    return c


# ------------------------------------------------------------------------------ masks

def _config(case):
    base = inputs.CONFIGS[case["recipe"]]
    rho = (case["density"], case["density"]) if case["density"] > 0 else base.rho
    return dataclasses.replace(base, heads=case["heads"], frames=case["frames"], rho=rho, block=case["block"],
                               head_dim=case["head_dim"], seq=case["frames"] * base.frame_tokens - case["cut"])


def _structured(cfg, parity):
    """Priority of the diagonal, the neighbours in the frame and the same place in nearby frames
    (more negative = taken earlier), inf elsewhere."""
    nb, lf = cfg.n_blocks, cfg.frame_tokens
    dev = "cuda"
    i = torch.arange(nb, device=dev)
    centre = torch.clamp(i * cfg.block + cfg.block // 2, max=cfg.seq - 1)
    frame, off = centre // lf, centre % lf
    pri = torch.full((nb, nb), float("inf"), device=dev)
    window, band = (2, cfg.frames - 1) if cfg.kind == "tiny" else (cfg.w_s[parity], cfg.f_band[parity])

    def put(j, ok, value):      # one entry per row; rows without such a neighbour keep what they have
        j = j.clamp(0, nb - 1)
        pri[i, j] = torch.where(ok, torch.full_like(pri[i, j], value), pri[i, j])

    for d in range(band, 0, -1):
        for s in (1, -1):
            f = frame + s * d
            put((f * lf + off) // cfg.block, (f >= 0) & (f < cfg.frames), -1.0 + 0.5 * d / (band + 1) + (0.01 if s < 0 else 0.0))
    for d in range(window, 0, -1):
        for s in (1, -1):
            j = i + s * d
            ok = (j >= 0) & (j < nb)
            put(j, ok & (frame[j.clamp(0, nb - 1)] == frame), -2.0 + 0.5 * d / (window + 1) + (0.01 if s < 0 else 0.0))
    pri[i, i] = -3.0
    return pri


def _head_density(cfg, head):
    lo, hi = cfg.rho
    return lo + (hi - lo) * (0.5 if cfg.heads == 1 else head / (cfg.heads - 1))     # spread evenly over the heads


def _draw_mask(cfg, kind, head, pri, gen):
    """Boolean block mask of one head on the GPU: the recipe of inputs.make_mask, or uniform columns."""
    nb, dev = cfg.n_blocks, "cuda"
    rho = _head_density(cfg, head)
    noise = torch.empty((nb, nb), device=dev).exponential_(generator=gen)
    if kind == "random":
        score, n_row = noise, torch.full((nb,), max(1, round(rho * nb)), device=dev)
    elif cfg.kind == "tiny":
        n_row = torch.isfinite(pri).sum(1) + 3 + torch.randint(0, 14, (nb,), generator=gen, device=dev)
        score = torch.where(torch.isfinite(pri), pri, noise)
    else:
        z = torch.randn((nb,), generator=gen, device=dev)
        n_row = torch.round(rho * nb * torch.exp(cfg.sigma * z - 0.5 * cfg.sigma ** 2)).clamp(min(cfg.n_min, nb), nb)
        pool = min(nb, max(1, math.ceil(cfg.kappa * rho * nb)))
        cols = torch.rand((cfg.pools, nb), generator=gen, device=dev).argsort(1)[:, :pool]
        weight = torch.full((cfg.pools, nb), (1.0 - cfg.pool_q) / nb, device=dev)
        weight.scatter_add_(1, cols, torch.full(cols.shape, cfg.pool_q / pool, device=dev))
        i = torch.arange(nb, device=dev)
        centre = torch.clamp(i * cfg.block + cfg.block // 2, max=cfg.seq - 1)
        score = noise / weight[cfg.pools * (centre % cfg.frame_tokens) // cfg.frame_tokens]
        score = torch.where(torch.isfinite(pri), pri, score)
        if cfg.sink_frac > 0:
            sink = torch.rand((nb,), generator=gen, device=dev) < cfg.sink_frac
            n_row = torch.where(sink, torch.full_like(n_row, nb), n_row)
    rank = score.argsort(1)
    take = torch.arange(nb, device=dev)[None, :] < n_row[:, None]
    return torch.zeros((nb, nb), dtype=torch.bool, device=dev).scatter_(1, rank, take)


def _pack(mask):
    """Mask rows as little-endian 64-bit words."""
    nb, n = mask.shape
    words = (n + 63) // 64
    bits = torch.zeros((nb, words * 64), dtype=torch.int64, device=mask.device)
    bits[:, :n] = mask
    return (bits.view(nb, words, 64) << torch.arange(64, device=mask.device)).sum(2)


def _bitmap(cfg, kind, seed):
    nb = cfg.n_blocks
    if kind == "dense":
        one = _pack(torch.ones((nb, nb), dtype=torch.bool, device="cuda"))
        return one.expand(cfg.heads, *one.shape).contiguous(), cfg.heads * nb * nb
    gen = torch.Generator("cuda")
    pri = [_structured(cfg, p) for p in (0, 1)]
    out, count = [], 0
    for h in range(cfg.heads):
        gen.manual_seed(seed * 1009 + 31 * h + 7)
        m = _draw_mask(cfg, kind, h, pri[h % 2], gen)
        out.append(_pack(m))
        count += int(m.sum())
    return torch.stack(out), count


# ------------------------------------------------------------------------------ state and pass

class _State:
    pass


def prepare(case, seed):
    """Q, K, V (independent N(0,1) in bf16, as everywhere in this repository), the block mask, and what a
    program keeps between calls: descriptors, workspaces, the output buffer; for a kept mask its
    index lists and row order too."""
    cfg, dev = _config(case), "cuda"
    s = _State()
    s.case, s.nb, s.block = case, cfg.n_blocks, cfg.block
    H, T, D = cfg.heads, cfg.seq_pad, cfg.head_dim
    s.bitmap, s.pairs = _bitmap(cfg, case["mask"], seed)
    s.pdesc = wb.plan_desc_default(heads=H, n_q_blocks=s.nb, n_kv_blocks=s.nb, wave_size=wb.default_wave_size(),
                                   mode=wb.AUTO if case["mode"] == "auto" else wb.FORCE_REORDER, seed=seed & 0xFFFF,
                                   kv_bytes_per_head=2 * T * D * 2)
    s.pws = torch.empty((wb.plan_workspace_bytes(s.pdesc) + 256,), dtype=torch.uint8, device=dev)
    gen = torch.Generator(dev)
    gen.manual_seed(seed + 77)

    def normal(*shape):
        x = torch.empty(shape, dtype=torch.bfloat16, device=dev)
        for part in x:                                   # head by head: no fp32 copy of the whole tensor
            part.copy_(torch.randn(part.shape, generator=gen, device=dev))
        return x

    s.lse = None
    if case["op"] in ("step", "attend"):
        if case["layout"] == "qkv":
            qkv = normal(3, H, T, D).permute(2, 0, 1, 3).contiguous()            # [tokens, 3, heads, D]
            s.q, s.k, s.v = (qkv[:, i].permute(1, 0, 2) for i in range(3))
            s.o = torch.zeros((T, H, D), dtype=torch.bfloat16, device=dev).permute(1, 0, 2)
        else:
            s.q, s.k, s.v = normal(H, T, D), normal(H, T, D), normal(H, T, D)
            s.o = torch.zeros((H, T, D), dtype=torch.bfloat16, device=dev)
        if case["lse"]:
            s.lse = torch.zeros((H, cfg.seq), dtype=torch.float32, device=dev)
        s.adesc = wb.attn_desc(s.q, s.k, s.v, s.o, cfg.seq, cfg.seq, cfg.block)
        s.aws = torch.empty((wb.bsattn_workspace_bytes(s.adesc),), dtype=torch.uint8, device=dev)
        s.status = torch.zeros((4,), dtype=torch.int32, device=dev)
    elif case["op"] == "deploy":
        s.q, s.gathered = normal(H, T, D), torch.zeros((H, T, D), dtype=torch.bfloat16, device=dev)
        s.o, s.back = normal(H, T, D), torch.zeros((H, T, D), dtype=torch.bfloat16, device=dev)
    if case["op"] == "attend" or case["lists"]:
        s.ptr, s.idx = wb.bitmap_to_csr(s.bitmap, s.nb, capacity=s.pairs)
    if case["op"] == "attend":
        s.order = wb.plan_bitmap(s.pdesc, s.bitmap, workspace=s.pws).row_order
    return s


def run(s):
    op = s.case["op"]
    if op == "step":
        # the mask builder knows how many blocks it selected, so the lists are sized without a read-back
        ptr, idx = wb.bitmap_to_csr(s.bitmap, s.nb, capacity=s.pairs)
        plan = wb.plan_bitmap(s.pdesc, s.bitmap, workspace=s.pws)
        wb.bsattn_fwd(s.adesc, s.q, s.k, s.v, s.o, ptr, idx, row_order=plan.row_order, lse=s.lse, workspace=s.aws,
                      dev_status=s.status)
        # (the index list's length differs from mask to mask; what it holds shows in o)
        return {"o": s.o, "lse": s.lse, "ptr": ptr, "order": plan.row_order, "nnz": plan.row_nnz,
                "flags": plan.skip_flags, "status": s.status}
    if op == "attend":
        wb.bsattn_fwd(s.adesc, s.q, s.k, s.v, s.o, s.ptr, s.idx, row_order=s.order, lse=s.lse, workspace=s.aws,
                      dev_status=s.status)
        return {"o": s.o, "lse": s.lse, "status": s.status}
    if s.case["lists"]:
        plan = wb.plan_csr(s.pdesc, s.ptr, s.idx, workspace=s.pws)
    else:
        plan = wb.plan_bitmap(s.pdesc, s.bitmap, workspace=s.pws)
    out = {"order": plan.row_order, "nnz": plan.row_nnz, "flags": plan.skip_flags, "status": plan.dev_status}
    if op == "deploy":
        wb.gather_rows(s.q, s.gathered, plan.row_order, s.block)
        wb.scatter_rows(s.o, s.back, plan.row_order, s.block)
        out.update(q=s.gathered, o=s.back)
    return out


# ------------------------------------------------------------------------------ what a pass cannot do without

def _pairs(case):
    """Block pairs the mask is expected to select."""
    cfg = _config(case)
    nb = cfg.n_blocks
    if case["mask"] == "dense":
        return cfg.heads * nb * nb
    if cfg.kind == "tiny" and case["mask"] == "video":
        per_row = 4 + 2 * (cfg.frames - 1) * 0.5 + 1 + 9.5          # window, band inside the clip, diagonal, extras
        return cfg.heads * nb * min(nb, per_row)
    rho = sum(_head_density(cfg, h) for h in range(cfg.heads)) / cfg.heads
    sink = cfg.sink_frac if case["mask"] == "video" else 0.0
    return cfg.heads * nb * min(nb, (rho * (1 - sink) + sink) * nb)


def _flops(case):
    return 4.0 * case["block"] ** 2 * case["head_dim"] * _pairs(case) if case["op"] in ("step", "attend") else 0.0


def work(case):
    """The two matrix products over the selected block pairs; each tensor, mask and list once.  The plan's
    own arithmetic (two sparse products of width two per iteration) is counted where it is the call."""
    cfg = _config(case)
    rows = cfg.heads * cfg.n_blocks
    tensor = 2.0 * cfg.heads * cfg.seq * cfg.head_dim
    bitmap, lists, order = rows * ((cfg.n_blocks + 63) // 64) * 8.0, 4.0 * (_pairs(case) + rows + 1), 4.0 * rows
    if case["op"] == "step":
        nbytes = 4 * tensor + bitmap + lists + 2 * order
    elif case["op"] == "attend":
        nbytes = 4 * tensor + lists + order
    else:
        nbytes = (lists if case["lists"] else bitmap) + 2 * order + (4 * tensor if case["op"] == "deploy" else 0)
    if case["lse"]:
        nbytes += 4.0 * cfg.heads * cfg.seq
    flops = _flops(case)
    if case["op"] in ("plan", "deploy"):
        flops = 2 * 2 * 6 * _pairs(case)          # 2 columns, 2 products, T + 1 = 6 sweeps, one addition each
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # whole numbers (orders, lists, counts, flags) and copies have one right answer; the orders come from
    # fp64 and are the same with the sums of a sweep taken in another order (24,644 rows compared).
    # O against fp64 with another rounding of the probabilities and of O: rel 3.3e-3, max 2.6e-2
    if case["op"] in ("plan", "deploy"):
        return "exact"
    return {"rel": 1.2e-2, "max": 0.1}
