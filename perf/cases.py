"""Workloads of the compression path, as a program that uses the package runs it.

A pass is what a prefill does with the package: at every compression layer of the schedule the layer's hidden states,
queries and keys go through compress_layer, and the K/V caches that hold the same tokens go through compact_kv; the
positions and counts that a stage leaves on the device are the next stage's inputs.  The plan, the output and scratch
buffers and the streams are made once and kept, as a serving program keeps them.

A case is a dict of
  batch, grid ("5*24x24": tiles per sample), text (rows before the vision block), after (rows behind it), hidden,
  heads, kv_heads, head_dim, windows / keep (one value per stage), dtype ("bf16", "fp32"),
  xi: "full" (from Q and K), "lse" (from Q, the prompt's K and the row log-sum-exp of the caller's attention),
      "given" (the caller's own token scores), "uniform" (plain group means)
  kv: "head_major" or "token_major" (contiguous caches into second buffers), "paged" (pages of 16 tokens into other
      pages), "in_place" / "paged_in_place" (the cache shrinks inside its own rows / pages)
  kv_mode ("merge", "gather"), caches (how many layers' caches a stage compacts),
  packed: samples of unequal length, each with its own subset of the grid, stored back to back without padding
  streams: the second stream inside compress_layer and the compaction behind its map event on a third one
"""
from __future__ import annotations

import math

import torch

import paper_2605_00789_b200 as L

PAGE = 16


def _case(name, batch, grid, text, hidden, heads, kv_heads, head_dim, windows, keep, xi="full", dtype="bf16",
          kv="head_major", kv_mode="merge", caches=1, after=0, packed=False, streams=False):
    case = dict(batch=batch, grid=grid, text=text, after=after, hidden=hidden, heads=heads, kv_heads=kv_heads,
                head_dim=head_dim, windows=windows, keep=keep, xi=xi, dtype=dtype, kv=kv, kv_mode=kv_mode,
                caches=caches, packed=packed, streams=streams)
    return case if name is None else dict(name=name, **case)


def listed():
    return [
        # two small crops per sample with ragged windows and odd sizes: every launch is short, latency and host count
        _case("small_crops", 3, "12x10,9x11", 19, 264, 6, 2, 128, "3,2,1", "0.55,0.6,0.5"),
        # one image in a 7B model, one compression layer: what an interactive request pays at that layer
        _case("one_image_step", 1, "24x24", 32, 4096, 32, 32, 128, "4", "0.55"),
        # the same model over its whole schedule (three halvings)
        _case("one_image_schedule", 1, "24x24", 64, 4096, 32, 32, 128, "4,2,1", "0.5,0.5,0.5"),
        # a serving engine: fused attention hands over its row log-sum-exp, the paged caches of several layers shrink
        # inside their own pages, the question stands behind the image
        _case("serving_paged_lse", 4, "24x24", 35, 4096, 32, 8, 128, "4,2", "0.5,0.6", xi="lse", kv="paged_in_place",
              caches=3, after=41),
        # samples of unequal length without padding, heads of 64
        _case("packed_batch", 16, "24x24", 48, 2048, 32, 8, 64, "4,2", "0.5,0.5", kv="in_place", packed=True),
        # any-resolution input (five tiles), batch of 8, whole schedule: the throughput workload
        _case("anyres_batch", 8, "5*24x24", 128, 4096, 32, 32, 128, "6,4,2", "0.5,0.5,0.5", streams=True),
        # the same batch where the caller's attention supplies the row log-sum-exp
        _case("anyres_batch_lse", 8, "5*24x24", 128, 4096, 32, 32, 128, "6,4,2", "0.5,0.5,0.5", xi="lse"),
        # many single images through a 13B model
        _case("wide_batch", 32, "24x24", 64, 5120, 40, 40, 128, "4,2,1", "0.5,0.5,0.5"),
        # eight video frames, grouped-query attention, paged caches
        _case("video_gqa", 2, "8*32x32", 256, 3584, 28, 4, 128, "4,2,1", "0.5,0.5,0.5", kv="paged"),
        # one tall stack of patches with windows of 512 to 2048 tokens: the pair scores are a real contraction
        _case("large_windows", 2, "256x32", 256, 3584, 28, 4, 128, "4,2,1", "0.5,0.5,0.5", xi="uniform"),
        # token scores from the caller, survivors' rows gathered, token-major caches of several layers
        _case("given_scores_gather", 4, "3*27x27", 77, 3072, 24, 8, 128, "5,3", "0.7,0.55", xi="given",
              kv="token_major", kv_mode="gather", caches=4),
        # single precision storage and arithmetic
        _case("single_precision", 2, "24x24", 33, 1024, 8, 8, 128, "4,2", "0.55,0.5", dtype="fp32"),
    ]


def _tiles(case):
    out = []
    for part in case["grid"].split(","):
        count, _, size = part.rpartition("*")
        rows, cols = size.split("x")
        out += [(int(rows), int(cols))] * int(count or 1)
    return out


def _schedule(case):
    return [int(w) for w in case["windows"].split(",")], [float(k) for k in case["keep"].split(",")]


def _stage_sizes(case):
    """(vision tokens in, out) per sample and stage, to within the rounding of single windows."""
    n = sum(r * c for r, c in _tiles(case))
    if case["packed"]:
        n = 3 * n // 4                                   # samples keep between half and all of the grid
    sizes = []
    for keep in _schedule(case)[1]:
        m = math.ceil(keep * n)
        sizes.append((n, m))
        n = m
    return sizes


def work(case):
    """Per stage: hidden states read once and written once; Q of the vision rows and K read once where xi comes from
    them (K of the prompt only with a given log-sum-exp; the K that is compacted is not counted twice); every cache
    read once and written once; two flops per (pair, channel) of the score and of the attention logits."""
    el = 2 if case["dtype"] == "bf16" else 4
    b, h, hk, dh, d = (case[k] for k in ("batch", "heads", "kv_heads", "head_dim", "hidden"))
    nt, na = case["text"], case["after"]
    tiles, windows = _tiles(case), _schedule(case)[0]
    n_bytes = flops = 0.0
    for (n, m), w in zip(_stage_sizes(case), windows):
        n_bytes += b * (2 * (nt + na) + n + m) * d * el
        n_bytes += case["caches"] * b * 2 * hk * dh * el * (2 * (nt + na) + n + m)
        if case["xi"] == "full":
            n_bytes += b * h * n * dh * el
            flops += 2.0 * b * h * dh * (n * (nt + 1) + n * (n - 1) / 2)
        elif case["xi"] == "lse":
            n_bytes += b * h * n * (dh * el + 4)
            flops += 2.0 * b * h * dh * n * nt
        flops += 2.0 * b * d * (n / 2) * (n / 2) / (len(tiles) * w * w)
        n_bytes += b * (n + m) * 4 * 6                                    # positions, map, weights, scores
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    """Rows are rounded to the storage type.  A pair of scores closer than single precision resolves may be ordered
    either way: then one token joins another group, which changes a few entries of the map and two merged rows."""
    if case["dtype"] == "fp32":
        return {"rel": 1e-4, "max": 1e-2, "differ": 1e-3}
    return {"rel": 1e-2, "max": 0.4, "differ": 5e-3}


# ------------------------------------------------------------------------------------------------------ drawn cases

def _cost(case):
    """Rough microseconds of a pass: memory traffic, one exponential per logit, and the plain-FMA kernels for what the
    tensor cores do not take.  Only for keeping drawn cases within the largest listed one."""
    w = work(case)
    logit_flops = 0.0
    for n, _ in _stage_sizes(case):
        if case["xi"] == "full":
            logit_flops += 2.0 * case["batch"] * case["heads"] * case["head_dim"] * n * (case["text"] + n / 2)
    simt = case["dtype"] == "fp32" or case["head_dim"] not in (64, 128)
    return w["bytes"] / 3e6 + logit_flops / (128 if simt else 2 * case["head_dim"]) / (1e5 if simt else 2.6e6) + \
        ((w["flops"] - logit_flops) / 1e6 if case["dtype"] == "fp32" else (w["flops"] - logit_flops) / 2e8)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the ranges above: 1 to 40 samples of 1 to 8 tiles with 8 to 36 patches a side (or one tall stack),
    prompts of 8 to 300 rows, hidden sizes 256 to 5120, one to three stages."""
    limit = _cost(next(c for c in listed() if c["name"] == "anyres_batch"))
    while True:
        head_dim = rng.choice([64, 128, 128, 128, 128, 96])
        kv_heads = rng.choice([1, 2, 4, 8, 8, 16, 32, 40])
        heads = kv_heads * rng.choice([1, 1, 2, 4, 7])
        if heads > 40:
            continue
        hidden = rng.choice([heads * head_dim, heads * head_dim, 8 * _log_int(rng, 32, 640)])
        if not 256 <= hidden <= 5120:
            continue
        side, n_tiles = rng.randint(8, 36), rng.choice([1, 1, 1, 2, 3, 5, 8])
        rows, cols = side, max(8, side + rng.choice([0, 0, 0, -3, 2, 5]))
        if rng.random() < 0.08:
            rows, n_tiles = rows * 8, 1
        grid = ("%d*" % n_tiles if n_tiles > 1 else "") + "%dx%d" % (rows, cols)
        stages = rng.choice([1, 2, 3, 3])
        smallest = min(rows, cols)
        w = rng.randint(2, min(8, smallest // 3) if smallest >= 9 else 2)
        windows = [max(1, w // (2 ** i)) for i in range(stages)]
        keep = [rng.choice([0.5, 0.5, 0.5, 0.55, 0.6, 0.75]) for _ in range(stages)]
        dtype = "fp32" if rng.random() < 0.1 else "bf16"
        kv = rng.choice(["head_major", "head_major", "token_major", "paged", "in_place", "paged_in_place"])
        packed = dtype == "bf16" and rng.random() < 0.2
        if packed and kv.startswith("paged"):
            kv = "in_place"
        case = _case(None, _log_int(rng, 1, 40), grid, _log_int(rng, 8, 300), hidden, heads, kv_heads, head_dim,
                     ",".join(map(str, windows)), ",".join(map(str, keep)),
                     xi=rng.choice(["full", "full", "full", "lse", "lse", "given", "uniform"]), dtype=dtype, kv=kv,
                     kv_mode=rng.choice(["merge", "merge", "merge", "gather"]), caches=rng.choice([1, 1, 2, 4]),
                     after=rng.choice([0, 0, rng.randint(1, 64)]), packed=packed, streams=rng.random() < 0.25)
        n = sum(r * c for r, c in _tiles(case))
        if n <= 9000 and n * case["batch"] >= 64 and _cost(case) <= 0.7 * limit:
            return case


# ----------------------------------------------------------------------------------------------------------- inputs

def _filter(size, device, sigma=3.0 / math.sqrt(2.0)):
    """[size, size] Gaussian smoothing with rows of unit length (variance is kept)."""
    x = torch.arange(size, device=device, dtype=torch.float32)
    f = torch.exp(-(x[:, None] - x[None, :]) ** 2 / (2 * sigma * sigma))
    return f / f.norm(dim=1, keepdim=True)


def _vision(tiles, channels, gen, device):
    """[tokens, channels]: a smooth field over every tile (neighbouring patches look alike, correlation length three
    patches) plus noise whose level differs from patch to patch, as flat and busy regions of an image do."""
    parts = []
    for rows, cols in tiles:
        white = torch.randn((rows, cols, channels), generator=gen, device=device)
        f = torch.matmul(_filter(rows, device), white.reshape(rows, -1)).reshape(rows, cols, channels)
        f = torch.matmul(_filter(cols, device), f)
        level = 0.05 + 0.75 * torch.rand((rows, cols, 1), generator=gen, device=device)
        f += level * torch.randn((rows, cols, channels), generator=gen, device=device)
        parts.append(f.reshape(rows * cols, channels))
    return torch.cat(parts)


def _rows(case, tiles, pos, channels, gen, device, dtype):
    """[B, text + cap + after, channels]: text rows, the vision rows at `pos` ([B, cap], -1 behind a sample's last
    token), text rows.  With pos = None the samples hold their whole grid."""
    b, nt, na = case["batch"], case["text"], case["after"]
    n_grid = sum(r * c for r, c in tiles)
    cap = n_grid if pos is None else pos.shape[1]
    out = torch.empty((b, nt + cap + na, channels), device=device, dtype=dtype)
    for i in range(b):
        vis = _vision(tiles, channels, gen, device)
        out[i, nt:nt + cap] = vis if pos is None else vis[pos[i].clamp(min=0).long()]
    out[:, :nt] = torch.randn((b, nt, channels), generator=gen, device=device)
    out[:, nt + cap:] = torch.randn((b, na, channels), generator=gen, device=device)
    return out


def _heads(x, heads, head_dim):
    """[B, N, heads * head_dim] -> [B, heads, N, head_dim], head-major in memory."""
    b, n, _ = x.shape
    return x.view(b, n, heads, head_dim).permute(0, 2, 1, 3).contiguous()


def _pack(x, lens, starts, total, axis):
    """[B, (H,) N, w] -> [1, (H,) total, w]: sample b's first lens[b] rows from row starts[b] on."""
    shape = list(x.shape)
    shape[0], shape[axis] = 1, total
    out = torch.zeros(shape, device=x.device, dtype=x.dtype)
    for i, (n, s) in enumerate(zip(lens, starts)):
        out[0].narrow(axis - 1, s, n).copy_(x[i].narrow(axis - 1, 0, n))
    return out


def _paged(x, blocks, gen):
    """[B, H, N, dh] -> (page pool [B * blocks, H, PAGE, dh], block table [B, blocks]), pages in shuffled order."""
    b, h, n, dh = x.shape
    table = torch.randperm(b * blocks, generator=gen, device=x.device).view(b, blocks)
    full = torch.zeros((b, h, blocks * PAGE, dh), device=x.device, dtype=x.dtype)
    full[:, :, :n] = x
    pool = torch.empty((b * blocks, h, PAGE, dh), device=x.device, dtype=x.dtype)
    pool[table.reshape(-1)] = full.view(b, h, blocks, PAGE, dh).permute(0, 2, 1, 3, 4).reshape(b * blocks, h, PAGE, dh)
    return pool, table.int()


def _caches(case, info, k, gen, device, layout):
    """The stage's K/V caches with their destinations: a list of (k_src, v_src, k_dst, v_dst, keywords)."""
    b, hk, dh = case["batch"], case["kv_heads"], case["head_dim"]
    n_out = case["text"] + info.cap_out + case["after"]
    found = []
    for layer in range(case["caches"]):
        ks = k if layer == 0 else torch.randn(k.shape, generator=gen, device=device).to(k.dtype)
        vs = torch.randn(k.shape, generator=gen, device=device).to(k.dtype)
        kw = {}
        if case["kv"].startswith("paged"):
            blocks = -(-(case["text"] + info.cap_in + case["after"]) // PAGE)
            ks, table = _paged(ks, blocks, gen)
            vs_pool = torch.empty_like(ks)
            vs_full = torch.zeros((b, hk, blocks * PAGE, dh), device=device, dtype=k.dtype)
            vs_full[:, :, :vs.shape[2]] = vs
            vs_pool[table.reshape(-1).long()] = vs_full.view(b, hk, blocks, PAGE, dh).permute(0, 2, 1, 3, 4).reshape(ks.shape)
            vs = vs_pool
            kw = dict(page_size=PAGE, src_block_table=table, dst_block_table=table)
            if case["kv"] == "paged":
                kw["dst_block_table"] = torch.randperm(b * blocks, generator=gen, device=device).view(b, blocks).int()
                kd, vd = torch.zeros_like(ks), torch.zeros_like(vs)
            else:
                kd, vd = ks, vs
        elif case["kv"] == "in_place":
            ks = ks.clone() if layer == 0 else ks          # compress_layer's K stays what it was
            kd, vd = ks, vs
        elif layout is not None:                           # packed, into a second buffer of reserved rows
            kd = torch.zeros((1, hk, b * n_out, dh), device=device, dtype=k.dtype)
            vd = torch.zeros_like(kd)
        else:
            kd = torch.zeros((b, hk, n_out, dh), device=device, dtype=k.dtype)
            vd = torch.zeros_like(kd)
        if case["kv"] == "token_major":
            ks, vs, kd, vd = (t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for t in (ks, vs, kd, vd))
        if layout is not None:
            kw.update(src_seq_start=layout["start"],
                      dst_seq_start=layout["start"] if case["kv"] == "in_place" else layout["start_out"])
        found.append((ks, vs, kd, vd, kw))
    return found


XI = {"full": L.XI_ATTN_FULL, "lse": L.XI_ATTN_LSE, "given": L.XI_GIVEN, "uniform": L.XI_UNIFORM}


def _event():
    e = torch.cuda.Event()
    e.record()                                             # torch makes the event when it is first recorded
    return e


def prepare(case, seed):
    device = torch.device("cuda")
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    tiles, (windows, keep) = _tiles(case), _schedule(case)
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    b, h, hk, dh, nt, na = (case[k] for k in ("batch", "heads", "kv_heads", "head_dim", "text", "after"))
    stages = len(windows)

    def plan_for(xi):
        return L.Plan(b, case["hidden"], h, hk, dh, 4 * stages, tiles, [4 * i + 2 for i in range(stages)], windows,
                      keep, nt + na, dtype=L.BF16 if case["dtype"] == "bf16" else L.FP32, xi_mode=XI[xi],
                      ragged_input=case["packed"])

    plan = plan_for(case["xi"])
    n_grid = sum(r * c for r, c in tiles)
    n_vis, pos, lens = None, None, None
    if case["packed"]:                                     # every sample keeps its own half to whole of the grid
        order = torch.rand((b, n_grid), generator=gen, device=device).argsort(dim=1)
        counts = [int(v) for v in torch.randint(n_grid // 2, n_grid + 1, (b,), generator=gen, device=device)]
        pos = torch.full((b, n_grid), -1, device=device, dtype=torch.int32)
        for i, n in enumerate(counts):
            pos[i, :n] = order[i, :n].sort().values.int()
        n_vis = torch.tensor(counts, device=device, dtype=torch.int32)
        lens = [nt + n + na for n in counts]
    state = dict(case=case, plan=plan, stages=[], side=None, aux=None)
    if case["streams"]:
        state["side"], state["aux"] = torch.cuda.Stream(), torch.cuda.Stream()
    for st in range(stages):
        info = plan.stage_info(st)
        hidden = _rows(case, tiles, pos, case["hidden"], gen, device, dtype)
        n_rows, n_out = hidden.shape[1], nt + info.cap_out + na
        q = k = None
        if case["xi"] in ("full", "lse"):
            q = _heads(_rows(case, tiles, pos, h * dh, gen, device, dtype), h, dh)
        k = _heads(_rows(case, tiles, pos, hk * dh, gen, device, dtype), hk, dh)
        layout, kw = None, dict(vis_begin=nt, n_text_after=na, n_vis=n_vis, pos=pos)
        if case["packed"]:
            if st > 0:
                lens = [n_rows] * b                        # rows reserved for what the stage before may leave
            starts = [sum(lens[:i]) for i in range(b)]
            total = b * n_rows                             # the token budget the buffers are sized for
            hidden, k = _pack(hidden, lens, starts, total, 1), _pack(k, lens, starts, total, 2)
            q = None if q is None else _pack(q, lens, starts, total, 2)
            layout = dict(start=torch.tensor(starts, device=device, dtype=torch.int32),
                          start_out=torch.arange(b, device=device, dtype=torch.int32) * n_out)
            kw.update(seq_start=layout["start"], seq_start_out=layout["start_out"],
                      hidden_out=torch.zeros((1, b * n_out, case["hidden"]), device=device, dtype=dtype))
        out = L.StageBuffers(plan, st, n_out, device)
        out.hidden_out.zero_()
        if q is not None:
            kw.update(q=q, k=k)
        if case["xi"] == "lse":                            # the row log-sum-exp of the layer's attention
            lse = torch.zeros(q.shape[:3], device=device, dtype=torch.float32)
            full = plan_for("full")
            L.compress_layer(full, st, hidden, L.StageBuffers(full, st, n_out, device), lse_out=lse, **kw)
            kw["lse"] = lse
        elif case["xi"] == "given":
            kw["xi"] = 0.05 + torch.rand((b, info.cap_in), generator=gen, device=device)
        if case["streams"]:
            kw.update(aux_stream=state["aux"], map_event=_event(), fork_event=_event(), join_event=_event())
        stage = dict(hidden=hidden, out=out, kw=kw, caches=_caches(case, info, k, gen, device, layout))
        state["stages"].append(stage)
        if st + 1 < stages:                                # where the next stage's tokens stand
            L.compress_layer(plan, st, hidden, out, **kw)
            pos, n_vis = out.pos_out, out.n_vis_out
    torch.cuda.synchronize()
    return state


def run(state):
    case, plan, side = state["case"], state["plan"], state["side"]
    mode = L.KV_MERGE if case["kv_mode"] == "merge" else L.KV_GATHER
    results = []
    for st, stage in enumerate(state["stages"]):
        out, kw = stage["out"], stage["kw"]
        L.compress_layer(plan, st, stage["hidden"], out, **kw)
        if side is not None:
            side.wait_event(kw["map_event"])
        for ks, vs, kd, vd, more in stage["caches"]:
            L.compact_kv(plan, st, out, ks, vs, kd, vd, vis_begin=kw["vis_begin"], n_text_after=kw["n_text_after"],
                         mode=mode, n_vis=kw["n_vis"], stream=side, **more)
        results.append([kw.get("hidden_out", out.hidden_out), out.n_vis_out, out.pos_out, out.dst, out.weight,
                        out.grp_off, out.grp_src, out.xi_out, out.status] + [t for c in stage["caches"] for t in c[2:4]])
    if side is not None:
        torch.cuda.current_stream().wait_stream(side)
    return results
