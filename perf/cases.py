"""The work that users of this library have it do, as cases that can be timed and compared.

Every case is one call sequence of the public Python binding over a seeded synthetic input of the repository's own
kind: Q and K are a smooth low-frequency field over the (T, Hg, Wg) latent grid plus white noise, V is white noise.
"path" names the sequence:

  attention   block selection, then the bf16 forward over the kept lists
  lists       the bf16 forward alone, over lists the caller already has (a random block mask with the diagonal kept)
  fp8         quantise + pool Q and K, quantise V, top-k on the pooled means, FP8 forward
  causal      selection and forward restricted to a causal window of frames, with the log-sum-exp (a decoder that
              emits frames one after another merges on it)
  module      selection, forward, low-rank state, gated apply: the attention module's output in two passes
  gated       selection, low-rank state, the forward with the gate in its epilogue: the same output in one pass
  bricks      raster tokens gathered into padded 3-D bricks, selection and forward there, gathered back
  activation  per-token FP8 quantisation of an activation tensor
  host        the whole chain on host buffers (copies in, kernels, copy out)

The workspaces and outputs are the ones the calls allocate by themselves (host: the pinned output and the device arena
are the caller's, as the call intends).
"""
import math

import torch

import paper_2609_23153_b200 as sa

RANK = 64            # of the compensation branch
LARGEST_FLOPS = 4.0 * 128 * 40 * 75600 ** 2    # dense attention at the largest shape


def listed():
    def case(name, path, H, grid, sparsity, **more):
        c = dict(name=name, path=path, B=1, H=H, T=grid[0], Hg=grid[1], Wg=grid[2], d=128, block=128, sparsity=sparsity,
                 layout="bhnd")
        c.update(more)
        return c

    w480, w720 = (21, 30, 52), (21, 45, 80)      # 480 x 832 and 720 x 1280 video, 81 frames, on the latent grid
    return [
        # the unit-test sized call: one short clip, explicit lists, d = 64; launch latency and idle SMs are all there is
        case("tiny_lists", "lists", 2, (2, 32, 32), 0.5, d=64, block=64),
        # a few frames at low resolution, ragged last block: selection and forward together are a handful of launches
        case("small_attention", "attention", 3, (5, 12, 20), 0.8),
        # the 1.3B model's layer at 480P: the everyday call
        case("w480_attention", "attention", 12, w480, 0.90),
        # the same layer in FP8, on the [B, N, H, d] tensors that a projection leaves
        case("w480_fp8", "fp8", 12, w480, 0.90, layout="bnhd"),
        # auto-regressive generation over an odd grid: window of three frames, log-sum-exp returned
        case("odd_causal", "causal", 12, (13, 37, 51), 0.85, window=3),
        # odd grid in brick order (every brick padded to a block), gathers included
        case("odd_bricks", "bricks", 12, (17, 33, 50), 0.90, bt=3, bh=5, bw=8),
        # host buffers in, host buffer out: what a process without a resident pipeline calls
        case("w480_host", "host", 12, w480, 0.90),
        # the 14B model's layer at 720P and 97 %: the headline workload
        case("w720_attention", "attention", 40, w720, 0.97),
        # the same in FP8
        case("w720_fp8", "fp8", 40, w720, 0.97),
        # the same with 64-token blocks, the size the paper trained with
        case("w720_block64", "attention", 40, w720, 0.97, block=64),
        # the layer's whole output with the compensation branch
        case("w720_module", "module", 40, w720, 0.97),
        # no sparsity: the baseline a user compares with, and the upper end of the sparsity sweep
        case("w720_dense", "lists", 40, w720, 0.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any path, heads 1-40, latent grids from a few frames of thumbnails to the 720P grid."""
    while True:
        path = rng.choice(["attention", "attention", "fp8", "fp8", "lists", "causal", "module", "gated", "bricks",
                           "activation", "host"])
        T = rng.randint(2, 21)
        Hg, Wg = _log_int(rng, 8, 45), _log_int(rng, 12, 80)
        H = _log_int(rng, 1, 40)
        d, block = 128, 128
        if path in ("attention", "fp8", "causal", "lists") and rng.random() < 0.3:
            block = 64
            if path in ("attention", "lists", "causal") and rng.random() < 0.4:
                d = 64
        n = T * Hg * Wg
        c = dict(path=path, B=rng.choice([1, 1, 1, 2]), H=H, T=T, Hg=Hg, Wg=Wg, d=d, block=block,
                 sparsity=rng.choice([0.0, 0.5, 0.75, 0.8, 0.9, 0.95, 0.97]),
                 layout=rng.choice(["bhnd", "bhnd", "bnhd"]))
        if path == "causal":
            c["window"] = rng.randint(1, 4)
        if path == "bricks":
            c["bt"], c["bh"], c["bw"] = rng.choice([(3, 5, 8), (2, 8, 8), (4, 4, 8)])
        if path == "host":
            c["layout"] = "bhnd"
        if n < 1000 or c["B"] * H * n > 40 * 75600 or work(c)["flops"] > LARGEST_FLOPS:
            continue
        if path == "host" and c["B"] * H * n > 12 * 32760:
            continue                                   # pinned buffers that take longer to make than to use
        return c


def _bricks(case):
    """(bricks, tokens of a brick): every brick of the grid takes one block."""
    return (-(-case["T"] // case["bt"])) * (-(-case["Hg"] // case["bh"])) * (-(-case["Wg"] // case["bw"]))


def _budget(case):
    """(blocks per head, kept blocks per query block): the nearest integer to (1 - s) * nb, at least one."""
    n = case["T"] * case["Hg"] * case["Wg"]
    nb = _bricks(case) if case["path"] == "bricks" else -(-n // case["block"])
    return nb, max(1, int(math.floor((1.0 - case["sparsity"]) * nb + 0.5)))


def work(case):
    B, H, d, block = case["B"], case["H"], case["d"], case["block"]
    n = case["T"] * case["Hg"] * case["Wg"]
    nb, topk = _budget(case)
    row = B * H * n * d
    if case["path"] == "activation":
        return {"bytes": 3 * row + 4 * B * H * n, "flops": 2 * row}
    keys = min(topk * block, n)
    if case["path"] == "bricks":
        keys = min(topk * case["bt"] * case["bh"] * case["bw"], n)
    flops = 4 * row * keys
    if case["path"] == "causal":                       # a row sees at most its window's frames; the first frames see fewer
        frame = case["Hg"] * case["Wg"]
        flops = sum(4 * B * H * frame * d * min(keys, frame * min(f + 1, case["window"])) for f in range(case["T"]))
    size = 2 * 4 * row                                 # q, k, v read, the output written
    if case["path"] not in ("host", "bricks"):
        size += 4 * B * H * nb * (topk + 1)            # kept lists, written or read
    if case["path"] == "causal":
        size += 4 * B * H * n
    if case["path"] in ("module", "gated"):
        size += 4 * B * H * n + 4 * H * RANK * d + 4 * B * H * RANK * d
        flops += 2 * 4 * row * RANK                    # two projections, the state's and the branch's product
    return {"bytes": size, "flops": flops}


def tolerance(case):
    if case["path"] == "activation":
        return "exact"
    # 2.3e-3 of the result is what the bf16 outputs are off the 64-bit reference (P and the output are rounded to bf16);
    # FP8 rounds P to a 3-bit mantissa: 2.6e-2 off the reference.  Lists and counts are whole numbers and stay the same.
    return {"rel": 3e-2 if case["path"] == "fp8" else 1e-2}


def _fields(case, gen):
    """q, k, v bf16 [B, H, N, d]: eight sinusoids over the grid (four without x-frequency) + noise, v noise."""
    B, H, d = case["B"], case["H"], case["d"]
    T, Hg, Wg = case["T"], case["Hg"], case["Wg"]
    n = T * Hg * Wg
    dev = "cuda"
    i = torch.arange(n, device=dev)
    pos = torch.stack([(i // (Wg * Hg)) / T, (i // Wg % Hg) / Hg, (i % Wg) / Wg]).float()       # [3, n]
    shape = (B, n, H, d) if case["layout"] == "bnhd" else (B, H, n, d)
    q, k, v = (torch.empty(shape, dtype=torch.bfloat16, device=dev) for _ in range(3))
    if case["layout"] == "bnhd":
        q, k, v = (t.permute(0, 2, 1, 3) for t in (q, k, v))

    def rand(*s):
        return torch.rand(s, generator=gen, device=dev)

    for b in range(B):
        for h in range(H):
            f = torch.stack([torch.floor(3 * rand(8)), torch.floor(4 * rand(8)), torch.floor(4 * rand(8))], 1)
            f[:4, 2] = 0
            f[:, 1] += (f.sum(1) == 0)                 # no constant component
            theta = 2 * math.pi * (f @ pos)            # [8, n]
            wave = torch.cat([torch.sin(theta), torch.cos(theta)])                               # [16, n]
            phi = 2 * math.pi * rand(8, d)
            for x, p in ((q, phi), (k, phi + (rand(8, d) - 0.5) * (math.pi / 2))):
                x[b, h] = wave.T @ (0.5 * torch.cat([torch.cos(p), torch.sin(p)])) + 0.5 * torch.randn(
                    (n, d), generator=gen, device=dev)
            v[b, h] = torch.randn((n, d), generator=gen, device=dev)
    return q, k, v


def _rope_schedule(d):
    """Three-axis rotary schedule of this model family (22 / 21 / 21 pairs at d = 128), cut to the branch's rank."""
    pairs = [(a, 10000.0 ** (-p / m)) for a, m in enumerate((d // 2 - 2 * (d // 6), d // 6, d // 6)) for p in range(m)]
    axis, freq = zip(*pairs[: RANK // 2])
    return torch.tensor(axis, dtype=torch.int32), torch.tensor(freq, dtype=torch.float32)


def prepare(case, seed):
    B, H, d, block = case["B"], case["H"], case["d"], case["block"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    nb, topk = _budget(case)
    grid = (case["T"], case["Hg"], case["Wg"])
    n = grid[0] * grid[1] * grid[2]
    s = {"path": case["path"], "block": block, "topk": topk, "grid": grid}
    if case["path"] == "activation":
        s["x"] = _fields(case, gen)[0]
        return s
    s["q"], s["k"], s["v"] = _fields(case, gen)
    if case["path"] == "lists":
        if topk == nb:
            s["idx"] = torch.arange(nb, dtype=torch.int32, device="cuda").expand(B, H, nb, nb).contiguous()
        else:
            r = torch.rand((B, H, nb, nb), generator=gen, device="cuda")
            r.diagonal(dim1=2, dim2=3).fill_(2.0)      # the query block's own key block is always kept
            s["idx"] = r.topk(topk, dim=-1).indices.sort(dim=-1).values.to(torch.int32)
        s["cnt"] = torch.full((B, H, nb), topk, dtype=torch.int32, device="cuda")
    elif case["path"] == "causal":
        s["frame"], s["window"] = grid[1] * grid[2], case["window"]
    elif case["path"] == "bricks":
        s["gather"], s["valid"], s["scatter"] = sa.brick_layout(grid, (case["bt"], case["bh"], case["bw"]), block)
    elif case["path"] in ("module", "gated"):
        s["pq"], s["pk"] = ((torch.randn((H, RANK, d), generator=gen, device="cuda") / math.sqrt(d)).to(torch.bfloat16)
                            for _ in range(2))
        s["gate"] = 0.3 * torch.rand((B, H, n), generator=gen, device="cuda")
        s["axis"], s["freq"] = _rope_schedule(d)
    elif case["path"] == "host":
        s["q"], s["k"], s["v"] = (t.cpu().pin_memory() for t in (s["q"], s["k"], s["v"]))
        s["out"] = torch.empty_like(s["q"]).pin_memory()
        s["arena"] = torch.empty(sa.arena_bytes(sa.make_shape(s["q"], block), sa.BF16, topk), dtype=torch.uint8,
                                 device="cuda")
    return s


def run(s):
    block, topk = s["block"], s["topk"]
    if s["path"] == "activation":
        return sa.quant_fp8_per_token(s["x"])
    q, k, v = s["q"], s["k"], s["v"]
    if s["path"] == "lists":
        return sa.fwd(q, k, v, s["idx"], s["cnt"], block)
    if s["path"] == "host":
        return sa.attention_host(q, k, v, block, topk, out=s["out"], arena=s["arena"])
    if s["path"] == "fp8":
        ws = sa.alloc_workspace(sa.make_shape(q, block), 0, topk, q.device)
        cq, sq = sa.quant_fp8_pooled(q, block, False, ws)
        ck, sk = sa.quant_fp8_pooled(k, block, True, ws)
        cv, sv = sa.quant_fp8(v, block)
        idx, cnt = sa.select_pooled(q, block, topk, ws)
        return sa.fwd(cq, ck, cv, idx, cnt, block, scales=(sq, sk, sv)), idx, cnt
    if s["path"] == "causal":
        idx, cnt = sa.select(q, k, block, topk, frame_tokens=s["frame"], window=s["window"])
        out, lse = sa.fwd(q, k, v, idx, cnt, block, return_lse=True, frame_tokens=s["frame"], window=s["window"])
        return out, lse, idx, cnt
    if s["path"] == "bricks":
        qb, kb, vb = (sa.gather_tokens(t, s["gather"]) for t in (q, k, v))
        idx, cnt = sa.select(qb, kb, block, topk, block_valid=s["valid"])
        out = sa.fwd(qb, kb, vb, idx, cnt, block, block_valid=s["valid"])
        return sa.gather_tokens(out, s["scatter"]), idx, cnt
    idx, cnt = sa.select(q, k, block, topk)
    if s["path"] == "attention":
        return sa.fwd(q, k, v, idx, cnt, block), idx, cnt
    state = sa.comp_state(k, v, s["pk"], s["grid"], s["axis"], s["freq"])
    if s["path"] == "gated":
        out = sa.fwd_gated(q, k, v, idx, cnt, s["pq"], state, s["gate"], s["grid"], s["axis"], s["freq"])
    else:
        out = sa.fwd(q, k, v, idx, cnt, block)
        out = sa.comp_apply(q, s["pq"], state, s["gate"], out, s["grid"], s["axis"], s["freq"])
    return out, state, idx, cnt


EXACT_FLOPS = 1e13          # above it the 64-bit evaluation takes too long


def _pooled(x, block, valid=None):
    """Block means [nb, d] of [N, d], over the first valid[b] rows of block b (default: those below N)."""
    n, d = x.shape
    nb = -(-n // block)
    rows = torch.arange(nb * block, device=x.device).view(nb, block)
    real = rows < n if valid is None else (rows % block) < valid[:, None]
    x = torch.nn.functional.pad(x, (0, 0, 0, nb * block - n)).view(nb, block, d)
    return (x * real[..., None]).sum(1) / real.sum(1, keepdim=True)


def _chosen(q, k, block, topk, valid=None, frame=0, window=0):
    """Top-k key blocks of every query block of one head by the product of block means; -1 beyond the candidates."""
    n = q.shape[0]
    score = _pooled(q, block, valid) @ _pooled(k, block, valid).T
    if frame:
        first = torch.arange(0, n, block, device=q.device)
        last = (first + block - 1).clamp(max=n - 1)
        lo, hi = ((first // frame - window + 1).clamp(min=0) * frame)[:, None], (last // frame + 1)[:, None] * frame
        score = score.masked_fill((first[None] >= hi) | (last[None] < lo), -math.inf)
    best, idx = score.topk(topk, dim=1)
    return torch.where(best == -math.inf, -1, idx)


def _attend(q, k, v, idx, block, valid=None, frame=0, window=0):
    """Softmax attention of one head over the listed key blocks, [N, d] in 64 bits -> output and log-sum-exp."""
    n, d = q.shape
    nb, topk = idx.shape
    pad = (0, 0, 0, nb * block - n)
    q, k, v = (torch.nn.functional.pad(t, pad).view(nb, block, d) for t in (q, k, v))
    out, lse = torch.empty_like(q), torch.empty((nb, block), dtype=q.dtype, device=q.device)
    lane = torch.arange(block, device=q.device)
    step = max(1, int(1e8) // (topk * block * block))
    for i in range(0, nb, step):
        at = idx[i: i + step].clamp(min=0)
        c = at.shape[0]
        key = at[..., None] * block + lane                                     # [c, topk, block]
        real = (idx[i: i + step] >= 0)[..., None] & (key < n)
        if valid is not None:
            real &= lane < valid[at][..., None]
        real = real.view(c, 1, -1)
        if frame:
            row = (i + torch.arange(c, device=q.device))[:, None] * block + lane
            fq, fk = (row.clamp(max=n - 1) // frame)[..., None], (key // frame).view(c, 1, -1)
            real = real & (fk <= fq) & (fk > fq - window)
        s = (q[i: i + step] @ k[at].view(c, -1, d).mT) * (1.0 / math.sqrt(d))
        s.masked_fill_(~real, -math.inf)
        lse[i: i + step] = torch.logsumexp(s, -1)
        s.sub_(lse[i: i + step].nan_to_num(neginf=0.0)[..., None]).exp_()
        out[i: i + step] = s @ v[at].view(c, -1, d)
    return out.view(-1, d)[:n], lse.view(-1)[:n]


def _dequantised(x, block):
    """What one head's E4M3 codes with a scale per block stand for, in 64 bits."""
    n, d = x.shape
    x = torch.nn.functional.pad(x.float(), (0, 0, 0, -n % block)).view(-1, block, d)
    amax = x.abs().amax((1, 2), keepdim=True).clamp(min=1e-12)
    return ((x * (448.0 / amax)).to(torch.float8_e4m3fn).double() * (amax / 448.0).double()).view(-1, d)[:n]


def _feature(x, p, grid, axis, freq):
    """Rotated silu features [N, rank] of one head's rows."""
    i = torch.arange(x.shape[0], device=x.device)
    pos = torch.stack([i // (grid[1] * grid[2]), i // grid[2] % grid[1], i % grid[2]], 1).double()
    a = pos[:, axis.long().to(x.device)] * freq.double().to(x.device)
    z = torch.nn.functional.silu(x @ p.T).view(-1, RANK // 2, 2)
    even, odd = z.unbind(2)
    return torch.stack([even * a.cos() - odd * a.sin(), even * a.sin() + odd * a.cos()], 2).view(-1, RANK)


def _brick_rows(case):
    """(raster token at each row of the brick order, -1 for padding; tokens of each brick)."""
    T, Hg, Wg, bt, bh, bw = (case[a] for a in ("T", "Hg", "Wg", "bt", "bh", "bw"))
    n = torch.arange(T * Hg * Wg).view(T, Hg, Wg)
    rows, valid = [], []
    for t in range(0, T, bt):
        for y in range(0, Hg, bh):
            for x in range(0, Wg, bw):
                cells = n[t: t + bt, y: y + bh, x: x + bw].reshape(-1)
                valid.append(cells.numel())
                rows.append(torch.nn.functional.pad(cells, (0, case["block"] - cells.numel()), value=-1))
    return torch.cat(rows).cuda(), torch.tensor(valid, device="cuda")


def exact(case, seed):
    """What run() returns, in 64 bits from the same inputs; no counterpart for lists and codes."""
    if work(case)["flops"] > EXACT_FLOPS:
        return None
    s = prepare(case, seed)
    path, block = s["path"], s["block"]
    if path == "activation":
        return None, s["x"].double().abs().amax(-1).clamp(min=1e-12) / 448.0
    q, k, v = (t.cuda() for t in (s["q"], s["k"], s["v"]))
    B, H, n, d = q.shape
    out = torch.empty((B, H, n, d), dtype=torch.float64, device="cuda")
    lse, state = out.new_empty((B, H, n)), out.new_empty((B, H, RANK, d))
    rows, valid = _brick_rows(case) if path == "bricks" else (None, None)
    window = (s["frame"], s["window"]) if path == "causal" else (0, 0)
    for b in range(B):
        for h in range(H):
            x, y, z = (t[b, h].double() for t in (q, k, v))
            if path == "bricks":
                x, y, z = (t[rows.clamp(min=0)] * (rows >= 0)[:, None] for t in (x, y, z))
            idx = s["idx"][b, h].long() if path == "lists" else _chosen(x, y, block, s["topk"], valid, *window)
            if path == "fp8":
                x, y, z = (_dequantised(t, block) for t in (x, y, z))
            o, lse[b, h] = _attend(x, y, z, idx, block, valid, *window) if path != "bricks" else (
                _attend(x, y, z, idx, block, valid)[0], 0.0)
            if path == "bricks":
                out[b, h, rows[rows >= 0]] = o[rows >= 0]
                continue
            if path in ("module", "gated"):
                args = s["grid"], s["axis"], s["freq"]
                state[b, h] = _feature(y, s["pk"][h].double(), *args).T @ z
                low = _feature(x, s["pq"][h].double(), *args) @ state[b, h]
                low = low / (low.square().mean(-1, keepdim=True) + 1e-6).sqrt()
                o = o + s["gate"][b, h].double()[:, None] * o.square().mean(-1, keepdim=True).sqrt() * low
            out[b, h] = o
    if path in ("lists", "host"):
        return out
    if path == "causal":
        return out, lse, None, None
    if path in ("module", "gated"):
        return out, state, None, None
    return out, None, None
