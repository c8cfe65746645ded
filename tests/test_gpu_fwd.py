"""GPU parity: sparkattn_fwd against the fp64 CPU oracle.

Tolerances (from the acceptance statement of the task): bf16 output relative
RMS error <= 1e-2 and max abs error <= 3e-2; FP8 output (oracle evaluated on
the same quantised inputs) relative RMS error <= 5e-2.  lse: abs <= 1e-2."""
import math

import pytest
import torch

import oracle
import paper_2609_23153_b200 as sa
import workloads

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
BF16_RELRMS, BF16_MAXABS, FP8_RELRMS, LSE_ABS = 1e-2, 3e-2, 5e-2, 1e-2
FP8_ROW_RELRMS = 1.5e-1   # per-row guard beside the aggregate FP8 bound


def _errors(got, ref):
    got, ref = got.double(), ref.double()
    relrms = math.sqrt(float(((got - ref) ** 2).sum()) / max(float((ref ** 2).sum()), 1e-300))
    return relrms, float((got - ref).abs().max())


def _compare_items(out_dev, lse_dev, ref_out, ref_lse, items, block, N, tol_rel, tol_abs, lse_tol=LSE_ABS):
    """out_dev [H,N,d] (device), ref_out [n_items, block, d] fp64."""
    got, ref, gl, rl = [], [], [], []
    for n, (h, qb) in enumerate(items):
        r0, r1 = qb * block, min(N, (qb + 1) * block)
        got.append(out_dev[h, r0:r1].cpu()); ref.append(ref_out[n, : r1 - r0])
        if lse_dev is not None:
            gl.append(lse_dev[h, r0:r1].cpu()); rl.append(ref_lse[n, : r1 - r0])
    relrms, maxabs = _errors(torch.cat(got), torch.cat(ref))
    assert relrms <= tol_rel, f"relative RMS {relrms:.3e} > {tol_rel}"
    if tol_abs is not None:
        assert maxabs <= tol_abs, f"max abs {maxabs:.3e} > {tol_abs}"
    else:
        # FP8 has no absolute bound: guard every row by itself so that one wrong row cannot hide in the aggregate
        g, r = torch.cat(got).double(), torch.cat(ref).double()
        rows = (((g - r) ** 2).sum(-1) / (r ** 2).sum(-1).clamp_min(1e-300)).sqrt()
        assert float(rows.max()) <= FP8_ROW_RELRMS, f"worst row relative RMS {float(rows.max()):.3e} > {FP8_ROW_RELRMS}"
    if lse_dev is not None:
        dl = (torch.cat(gl).double() - torch.cat(rl)).abs().max().item()
        assert dl <= lse_tol, f"lse abs error {dl:.3e}"
    return relrms, maxabs


def test_tiny_workload_full_parity():
    w = workloads.TINY
    q, k, v = workloads.tiny_inputs(w)
    idx, cnt = workloads.random_block_mask(w.B, w.H, w.nb, w.topk)
    assert w.topk == 16
    out, lse = sa.fwd(q.to(DEV), k.to(DEV), v.to(DEV), idx.to(DEV), cnt.to(DEV), w.block,
                      return_lse=True, check_status=True)
    ref_out, ref_lse = oracle.attention(q[0], k[0], v[0], idx[0], cnt[0], w.block)
    items = [(h, i) for h in range(w.H) for i in range(w.nb)]
    _compare_items(out[0], lse[0], ref_out, ref_lse, items, w.block, w.N, BF16_RELRMS, BF16_MAXABS)


def _small(cfg_id, H, d, grid, block, sparsity):
    return workloads.small_structured(H=H, d=d, grid=grid, block=block, sparsity=sparsity, cfg_id=cfg_id)


SMALL = [
    _small(31, 3, 128, (5, 12, 20), 128, 0.7),    # N=1200, tail 48
    _small(32, 2, 128, (3, 16, 16), 128, 0.5),    # N=768, no tail
    _small(33, 2, 64, (3, 10, 21), 64, 0.8),      # N=630, tail 54
    _small(34, 2, 128, (4, 11, 23), 128, 0.0),    # dense, N=1012, tail 116
    _small(35, 1, 128, (1, 1, 5), 128, 0.0),      # single ragged block of 5 tokens
    _small(39, 2, 128, (4, 9, 25), 64, 0.75),     # d=128 with the paper's 64x64 blocks: N=900, tail 4
]


@pytest.mark.parametrize("w", SMALL, ids=lambda w: f"{w.name}-N{w.N}-d{w.d}-s{w.sparsity}")
def test_small_structured_full_parity_bf16(w):
    q, k, v = workloads.structured_qkv(w)
    idx, cnt = oracle.select(q[0], k[0], w.block, w.topk)
    out, lse = sa.fwd(q.to(DEV), k.to(DEV), v.to(DEV), idx[None].to(DEV), cnt[None].to(DEV), w.block,
                      return_lse=True, check_status=True)
    ref_out, ref_lse = oracle.attention(q[0], k[0], v[0], idx, cnt, w.block)
    items = [(h, i) for h in range(w.H) for i in range(w.nb)]
    _compare_items(out[0], lse[0], ref_out, ref_lse, items, w.block, w.N, BF16_RELRMS, BF16_MAXABS)


def test_variable_counts_empty_lists_permutation_and_scale():
    w = _small(36, 2, 128, (4, 12, 16), 128, 0.5)   # N=768, nb=6
    q, k, v = workloads.structured_qkv(w)
    g = torch.Generator().manual_seed(5)
    kmax = 5
    idx = torch.stack([torch.stack([torch.randperm(w.nb, generator=g)[:kmax] for _ in range(w.nb)])
                       for _ in range(w.H)]).to(torch.int32)            # unsorted lists
    cnt = torch.randint(0, kmax + 1, (w.H, w.nb), generator=g, dtype=torch.int32)
    cnt[0, 0] = 0; cnt[1, 3] = kmax
    qd, kd, vd = q.to(DEV), k.to(DEV), v.to(DEV)
    out, lse = sa.fwd(qd, kd, vd, idx[None].to(DEV), cnt[None].to(DEV), w.block, softmax_scale=0.05,
                      return_lse=True, check_status=True)
    ref_out, ref_lse = oracle.attention(q[0], k[0], v[0], idx, cnt, w.block, softmax_scale=0.05)
    items = [(h, i) for h in range(w.H) for i in range(w.nb) if cnt[h, i] > 0]
    sel = [n for n, (h, i) in enumerate((h, i) for h in range(w.H) for i in range(w.nb)) if cnt[h, i] > 0]
    _compare_items(out[0], lse[0], ref_out[sel], ref_lse[sel], items, w.block, w.N, BF16_RELRMS, BF16_MAXABS)
    for h in range(w.H):
        for i in range(w.nb):
            if cnt[h, i] == 0:
                rows = slice(i * w.block, (i + 1) * w.block)
                assert torch.all(out[0, h, rows] == 0) and torch.all(torch.isneginf(lse[0, h, rows]))
    # kept_cnt = NULL means every list is full; sorting the lists must not change the result beyond rounding
    out_a = sa.fwd(qd, kd, vd, idx[None].to(DEV), None, w.block)
    out_b = sa.fwd(qd, kd, vd, torch.sort(idx, dim=-1).values[None].to(DEV), None, w.block)
    rel, _ = _errors(out_a.cpu(), out_b.cpu())
    assert rel < 5e-3


def test_bad_index_is_reported_and_skipped():
    w = _small(37, 1, 128, (2, 8, 16), 128, 0.0)   # N=256, nb=2
    q, k, v = workloads.structured_qkv(w)
    idx = torch.tensor([[[[0, 7], [-1, 1]]]], dtype=torch.int32)
    ws = torch.zeros(sa.workspace_bytes(sa.make_shape(q, w.block), 1, 2), dtype=torch.uint8, device=DEV)
    out = sa.fwd(q.to(DEV), k.to(DEV), v.to(DEV), idx.to(DEV), None, w.block, workspace=ws)
    assert sa.read_status(ws) == sa.E_BAD_INDEX
    good = torch.tensor([[[0, 0], [1, 0]]], dtype=torch.int32)
    ref_out, _ = oracle.attention(q[0], k[0], v[0], good, torch.ones((1, 2), dtype=torch.int32), w.block)
    _compare_items(out[0], None, ref_out, None, [(0, 0), (0, 1)], w.block, w.N, BF16_RELRMS, BF16_MAXABS)
    # the next call on the same workspace starts clean
    sa.fwd(q.to(DEV), k.to(DEV), v.to(DEV), good[None].to(DEV), None, w.block, workspace=ws)
    assert sa.read_status(ws) == sa.OK


def test_strided_layout_and_batches_bf16():
    H, d, block = 2, 128, 128
    ws_ = [_small(40 + b, H, d, (3, 9, 14), block, 0.6) for b in range(2)]   # N=378, nb=3
    qs, ks, vs = zip(*[workloads.structured_qkv(w) for w in ws_])
    q, k, v = torch.cat(qs), torch.cat(ks), torch.cat(vs)
    w = ws_[0]
    idxs, cnts = zip(*[oracle.select(q[b], k[b], block, w.topk) for b in range(2)])
    idx, cnt = torch.stack(idxs), torch.stack(cnts)
    to_bnhd = lambda t: t.permute(0, 2, 1, 3).contiguous().to(DEV).permute(0, 2, 1, 3)
    out = sa.fwd(to_bnhd(q), to_bnhd(k), to_bnhd(v), idx.to(DEV), cnt.to(DEV), block, check_status=True)
    assert out.stride() == to_bnhd(q).stride()
    items = [(h, i) for h in range(H) for i in range(w.nb)]
    for b in range(2):
        ref_out, _ = oracle.attention(q[b], k[b], v[b], idx[b], cnt[b], block)
        _compare_items(out[b], None, ref_out, None, items, block, w.N, BF16_RELRMS, BF16_MAXABS)


def test_deterministic_and_rows_past_n_untouched():
    w = _small(38, 2, 128, (3, 10, 17), 128, 0.5)   # N=510, tail 126
    q, k, v = (t.to(DEV) for t in workloads.structured_qkv(w))
    idx, cnt = sa.select(q, k, w.block, w.topk)
    pad = torch.full((1, w.H, w.N + 64, w.d), 7.0, dtype=torch.bfloat16, device=DEV)
    qp = torch.zeros_like(pad); kp = torch.zeros_like(pad); vp = torch.zeros_like(pad)
    qp[:, :, : w.N] = q; kp[:, :, : w.N] = k; vp[:, :, : w.N] = v
    kp[:, :, w.N:] = 100.0; vp[:, :, w.N:] = 1e4        # poison behind the valid range
    a = sa.fwd(qp[:, :, : w.N], kp[:, :, : w.N], vp[:, :, : w.N], idx, cnt, w.block, out=pad[:, :, : w.N]).clone()
    assert torch.all(pad[:, :, w.N:] == 7.0)
    b = sa.fwd(q, k, v, idx, cnt, w.block)
    assert torch.equal(a, b)


@pytest.mark.parametrize("w", [SMALL[0], SMALL[1], SMALL[3], SMALL[5]], ids=lambda w: f"{w.name}-N{w.N}-b{w.block}-s{w.sparsity}")
def test_small_structured_full_parity_fp8(w):
    q, k, v = workloads.structured_qkv(w)
    idx, cnt = oracle.select(q[0], k[0], w.block, w.topk)      # selection always reads bf16
    dev = [t.to(DEV) for t in (q, k, v)]
    cs = [sa.quant_fp8(t, w.block) for t in dev]
    codes = [c for c, _ in cs]; scales = tuple(s for _, s in cs)
    out, lse = sa.fwd(codes[0], codes[1], codes[2], idx[None].to(DEV), cnt[None].to(DEV), w.block,
                      scales=scales, return_lse=True, check_status=True)
    ref_out, ref_lse = oracle.attention(codes[0][0].cpu(), codes[1][0].cpu(), codes[2][0].cpu(), idx, cnt, w.block,
                                        scales=tuple(s[0].cpu() for s in scales))
    items = [(h, i) for h in range(w.H) for i in range(w.nb)]
    _compare_items(out[0], lse[0], ref_out, ref_lse, items, w.block, w.N, FP8_RELRMS, None, lse_tol=2e-2)


@pytest.mark.parametrize("seed,kmax,block", [(0, 3, 128), (1, 6, 128), (2, 3, 64), (3, 7, 64)])
def test_persistent_path_short_and_empty_lists(seed, kmax, block):
    """bf16, d = 128 with more work items than SMs: every CTA of the persistent kernel walks several items
    whose kept lists have 0, 1, 2, ... blocks (item boundaries, hand-over of the row sums between the two
    softmax warpgroups, empty items), ragged last block included.  With 64-token blocks the items are
    pairs of query blocks over the merged lists (one list empty, disjoint lists, odd merged length, an odd
    number of query blocks).  Compared in full against the oracle, and two runs must agree bitwise."""
    grid = (5, 18, 19) if seed == 3 else (5, 18, 18)        # N = 1620: 13 (ragged) or 26 blocks; N = 1710: 27 blocks of 64
    w = _small(41 + seed, 3, 128, grid, block, 0.0)
    w = workloads.Workload(w.name, w.cfg_id, 1, 12 if block == 128 else 13, w.d, w.grid, w.block, w.sparsity)   # > 148 items
    q, k, v = workloads.structured_qkv(w)
    g = torch.Generator().manual_seed(100 + seed)
    idx = torch.stack([torch.stack([torch.randperm(w.nb, generator=g)[:kmax] for _ in range(w.nb)]) for _ in range(w.H)]).to(torch.int32)
    cnt = torch.randint(0, kmax + 1, (w.H, w.nb), generator=g, dtype=torch.int32)
    cnt[0, 0] = 0; cnt[0, 1] = 1; cnt[0, 2] = 1; cnt[0, 3] = 2; cnt[0, 4] = 0; cnt[0, 5] = 0; cnt[0, 6] = kmax
    qd, kd, vd = q.to(DEV), k.to(DEV), v.to(DEV)
    out, lse = sa.fwd(qd, kd, vd, idx[None].to(DEV), cnt[None].to(DEV), w.block, return_lse=True, check_status=True)
    out2, lse2 = sa.fwd(qd, kd, vd, idx[None].to(DEV), cnt[None].to(DEV), w.block, return_lse=True, check_status=True)
    assert torch.equal(out, out2) and torch.equal(lse.view(torch.int32), lse2.view(torch.int32))
    ref_out, ref_lse = oracle.attention(q[0], k[0], v[0], idx, cnt, w.block)
    items = [(h, i) for h in range(w.H) for i in range(w.nb) if cnt[h, i] > 0]
    sel = [n for n, (h, i) in enumerate((h, i) for h in range(w.H) for i in range(w.nb)) if cnt[h, i] > 0]
    _compare_items(out[0], lse[0], ref_out[sel], ref_lse[sel], items, w.block, w.N, BF16_RELRMS, BF16_MAXABS)
    for h in range(w.H):
        for i in range(w.nb):
            if cnt[h, i] == 0:
                rows = slice(i * w.block, min(w.N, (i + 1) * w.block))
                assert torch.all(out[0, h, rows] == 0) and torch.all(torch.isneginf(lse[0, h, rows]))


@pytest.mark.parametrize("block,kmax", [(128, 33), (128, 4), (64, 5), (64, 40)])
def test_bad_indices_are_dropped_and_reported(block, kmax):
    """d = 128: an index outside [0, nb) is dropped where the lists are cleaned and reported at the end of the CTA (64-token
    blocks: pairs of lists, one with a bad index, an odd number of blocks left).  The output is that of the lists
    without it, bit for bit; the next call's status is clean."""
    nbk, H = 41, 5
    N = nbk * block - 5
    g = torch.Generator().manual_seed(kmax)
    q, k, v = (torch.randn((1, H, N, 128), generator=g).to(torch.bfloat16).to(DEV) for _ in range(3))
    idx = torch.stack([torch.stack([torch.randperm(nbk, generator=g)[:kmax] for _ in range(nbk)]) for _ in range(H)]).to(torch.int32)
    cnt = torch.full((H, nbk), kmax - 1, dtype=torch.int32)
    bad, bad_cnt = idx.clone(), cnt.clone()
    for h, i, at, value in [(0, 0, 0, -1), (1, 7, kmax - 1, nbk), (2, 40, 1, 1 << 30), (4, 11, 2, -(1 << 31))]:
        bad[h, i] = torch.cat([idx[h, i, :at], torch.tensor([value], dtype=torch.int32), idx[h, i, at:kmax - 1]])
        bad_cnt[h, i] = kmax
    ws = sa.alloc_workspace(sa.make_shape(q, block), 1, kmax, DEV)
    out = sa.fwd(q, k, v, bad[None].to(DEV), bad_cnt[None].to(DEV), block, workspace=ws)
    assert sa.read_status(ws) == sa.E_BAD_INDEX
    ref = sa.fwd(q, k, v, idx[None].to(DEV), cnt[None].to(DEV), block, workspace=ws)
    assert sa.read_status(ws) == sa.OK
    assert torch.equal(out.view(torch.int16), ref.view(torch.int16))


@pytest.mark.parametrize("block,kmax", [(128, 5), (128, 33), (128, 128), (128, 129), (64, 9), (64, 70)])
def test_lists_cleaned_ahead_or_by_the_cta(block, kmax):
    """bf16, d = 128: up to 16 items per CTA the forward's CTAs clean their lists themselves, beyond (18 heads of 140 items) a
    pre-pass does.  Lists of every kind (own block first, in the middle, last, missing, twice; invalid indices; empty), strides
    on both sides of a warp and of what is held in registers: the same output, lse and status bit for bit, in a
    workspace of any content."""
    nbk, H = 140 * 128 // block, 18
    N = nbk * block - 5
    g = torch.Generator().manual_seed(block + kmax)
    q, k, v = (torch.randn((1, H, N, 128), generator=g).to(torch.bfloat16).to(DEV) for _ in range(3))
    idx = torch.randint(0, nbk, (1, H, nbk, kmax), generator=g, dtype=torch.int32)
    cnt = torch.randint(0, 7, (1, H, nbk), generator=g, dtype=torch.int32).clamp(max=kmax)
    at = torch.randint(0, 8, (1, H, nbk, 1), generator=g).clamp(max=kmax - 1)
    idx.scatter_(-1, at, torch.arange(nbk, dtype=torch.int32)[None, None, :, None].expand(1, H, nbk, 1).contiguous())
    cnt[0, :, 7], cnt[0, :, 11] = kmax, kmax                      # (a few full ones)
    bad = idx.clone()
    bad[0, ::3, 3, 0], bad[0, ::3, 7, kmax - 1], bad[0, ::3, 11, kmax // 2] = -1, nbk, 1 << 30
    cnt[0, ::3, 3] = cnt[0, ::3, 3].clamp(min=1)
    halves = (slice(0, 9), slice(9, 18))
    for lists, want in ((idx, sa.OK), (bad, sa.E_BAD_INDEX)):
        ws = sa.alloc_workspace(sa.make_shape(q, block), 1, kmax, DEV)
        ws.fill_(0xA5)
        out, lse = sa.fwd(q, k, v, lists.to(DEV), cnt.to(DEV), block, return_lse=True, workspace=ws)
        assert sa.read_status(ws) == want
        ws.fill_(0x5A)
        for h in halves:
            one, lse_one = sa.fwd(q[:, h], k[:, h], v[:, h], lists[:, h].contiguous().to(DEV), cnt[:, h].contiguous().to(DEV), block,
                                  return_lse=True, workspace=ws)
            assert sa.read_status(ws) == want
            assert torch.equal(out[:, h].view(torch.int16), one.view(torch.int16))
            assert torch.equal(lse[:, h].view(torch.int32), lse_one.view(torch.int32))


@pytest.mark.parametrize("form,block,kmax", [("window", 128, 9), ("window", 128, 129), ("window", 64, 9), ("window", 64, 70), ("padded", 128, 9),
                                             ("padded", 64, 9), ("gated", 128, 9), ("gated", 128, 129)])
def test_lists_cleaned_ahead_or_by_the_cta_in_every_form(form, block, kmax):
    """The same for the windowed, padded and gated forwards: 18 heads at once take the pre-pass, 9 and 9 clean their own
    lists (64-token blocks up to 64 entries in the variant with a closing warpgroup, beyond in the other).  Bad indices in some of
    the lists, then good lists in the workspace that a bad call has left and in memory that reads as a status code."""
    nbk, H = 140 * 128 // block, 18
    N, grid = nbk * block, (7, 40, 64)
    g = torch.Generator().manual_seed(block + kmax)
    q, k, v = (torch.randn((1, H, N, 128), generator=g).to(torch.bfloat16).to(DEV) for _ in range(3))
    idx = torch.randint(0, nbk, (1, H, nbk, kmax), generator=g, dtype=torch.int32)
    cnt = torch.randint(0, 7, (1, H, nbk), generator=g, dtype=torch.int32)
    cnt[0, :, 7] = kmax
    bad = idx.clone()
    bad[0, ::3, 7, kmax - 1] = nbk
    valid = torch.randint(1, block + 1, (nbk,), generator=g, dtype=torch.int32).to(DEV)
    if form == "gated":
        pq = (torch.randn((H, 64, 128), generator=g) / 128 ** 0.5).to(torch.bfloat16).to(DEV)
        state, gate = torch.randn((1, H, 64, 128), generator=g).to(DEV), torch.rand((1, H, N), generator=g).to(DEV)
        axis, freq = workloads.rope_schedule(128, 64)

    def run(lists, h, ws):
        args = [t[:, h] for t in (q, k, v)] + [t[:, h].contiguous().to(DEV) for t in (lists, cnt)]
        kw = dict(return_lse=True, workspace=ws)
        if form == "gated":
            return sa.fwd_gated(*args, pq[h].contiguous(), state[:, h].contiguous(), gate[:, h].contiguous(), grid, axis, freq, **kw)
        return sa.fwd(*args, block, **kw, **(dict(frame_tokens=450, window=20) if form == "window" else dict(block_valid=valid)))

    shape = sa.make_shape(q, block)
    size = sa.fwd_gated_workspace_bytes(shape, kmax, grid) if form == "gated" else sa.workspace_bytes(shape, 1, kmax)
    ws = torch.full((size,), 0xFF, dtype=torch.uint8, device=DEV)
    for lists, want in ((idx, sa.OK), (bad, sa.E_BAD_INDEX), (idx, sa.OK)):
        out, lse = run(lists, slice(0, H), torch.full_like(ws, 0xA5) if lists is bad else ws)
        for h in (slice(0, 9), slice(9, 18)):
            one, lse_one = run(lists, h, ws)
            assert sa.read_status(ws) == want
            assert torch.equal(out[:, h].view(torch.int16), one.view(torch.int16))
            assert torch.equal(lse[:, h].view(torch.int32), lse_one.view(torch.int32))


@pytest.mark.parametrize("H,window", [(3, 0), (7, 0), (3, 2)])
def test_d64_chains_of_every_length(H, window):
    """d = 64: the pairs of blocks of an item go to two chains (H = 3: 123 items, no SM gets a second one) or one (H = 7), so lists
    of 0 .. 9 blocks leave chains empty, level, a pair and half a pair apart; ragged last block, and rows whose tiles are all
    masked in some chains (causal window).  Scores large enough that references are raised on the way."""
    nbk, block, frame = 41, 64, 300
    N = nbk * block - 21
    g = torch.Generator().manual_seed(H + window)
    q, k, v = (torch.randn((1, H, N, 64), generator=g) for _ in range(3))
    q, k, v = (3.0 * q).to(torch.bfloat16), (k * (1.0 + torch.arange(N)[None, None, :, None] / N)).to(torch.bfloat16), v.to(torch.bfloat16)
    idx = torch.stack([torch.stack([torch.randperm(nbk, generator=g)[:9] for _ in range(nbk)]) for _ in range(H)]).to(torch.int32)
    cnt = (torch.arange(H * nbk) % 10).reshape(H, nbk).to(torch.int32)
    kw = dict(frame_tokens=frame, window=window) if window else {}
    out, lse = sa.fwd(q.to(DEV), k.to(DEV), v.to(DEV), idx[None].to(DEV), cnt[None].to(DEV), block, return_lse=True,
                      check_status=True, **kw)
    ref_out, ref_lse = oracle.attention(q[0], k[0], v[0], idx, cnt, block, **kw)
    got, ref = out[0].cpu().double(), ref_out.reshape(H, -1, 64)[:, :N]
    gl, rl = lse[0].cpu().double(), ref_lse.reshape(H, -1)[:, :N]
    empty = torch.isneginf(rl) | (cnt.repeat_interleave(block, 1)[:, :N] == 0)
    assert torch.equal(torch.isneginf(gl), empty) and torch.all(got[empty] == 0)
    relrms, maxabs = _errors(got[~empty], ref[~empty])
    assert relrms <= BF16_RELRMS and maxabs <= BF16_MAXABS and float((gl - rl)[~empty].abs().max()) <= LSE_ABS


@pytest.mark.parametrize("block,fp8", [(128, False), (128, True), (64, False)])
def test_long_permuted_lists_own_block_anywhere(block, fp8):
    """Kept lists of 70-100 entries in random order: cleaning them moves the query block's own
    key block to the front, wherever it stands (first, inside the first 32 entries, beyond them, at a
    multiple of 32, last, absent), and must keep every other entry exactly once.  Compared with the oracle,
    which walks the lists as given."""
    nbk = 100
    N = nbk * block - 17
    g = torch.Generator().manual_seed(7 + block + int(fp8))
    H, d, kmax = 2, 128, 100
    q, k, v = (torch.randn((1, H, N, d), generator=g).to(torch.bfloat16) for _ in range(3))
    idx = torch.stack([torch.stack([torch.randperm(nbk, generator=g) for _ in range(nbk)]) for _ in range(H)]).to(torch.int32)
    cnt = torch.randint(70, kmax + 1, (H, nbk), generator=g, dtype=torch.int32)
    for h in range(H):                      # the own block at chosen places of some lists
        for qb, pos in [(0, 0), (1, 5), (2, 31), (3, 32), (4, 33), (5, 64), (6, 69), (7, 96)]:
            row = idx[h, qb].tolist()
            row.remove(qb)
            row.insert(pos, qb)
            idx[h, qb] = torch.tensor(row, dtype=torch.int32)
        cnt[h, 7] = 97                      # own block last
        cnt[h, 8] = 70
        row = [j for j in idx[h, 8].tolist() if j != 8] + [8]
        idx[h, 8] = torch.tensor(row, dtype=torch.int32)    # own block beyond the count: absent
    qd, kd, vd = q.to(DEV), k.to(DEV), v.to(DEV)
    items = [(h, qb) for h in range(H) for qb in (0, 1, 2, 3, 4, 5, 6, 7, 8, 50, nbk - 1)]
    if fp8:
        cs = [sa.quant_fp8(t, block) for t in (qd, kd, vd)]
        out = sa.fwd(cs[0][0], cs[1][0], cs[2][0], idx[None].to(DEV), cnt[None].to(DEV), block,
                     scales=tuple(s for _, s in cs), check_status=True)
        ref, _ = oracle.attention(cs[0][0][0].cpu(), cs[1][0][0].cpu(), cs[2][0][0].cpu(), idx, cnt, block,
                                  scales=tuple(s[0].cpu() for _, s in cs), items=items)
    else:
        out = sa.fwd(qd, kd, vd, idx[None].to(DEV), cnt[None].to(DEV), block, check_status=True)
        ref, _ = oracle.attention(q[0], k[0], v[0], idx, cnt, block, items=items)
    num = den = 0.0
    for n, (h, qb) in enumerate(items):
        rows = slice(qb * block, min(N, (qb + 1) * block))
        got = out[0, h, rows].cpu().double()
        want = ref[n, : got.shape[0]]
        num += float(((got - want) ** 2).sum()); den += float((want ** 2).sum())
    assert (num / den) ** 0.5 <= (5e-2 if fp8 else 1e-2)


@pytest.mark.parametrize("block,window,fp8,stride", [(64, 0, False, 72), (64, 2, False, 72), (128, 0, True, 40), (128, 2, True, 40),
                                                     (64, 0, True, 72), (64, 2, True, 72), (128, 0, False, 40), (128, 2, False, 40)])
def test_both_kernels_agree_bitwise(block, window, fp8, stride):
    """d = 128: list strides of at most 64 (64-token blocks) or 32 (FP8, 128-token blocks) run the kernel with a closing warpgroup,
    longer ones the two-warpgroup kernel.  The same lists padded to a stride beyond that line (the counts say how
    many entries are real) must give the same output and lse bit for bit: both kernels take every step in the same
    arithmetic and order.  (bf16 with 128-token blocks has one kernel for every stride: there the padding alone must not
    matter.)  More items than SMs, counts 0 ... kmax, a ragged last block; with a causal window the same through the
    masked instantiations."""
    grid = (15, 18, 19)                                        # N = 5130: 41 blocks of 128 (last: 10 tokens) / 81 of 64
    w = _small(71 + block + window + int(fp8), 6, 128, grid, block, 0.0)
    q, k, v = workloads.structured_qkv(w)
    g = torch.Generator().manual_seed(500 + block + window)
    kmax = 9
    idx = torch.stack([torch.stack([torch.randperm(w.nb, generator=g)[:kmax] for _ in range(w.nb)]) for _ in range(w.H)]).to(torch.int32)
    cnt = torch.randint(0, kmax + 1, (w.H, w.nb), generator=g, dtype=torch.int32)
    cnt[0, 0] = 0; cnt[0, 1] = 1; cnt[0, 2] = 2; cnt[0, 3] = kmax
    wide = torch.full((w.H, w.nb, stride), -7, dtype=torch.int32)  # entries past the count are never read
    wide[:, :, :kmax] = idx
    qd, kd, vd = q.to(DEV), k.to(DEV), v.to(DEV)
    kw = dict(frame_tokens=18 * 19, window=window) if window else {}
    okw = dict(kw)
    if fp8:
        cs = [sa.quant_fp8(t, block) for t in (qd, kd, vd)]
        qd, kd, vd = (c for c, _ in cs)
        kw["scales"] = tuple(s for _, s in cs)
        okw["scales"] = tuple(s[0].cpu() for _, s in cs)
    a, la = sa.fwd(qd, kd, vd, idx[None].to(DEV), cnt[None].to(DEV), w.block, return_lse=True, check_status=True, **kw)
    b, lb = sa.fwd(qd, kd, vd, wide[None].to(DEV), cnt[None].to(DEV), w.block, return_lse=True, check_status=True, **kw)
    assert torch.equal(a.view(torch.int16), b.view(torch.int16))
    assert torch.equal(la.view(torch.int32), lb.view(torch.int32))
    items = [(h, i) for h in (0, w.H - 1) for i in list(range(0, w.nb, 5)) + [w.nb - 1] if cnt[h, i] > 0]
    oq, ok_, ov = (qd[0].cpu(), kd[0].cpu(), vd[0].cpu()) if fp8 else (q[0], k[0], v[0])
    ref_out, ref_lse = oracle.attention(oq, ok_, ov, idx, cnt, w.block, items=items, **okw)
    # (random lists under a causal window leave some rows without any admissible key: lse = -inf on both sides,
    # which test_gpu_window.py checks; here the output alone is compared with the oracle in that case)
    if fp8:
        _compare_items(b[0], None if window else lb[0], ref_out, ref_lse, items, w.block, w.N, FP8_RELRMS, None)
    else:
        _compare_items(b[0], None if window else lb[0], ref_out, ref_lse, items, w.block, w.N, BF16_RELRMS, BF16_MAXABS)


@pytest.mark.parametrize("block,fp8,window", [(128, True, 0), (64, True, 0), (64, True, 3), (128, True, 3), (128, False, 0), (64, False, 3)])
def test_tile_descriptors_around_their_ring(block, fp8, window):
    """The K producer hands the softmax warps a descriptor per tile through a ring of eight: items of 7, 8, 9, 15, 16 and 17
    tiles, eight or more of them per CTA, so that every item starts somewhere else in the ring; K and V blocks of
    different magnitude, so that a descriptor of another tile gives another result.  The same lists with a stride beyond the
    line of the kernel with a closing warpgroup run the two-warpgroup kernel, whose softmax warps also close the items and so
    follow the producer at another distance: the same bits."""
    grid = (15, 18, 19)                                        # N = 5130: 41 blocks of 128 (last: 10 tokens) / 81 of 64
    w = _small(91 + block + window + int(fp8), 30, 128, grid, block, 0.0)
    q, k, v = workloads.structured_qkv(w)
    g = torch.Generator().manual_seed(700 + block + window)
    size = lambda: (2.0 ** torch.randint(-1, 2, (w.H, w.nb), generator=g)).repeat_interleave(block, 1)[None, :, : w.N, None]
    k, v = (k * size()).to(torch.bfloat16), (v * size()).to(torch.bfloat16)
    per = 128 // block
    kmax = 17 * per
    own = torch.arange(w.nb)[None, :, None].expand(w.H, w.nb, 1)
    idx = torch.stack([torch.stack([torch.randperm(w.nb, generator=g)[:kmax] for _ in range(w.nb)]) for _ in range(w.H)])
    idx = torch.where((idx == own).any(-1, keepdim=True), idx, torch.cat([own, idx[..., 1:]], -1)).to(torch.int32)
    cnt = (torch.tensor([7, 8, 9, 15, 16, 17])[torch.randint(0, 6, (w.H, w.nb), generator=g)] * per).to(torch.int32)
    idx[..., 0], keep = idx.gather(-1, (idx == own).int().argmax(-1, keepdim=True))[..., 0], idx[..., 0].clone()
    at = (idx[..., 1:] == own).int()                           # the own block comes first, what stood there takes its place
    idx[..., 1:] = torch.where(at.bool(), keep[..., None], idx[..., 1:])
    qd, kd, vd = q.to(DEV), k.to(DEV), v.to(DEV)
    kw = dict(frame_tokens=18 * 19, window=window) if window else {}
    okw = dict(kw)
    if fp8:
        cs = [sa.quant_fp8(t, block) for t in (qd, kd, vd)]
        qd, kd, vd = (c for c, _ in cs)
        kw["scales"] = tuple(s for _, s in cs)
        okw["scales"] = tuple(s[0].cpu() for _, s in cs)
    out = sa.fwd(qd, kd, vd, idx[None].to(DEV), cnt[None].to(DEV), block, check_status=True, **kw)
    wide = torch.full((w.H, w.nb, 72 if block == 64 else 40), -7, dtype=torch.int32)      # entries past the count are never read
    wide[:, :, :kmax] = idx
    again = sa.fwd(qd, kd, vd, wide[None].to(DEV), cnt[None].to(DEV), block, check_status=True, **kw)
    assert torch.equal(out.view(torch.int16), again.view(torch.int16))
    items = [(h, i) for h in (0, w.H // 2, w.H - 1) for i in list(range(0, w.nb, 7)) + [w.nb - 1]]
    ref, _ = oracle.attention(qd[0].cpu(), kd[0].cpu(), vd[0].cpu(), idx, cnt, block, items=items, **okw)
    _compare_items(out[0], None, ref, None, items, block, w.N, FP8_RELRMS if fp8 else BF16_RELRMS, None)


@pytest.mark.parametrize("fp8,window", [(False, 0), (True, 0), (False, 4), (True, 4)])
@pytest.mark.parametrize("shared", [0, 1, 5])
def test_pairs_whose_lists_differ(shared, fp8, window):
    """64-token blocks: the two query blocks of a pair share 0, 1 or all 5 of their blocks, so that tiles hold two blocks of
    one, of the other, one of each and (an odd number in all) a half that is nobody's; the last pair is a single
    query block with a ragged tail.  A half tile that a query block does not list adds nothing to its rows, whatever stands in it:
    the blocks that only the other one lists hold keys with far larger scores."""
    H, nbk, block = 3, 33, 64
    N = nbk * block - 23
    g = torch.Generator().manual_seed(77 + shared + window)
    q, k, v = (torch.randn((1, H, N, 128), generator=g) for _ in range(3))
    idx = torch.empty((H, nbk, 5), dtype=torch.int32)
    for h in range(H):
        for i in range(0, nbk, 2):
            rest = [j for j in torch.randperm(nbk, generator=g).tolist() if j not in (i, i + 1)]
            both = ([i] + rest[:shared - 1]) if shared else []
            idx[h, i] = torch.tensor((both + [j for j in ([i] + rest[8:16]) if j not in both])[:5])
            if i + 1 < nbk:
                idx[h, i + 1] = torch.tensor((both + [j for j in ([i + 1] + rest[16:24]) if j not in both])[:5])
    cnt = torch.full((H, nbk), 5, dtype=torch.int32)
    cnt[:, 3::4] = 4                                            # an odd number of blocks in the pair's merged list
    k = k * (1.0 + 3.0 * (torch.arange(N) // block % 2))[None, None, :, None]      # odd blocks: larger scores
    q, k, v = (t.to(torch.bfloat16) for t in (q, k, v))
    t, kw = (q.to(DEV), k.to(DEV), v.to(DEV)), dict(frame_tokens=150, window=window) if window else {}
    okw = dict(kw)
    if fp8:
        t, sc = zip(*(sa.quant_fp8(x, block) for x in t))
        kw["scales"], okw["scales"] = sc, tuple(x[0].cpu() for x in sc)
    out = sa.fwd(*t, idx[None].to(DEV), cnt[None].to(DEV), block, check_status=True, **kw)
    items = [(h, i) for h in range(H) for i in range(nbk)]
    ref, _ = oracle.attention(*(x[0].cpu() for x in t), idx, cnt, block, items=items, **okw)
    _compare_items(out[0], None, ref, None, items, block, N, FP8_RELRMS if fp8 else BF16_RELRMS, None)


def _stream_of_short_items(streams, block, stride, H=16, N=74 * 128 - 17):
    """Kept lists whose item i has streams[i % SMs % len][i // SMs % 8] tiles: what the persistent kernel's CTA c works
    through (items c, c + SMs, ...).  Both query blocks of a 64-token pair keep the same blocks."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nb, per = -(-N // block), 128 // block
    nbq = -(-nb // per)
    g = torch.Generator().manual_seed(block + stride + len(streams))
    idx = torch.full((H, nb, stride), -7, dtype=torch.int32)          # entries past the count are never read
    cnt = torch.zeros((H, nb), dtype=torch.int32)
    for h in range(H):
        for i in range(nb):
            item = h * nbq + i // per
            if i % per == 0:
                n = streams[item % sms % len(streams)][item // sms % 8] * per
                keep = torch.randperm(nb, generator=g)[:n].to(torch.int32)
            cnt[h, i] = n
            idx[h, i, :n] = keep
    q, k, v = (torch.randn((1, H, N, 128), generator=g).to(torch.bfloat16).to(DEV) for _ in range(3))
    return q, k, v, idx[None].to(DEV), cnt[None].to(DEV), sms // nbq


STREAM_CASES = [(128, 6, "bf16"), (64, 6, "bf16"), (64, 72, "bf16"), (128, 6, "fp8"), (128, 40, "fp8"), (64, 6, "fp8"),
                (64, 72, "fp8"), (128, 6, "gated")]


def _check_stream(streams, block, stride, kind):
    """All items in one call, against the same items a few heads at a time, no CTA with more than one: bit for bit (an item's
    arithmetic does not depend on what its CTA did before), and those against fp32 attention over the lists."""
    q, k, v, idx, cnt, heads = _stream_of_short_items(streams, block, stride)
    H, N = q.shape[1], q.shape[2]
    if kind == "fp8":
        (q, sq), (k, sk), (v, sv) = (sa.quant_fp8(t, block) for t in (q, k, v))
    if kind == "gated":
        w = workloads.Workload("gatedstream", 83, 1, H, 128, (1, 1, N), 128, 0.0)
        pq, pk, gate = workloads.compensation_params(w, 64, device=DEV)
        axis, freq = workloads.rope_schedule(128, 64)
        state = sa.comp_state(k, v, pk, w.grid, axis, freq)

    def run(h):
        args = [t[:, h] for t in (q, k, v)] + [t[:, h].contiguous() for t in (idx, cnt)]
        if kind == "gated":
            return sa.fwd_gated(*args, pq[h], state[:, h].contiguous(), gate[:, h].contiguous(), (1, 1, N), axis, freq,
                                return_lse=True, check_status=True)
        kw = dict(scales=tuple(s[:, h].contiguous() for s in (sq, sk, sv))) if kind == "fp8" else {}
        return sa.fwd(*args, block, return_lse=True, check_status=True, **kw)

    out, lse = run(slice(0, H))
    for h0 in range(0, H, heads):
        h = slice(h0, min(H, h0 + heads))
        one, lse_one = run(h)
        assert torch.equal(out[:, h].view(torch.int16), one.view(torch.int16))
        assert torch.equal(lse[:, h].view(torch.int32), lse_one.view(torch.int32))
    if kind != "bf16":
        return
    nb = idx.shape[2]
    for h in (0, H // 2, H - 1):
        keep = torch.zeros((nb, nb + 8), dtype=torch.bool, device=DEV)
        keep.scatter_(1, torch.where(torch.arange(stride, device=DEV) < cnt[0, h][:, None], idx[0, h], nb).long(), True)
        keep = keep[:, :nb].repeat_interleave(block, 0).repeat_interleave(block, 1)[:N, :N]
        s = (q[0, h].float() @ k[0, h].float().T / math.sqrt(128)).masked_fill(~keep, -math.inf)
        ref, empty = torch.softmax(s, -1).nan_to_num(0.0) @ v[0, h].float(), ~keep.any(1)
        assert torch.all(out[0, h][empty] == 0) and torch.all(torch.isneginf(lse[0, h][empty]))
        if not bool(empty.all()):
            assert _errors(out[0, h].cpu(), ref.cpu())[0] <= BF16_RELRMS


@pytest.mark.parametrize("block,stride,kind", STREAM_CASES)
def test_streams_of_short_items(block, stride, kind):
    """Every item one tile, or one and two or three in turn: the warpgroups swap the roles of the item's last tile at each
    item and run as far ahead of the closing warpgroup as they can."""
    _check_stream([[1] * 8, [2, 1] * 4, [1, 2] * 4, [3, 1, 1, 1, 2, 1, 1, 1], [1, 3] * 4], block, stride, kind)


@pytest.mark.parametrize("block", [64, 128])
def test_fp8_streams_past_the_closing_warpgroup(block):
    """FP8 lists with a stride beyond 64 run the two-warpgroup kernel for both block sizes."""
    _check_stream([[1] * 8, [2, 1] * 4, [3, 1, 0, 1, 2, 1, 0, 1]], block, 72, "fp8")


STREAMS = [[1, 0, 0, 0, 1, 0, 0, 2], [2, 0, 0, 1, 0, 0, 0, 1], [0, 0, 1, 0, 0, 0, 1, 1], [1, 0, 1, 0, 1, 0, 0, 0],
           [0, 1, 0, 0, 1, 1, 0, 3], [0, 0, 0, 0, 0, 0, 0, 0]]     # tiles of the items that one CTA takes in turn


@pytest.mark.parametrize("block,stride,kind", STREAM_CASES)
def test_empty_lists_between_short_ones(block, stride, kind):
    """Items with an empty list between items of one to three tiles, so that the roles of a CTA are several items apart:
    an empty item must neither release nor take a Q slot that another item still uses."""
    _check_stream(STREAMS, block, stride, kind)


@pytest.mark.parametrize("H", [2, 5])
def test_d64_infinity_stays_where_it_belongs(H):
    """d = 64: the halves of a product take two key blocks at a time, and what one half makes of the other's block is computed
    but never read.  An infinite value in one key block (lists of one to six blocks, odd ones with half a pair left over)
    makes its channel infinite for the query blocks that keep it and leaves everything else as it is: no NaN.  82
    items run two chains each, 205 one."""
    nb, d = 41, 64
    N = nb * 64 - 7
    g = torch.Generator().manual_seed(900 + H)
    q, k, v = (0.3 * torch.randn((1, H, N, d), generator=g) for _ in range(3))
    idx = torch.stack([torch.stack([torch.randperm(nb, generator=g)[:6] for _ in range(nb)]) for _ in range(H)]).to(torch.int32)
    cnt = (1 + torch.arange(nb, dtype=torch.int32) % 6).expand(H, nb).contiguous()
    kept = (idx == 3) & (torch.arange(6) < cnt[..., None])
    assert 0 < int(kept.any(-1).sum()) < H * nb
    q, k, v = (t.to(torch.bfloat16).to(DEV) for t in (q, k, v))
    clean = sa.fwd(q, k, v, idx[None].to(DEV), cnt[None].to(DEV), 64, check_status=True)
    v[:, :, 3 * 64 + 11, 5] = math.inf
    out = sa.fwd(q, k, v, idx[None].to(DEV), cnt[None].to(DEV), 64, check_status=True)
    rows = kept.any(-1).to(DEV).repeat_interleave(64, 1)[:, :N]             # [H, N]
    assert torch.all(torch.isposinf(out[0, ..., 5]) == rows)
    clean[0, ..., 5] = torch.where(rows, math.inf, clean[0, ..., 5])
    assert torch.equal(out, clean)


@pytest.mark.parametrize("H", [2, 5])
def test_d64_status_in_a_workspace_of_any_content(H):
    """d = 64: up to one item per SM (82 items) the forward clears its status itself, beyond (205) a kernel in front does.
    Either way a call reports its own bad index and nothing that was in the workspace before."""
    nb = 41
    q = torch.randn((1, H, nb * 64, 64), generator=torch.Generator().manual_seed(H)).to(torch.bfloat16).to(DEV)
    idx = torch.arange(nb, dtype=torch.int32, device=DEV)[None, None, :, None].expand(1, H, nb, 3).contiguous()
    bad = idx.clone()
    bad[0, H - 1, nb - 1, 1] = nb
    for fill in (0x00, 0xA5, 0xFF):
        ws = sa.alloc_workspace(sa.make_shape(q, 64), 1, 3, DEV)
        ws.fill_(fill)
        for lists, want in ((idx, sa.OK), (bad, sa.E_BAD_INDEX), (bad, sa.E_BAD_INDEX), (idx, sa.OK)):
            sa.fwd(q, q, q, lists, None, 64, workspace=ws)
            assert sa.read_status(ws) == want


@pytest.mark.parametrize("H", [28, 56])
def test_lse_of_merged_chains_is_rounded_once(H):
    """d = 64: scores that fp32 holds exactly and one key that outweighs the others, so that the log-sum-exp is off by its
    own rounding (at most 2^-24 of it) and by what ln 2 and log2 e lose as fp32 constants (1.1e-8 together).  112 items
    run two chains each, 224 one."""
    N, nb = 256, 4
    a = 128 + torch.arange(N) % 128
    b = (200 + torch.arange(H))[:, None] - 16 * torch.ones((H, N), dtype=torch.int64)
    b[torch.arange(H), 37 * torch.arange(H) % N] += 16
    q, k = torch.zeros((1, H, N, 64)), torch.zeros((1, H, N, 64))
    q[0, :, :, 0], k[0, :, :, 0] = a, b                                    # integers below 256: exact in bf16
    idx = torch.arange(nb, dtype=torch.int32).expand(1, H, nb, nb).contiguous()
    q, k = (t.to(torch.bfloat16).to(DEV) for t in (q, k))
    _, lse = sa.fwd(q, k, k, idx.to(DEV), None, 64, return_lse=True, check_status=True)
    ref = torch.logsumexp(a.double()[None, :, None] * b.double()[:, None] / 8, -1)
    assert float(((lse[0].cpu().double() - ref) / ref).abs().max()) <= 2.0 ** -24 + 1.2e-8
