"""GPU parity: sparkattn_select and sparkattn_quant_fp8 against the CPU oracle, bit for bit."""
import threading

import pytest
import torch

import oracle
import paper_2609_23153_b200 as sa
import workloads

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _small_cases():
    return [
        workloads.small_structured(H=3, d=128, grid=(5, 12, 20), block=128, sparsity=0.8, cfg_id=11),   # N=1200: 9 full + tail 48
        workloads.small_structured(H=2, d=128, grid=(3, 16, 16), block=128, sparsity=0.5, cfg_id=12),   # N=768: no tail
        workloads.small_structured(H=2, d=64, grid=(3, 10, 21), block=64, sparsity=0.9, cfg_id=13),     # N=630: tail 54
        workloads.small_structured(H=1, d=64, grid=(1, 1, 37), block=64, sparsity=0.0, cfg_id=14),      # one ragged block
        workloads.small_structured(H=2, d=128, grid=(1, 1, 1), block=128, sparsity=0.0, cfg_id=15),     # N=1
        workloads.small_structured(H=2, d=128, grid=(4, 9, 25), block=64, sparsity=0.9, cfg_id=17),     # d=128, 64-token blocks, tail 4
    ]


@pytest.mark.parametrize("w", _small_cases(), ids=lambda w: f"{w.name}-N{w.N}-d{w.d}")
def test_select_matches_oracle(w):
    q, k, _ = workloads.structured_qkv(w)
    for topk in sorted({1, w.topk, w.nb}):
        ref_idx, ref_cnt = oracle.select(q[0], k[0], w.block, topk)
        idx, cnt = sa.select(q.to(DEV), k.to(DEV), w.block, topk)
        torch.cuda.synchronize()
        assert torch.equal(idx[0].cpu(), ref_idx)
        assert torch.equal(cnt[0].cpu(), ref_cnt)


def test_select_tiny_workload_and_ties():
    w = workloads.TINY
    q, k, _ = workloads.tiny_inputs(w)
    ref_idx, _ = oracle.select(q[0], k[0], w.block, 16)
    idx, _ = sa.select(q.to(DEV), k.to(DEV), w.block, 16)
    assert torch.equal(idx[0].cpu(), ref_idx)
    # exact ties: every key block identical -> lowest indices win
    kc = k.clone(); kc[:] = k[0, 0, 5]
    ref_idx, _ = oracle.select(q[0], kc[0], w.block, 7)
    idx, _ = sa.select(q.to(DEV), kc.to(DEV), w.block, 7)
    assert torch.equal(idx[0].cpu(), ref_idx)
    assert ref_idx[0, 0].tolist() == list(range(7))
    # zero queries: all scores +0/-0 -> still the lowest indices
    ref_idx, _ = oracle.select(torch.zeros_like(q[0]), -k[0], w.block, 5)
    idx, _ = sa.select(torch.zeros_like(q).to(DEV), (-k).to(DEV), w.block, 5)
    assert torch.equal(idx[0].cpu(), ref_idx)


def _crafted_qk(nb, block, d, pattern, tail=0):
    """Q/K whose pooled block scores are known exactly: channel 0 of key block j holds v_j on all its tokens,
    channel 0 of query block i holds a_i, every other channel is 0, so score(i, j) = a_i * v_j without rounding."""
    N = nb * block - tail
    j = torch.arange(nb)
    if pattern == "one_lane":          # the largest keys all sit in one lane (j % 32 == 5) of the selecting warp
        v = torch.where(j % 32 == 5, 64.0 + (j // 32).float(), ((j * 37) % 97).float() / 128.0)
    elif pattern == "ties":            # two values only: most of the kept keys are ties at the threshold
        v = (j % 3 == 0).float()
    elif pattern == "few_then_ties":   # three clear winners, then a long run of equal keys
        v = torch.where(j % 101 == 7, 5.0 + (j // 101).float(), torch.where((j % 4) != 1, 2.0, 0.25))
    else:
        raise ValueError(pattern)
    a = torch.tensor([1.0, -1.0, 0.5, -0.75, 2.0])[torch.arange(nb) % 5]      # sign flips reverse the order
    q = torch.zeros((1, 2, N, d), dtype=torch.bfloat16)
    k = torch.zeros((1, 2, N, d), dtype=torch.bfloat16)
    tok_blk = torch.arange(N) // block
    q[0, :, :, 0] = a[tok_blk].to(torch.bfloat16)
    k[0, 0, :, 0] = v[tok_blk].to(torch.bfloat16)
    k[0, 1, :, 0] = v.flip(0)[tok_blk].to(torch.bfloat16)
    return q, k


@pytest.mark.parametrize("nb,topk", [(100, 7), (300, 8), (300, 40), (1000, 30), (1000, 140), (1400, 12)])
@pytest.mark.parametrize("pattern", ["one_lane", "ties", "few_then_ties"])
def test_select_crafted_scores(nb, topk, pattern):
    """Score layouts aimed at the branches of the selection: many of the largest keys in one lane of the warp
    (the search over per-lane maxima must give way to the full search), long runs of ties at the threshold,
    every register-resident key count (nb <= 256, 640, 1280) and the shared-memory path above."""
    block, d = 64, 128
    q, k = _crafted_qk(nb, block, d, pattern, tail=13)
    ref_idx, ref_cnt = oracle.select(q[0], k[0], block, topk)
    idx, cnt = sa.select(q.to(DEV), k.to(DEV), block, topk)
    assert torch.equal(idx[0].cpu(), ref_idx)
    assert torch.equal(cnt[0].cpu(), ref_cnt)


@pytest.mark.parametrize("pattern", ["one_lane", "ties"])
def test_select_crafted_scores_with_window(pattern):
    nb, block, d, topk = 300, 64, 128, 9
    q, k = _crafted_qk(nb, block, d, pattern, tail=13)
    F, window = 1000, 6                       # frames of 1000 tokens straddle the 64-token blocks
    ref_idx, ref_cnt = oracle.select(q[0], k[0], block, topk, frame_tokens=F, window=window)
    idx, cnt = sa.select(q.to(DEV), k.to(DEV), block, topk, frame_tokens=F, window=window)
    assert torch.equal(idx[0].cpu(), ref_idx)
    assert torch.equal(cnt[0].cpu(), ref_cnt)


# (heads, key blocks, missing tokens of the last block, block, d): one side and the other of every line of the dispatch
# (256 key blocks; CTAs of 8, 16 and 32 rows; 16 and 8 rows of the wide kernel at 1680 blocks of d = 128, 1744 of d = 64)
# and of the key registers (640, 1280), with remainders of the row tiles and of the last block
@pytest.mark.parametrize("H,nb,tail,block,d", [(1, 1, 63, 64, 64), (1, 9, 1, 64, 64), (10, 241, 5, 64, 64), (30, 250, 63, 64, 64),
                                               (3, 256, 0, 64, 128), (2, 257, 17, 64, 64), (1, 640, 1, 64, 64), (1, 641, 0, 64, 64),
                                               (1, 1281, 30, 64, 64), (1, 1680, 3, 64, 128), (1, 1745, 9, 64, 64)])
def test_select_kernel_variants_match_oracle(H, nb, tail, block, d):
    g = torch.Generator().manual_seed(nb)
    N = nb * block - tail
    q, k = (torch.randn((1, H, N, d), generator=g).to(torch.bfloat16) for _ in range(2))
    qd, kd = q.to(DEV), k.to(DEV)
    for topk in sorted({t for t in (1, 32, 33, 128, 129, nb - 1, nb) if 1 <= t <= nb}):
        ref_idx, ref_cnt = oracle.select(q[0], k[0], block, topk)
        idx, cnt = sa.select(qd, kd, block, topk)
        assert torch.equal(idx[0].cpu(), ref_idx) and torch.equal(cnt[0].cpu(), ref_cnt), topk
    # the two launches under capture: same lists from a replay
    ws = sa.alloc_workspace(sa.make_shape(qd, block), 0, topk, DEV)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sa.select(qd, kd, block, topk, kept_idx=idx, kept_cnt=cnt, workspace=ws)
    idx.zero_(), cnt.zero_()
    graph.replay()
    assert torch.equal(idx[0].cpu(), ref_idx) and torch.equal(cnt[0].cpu(), ref_cnt)
    assert sa.read_status(ws) == sa.OK


@pytest.mark.parametrize("nb", [2, 7, 8, 9, 31, 32, 33, 63, 64, 65])
@pytest.mark.parametrize("d,block,window", [(64, 64, 0), (128, 64, 0), (128, 64, 2), (64, 64, 3)])
def test_select_few_blocks(nb, d, block, window):
    """Up to 64 key blocks have a kernel of their own: 8 query blocks per CTA, one or two key blocks per lane.  Both sides of those
    lines against the oracle, with key blocks that repeat (ties to the lowest index) and under a causal window."""
    g = torch.Generator().manual_seed(nb * d + window)
    N = nb * block - 3
    q, k = (torch.randn((2, 3, N, d), generator=g).to(torch.bfloat16) for _ in range(2))
    if nb > 7:
        k[1, :, 5 * block: 6 * block], k[1, :, (nb - 2) * block: (nb - 1) * block] = k[1, :, :block], k[1, :, :block]
    kw = dict(frame_tokens=100, window=window) if window else {}
    for topk in sorted({1, nb // 2, nb - 1}):
        idx, cnt = sa.select(q.to(DEV), k.to(DEV), block, topk, **kw)
        for b in range(2):
            want, count = oracle.select(q[b], k[b], block, topk, **kw)
            assert torch.equal(idx[b].cpu(), want) and torch.equal(cnt[b].cpu(), count), topk


def test_select_strided_layout_and_batch():
    # [B, N, H, d] storage viewed as [B, H, N, d]; two batches
    w = workloads.small_structured(H=2, d=128, grid=(2, 10, 26), block=128, sparsity=0.75, cfg_id=16)
    qs, ks = [], []
    for b in range(2):
        q, k, _ = workloads.structured_qkv(workloads.small_structured(2, 128, (2, 10, 26), 128, 0.75, cfg_id=16 + b))
        qs.append(q[0]); ks.append(k[0])
    q = torch.stack(qs); k = torch.stack(ks)
    qd = q.permute(0, 2, 1, 3).contiguous().to(DEV).permute(0, 2, 1, 3)
    kd = k.permute(0, 2, 1, 3).contiguous().to(DEV).permute(0, 2, 1, 3)
    idx, cnt = sa.select(qd, kd, w.block, w.topk)
    for b in range(2):
        ref_idx, _ = oracle.select(q[b], k[b], w.block, w.topk)
        assert torch.equal(idx[b].cpu(), ref_idx)


@pytest.mark.parametrize("w", _small_cases(), ids=lambda w: f"{w.name}-N{w.N}-d{w.d}")
def test_quant_matches_oracle(w):
    q, _, v = workloads.structured_qkv(w)
    for x in (q, v):
        ref_codes, ref_scales = oracle.quant_fp8(x[0], w.block)
        codes, scales = sa.quant_fp8(x.to(DEV), w.block)
        torch.cuda.synchronize()
        assert torch.equal(scales[0].cpu().view(torch.int32), ref_scales.view(torch.int32))
        assert torch.equal(codes[0].cpu(), ref_codes)


def test_quant_edge_values():
    H, N, d, block = 2, 300, 128, 128
    g = torch.Generator().manual_seed(21)
    x = (torch.randn((1, H, N, d), generator=g) * 4).to(torch.bfloat16)
    x[0, 0, :128] = 0                       # all-zero block
    x[0, 1, 130, 7] = -1000.0               # one huge negative element: the rest underflows towards zero
    x[0, 1, 131, 9] = 3.0e-3
    x[0, 0, 256:] *= 1e-20                  # tiny magnitudes in the tail block
    ref_codes, ref_scales = oracle.quant_fp8(x[0], block)
    # canary: rows past N of a padded buffer must stay untouched
    buf = torch.full((1, H, N + 20, d), 0xAB, dtype=torch.uint8, device=DEV)
    xd = torch.zeros((1, H, N + 20, d), dtype=torch.bfloat16, device=DEV)
    xd[:, :, :N] = x.to(DEV)
    codes, scales = sa.quant_fp8(xd[:, :, :N], block, codes=buf[:, :, :N])
    torch.cuda.synchronize()
    assert torch.equal(codes[0].cpu(), ref_codes)
    assert torch.equal(scales[0].cpu().view(torch.int32), ref_scales.view(torch.int32))
    assert torch.all(buf[:, :, N:] == 0xAB)


def test_select_and_quant_are_deterministic():
    w = workloads.small_structured(H=4, d=128, grid=(4, 12, 20), block=128, sparsity=0.8, cfg_id=19)
    q, k, v = (t.to(DEV) for t in workloads.structured_qkv(w))
    a = sa.select(q, k, w.block, w.topk)[0].clone()
    b = sa.select(q, k, w.block, w.topk)[0].clone()
    assert torch.equal(a, b)
    c1 = sa.quant_fp8(v, w.block)[0].clone()
    c2 = sa.quant_fp8(v, w.block)[0].clone()
    assert torch.equal(c1, c2)


@pytest.mark.parametrize("w", _small_cases(), ids=lambda w: f"{w.name}-N{w.N}-d{w.d}")
def test_per_token_quant_matches_oracle(w):
    q, _, v = workloads.structured_qkv(w)
    v = v * torch.logspace(-2, 1, w.N)[None, None, :, None].to(torch.bfloat16)   # widely varying row magnitudes
    v[0, 0, w.N // 2] = 0
    for x in (q, v):
        ref_codes, ref_scales = oracle.quant_fp8_per_token(x[0])
        codes, scales = sa.quant_fp8_per_token(x.to(DEV))
        torch.cuda.synchronize()
        assert torch.equal(scales[0].cpu().view(torch.int32), ref_scales.view(torch.int32))
        assert torch.equal(codes[0].cpu(), ref_codes)


def test_per_token_quant_strided_and_fullsize_sample():
    w = workloads.WAN_1P3B_480P
    q, _, _ = workloads.structured_qkv(w, device=DEV)
    qs = q.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)          # [B,N,H,d] storage
    codes, scales = sa.quant_fp8_per_token(qs)
    assert codes.stride() == qs.stride()
    for h in (0, 11):
        rc, rs = oracle.quant_fp8_per_token(q[0, h:h + 1].cpu())
        assert torch.equal(codes[0, h:h + 1].cpu(), rc) and torch.equal(scales[0, h:h + 1].cpu().view(torch.int32), rs.view(torch.int32))


def _pooled_from_workspace(ws, H, nb, d):
    """Pooled Q [H, nb, d] and pooled K [H, nb, d] out of a selection workspace (B = 1): pooled Q sits right
    behind the 256-byte header, pooled K transposed [H, d, nbp] (nbp = nb rounded up to 32) behind it."""
    nbp = (nb + 31) // 32 * 32
    f = ws[256:].view(torch.float32).cpu()
    pq = f[: H * nb * d].reshape(H, nb, d)
    pk = f[H * nb * d: H * nb * d + H * d * nbp].reshape(H, d, nbp)[:, :, :nb].transpose(1, 2).contiguous()
    return pq, pk


@pytest.mark.parametrize("w", _small_cases(), ids=lambda w: f"{w.name}-N{w.N}-d{w.d}")
def test_quant_with_pooling_and_select_from_pooled_match_oracle(w):
    """One pass over Q and one over K give codes, scales AND the selection's pooled means (same order of
    additions as the selection's own pooling: bit-exact against oracle.pool); scores + top-k on those means
    give the oracle's lists."""
    q, k, _ = workloads.structured_qkv(w)
    qd, kd = q.to(DEV), k.to(DEV)
    ws = sa.alloc_workspace(sa.make_shape(qd, w.block), 0, w.topk, DEV)
    ws.fill_(0x5A)                                           # stale contents must not matter
    cq, sq = sa.quant_fp8_pooled(qd, w.block, False, ws)
    ck, sk = sa.quant_fp8_pooled(kd, w.block, True, ws)
    for (codes, scales), x in (((cq, sq), q), ((ck, sk), k)):
        rc, rs = oracle.quant_fp8(x[0], w.block)
        assert torch.equal(codes[0].cpu(), rc)
        assert torch.equal(scales[0].cpu().view(torch.int32), rs.view(torch.int32))
    torch.cuda.synchronize()
    pq, pk = _pooled_from_workspace(ws, w.H, w.nb, w.d)
    assert torch.equal(pq.view(torch.int32), oracle.pool(q[0], w.block).view(torch.int32))
    assert torch.equal(pk.view(torch.int32), oracle.pool(k[0], w.block).view(torch.int32))
    for topk in sorted({1, w.topk, w.nb}):
        idx, cnt = sa.select_pooled(qd, w.block, topk, ws)
        ref_idx, ref_cnt = oracle.select(q[0], k[0], w.block, topk)
        assert sa.read_status(ws) == sa.OK
        assert torch.equal(idx[0].cpu(), ref_idx) and torch.equal(cnt[0].cpu(), ref_cnt)


@pytest.mark.parametrize("d,block", [(128, 128), (128, 64), (64, 64)])
@pytest.mark.parametrize("tail", [0, 1, 15, 16, 17])
def test_quant_with_pooling_at_every_tail(d, block, tail):
    """The last block holds a batch of the addition chain's 16 rows, one less, one more, one row or all of them: codes, scales and
    means against the oracle, bit for bit, with more CTAs than fit the chip at once."""
    H, nb = 40, 33
    N = (nb - 1) * block + (tail or block)
    x = torch.randn((1, H, N, d), generator=torch.Generator().manual_seed(d + block + tail)).to(torch.bfloat16)
    xd = x.to(DEV)
    ws = sa.alloc_workspace(sa.make_shape(xd, block), 0, 1, DEV)
    for key_side in (False, True):
        codes, scales = sa.quant_fp8_pooled(xd, block, key_side, ws)
        rc, rs = oracle.quant_fp8(x[0], block)
        assert torch.equal(codes[0].cpu(), rc) and torch.equal(scales[0].cpu().view(torch.int32), rs.view(torch.int32))
    want = oracle.pool(x[0], block).view(torch.int32)
    for pooled in _pooled_from_workspace(ws, H, nb, d):
        assert torch.equal(pooled.view(torch.int32), want)


@pytest.mark.parametrize("nb,H", [(65, 2), (65, 30), (65, 74), (250, 2), (250, 10), (250, 28), (257, 1), (257, 9)])
@pytest.mark.parametrize("d", [64, 128])
def test_select_from_pooled_clears_the_status(nb, H, d):
    """Scores + top-k on pooled means clear the status themselves.  More than 64 key blocks: 8, 16 and 32 query blocks per CTA
    (2, 30 or 10, 74 or 28 heads), beyond 256 blocks 8 and 16 (1 and 9 heads); in a workspace of any content, twice in the
    same one, and with the lists of the selection that pools for itself."""
    q, k = (torch.randn((1, H, nb * 64 - 3, d), generator=torch.Generator().manual_seed(nb + H + i)).to(torch.bfloat16).to(DEV) for i in (0, 1))
    topk = nb // 3
    want, count = sa.select(q, k, 64, topk)
    ws = sa.alloc_workspace(sa.make_shape(q, 64), 0, topk, DEV)
    for fill in (0xA5, 0xFF):
        ws.fill_(fill)
        sa.quant_fp8_pooled(q, 64, False, ws), sa.quant_fp8_pooled(k, 64, True, ws)
        for _ in range(2):
            idx, cnt = sa.select_pooled(q, 64, topk, ws)
            assert sa.read_status(ws) == sa.OK
            assert torch.equal(idx, want) and torch.equal(cnt, count)
            ws[:256] = fill


def test_quant_with_pooling_strided_batch_equals_separate_calls():
    """[B, N, H, d] buffers viewed as [B, H, N, d], two batch entries: the fused pass must reproduce the separate
    sparkattn_quant_fp8 / sparkattn_select calls bit for bit."""
    H, d, block, topk = 3, 128, 128, 2
    g = torch.Generator().manual_seed(21)
    q = torch.randn((2, 700, H, d), generator=g).to(torch.bfloat16).to(DEV).permute(0, 2, 1, 3)
    k = torch.randn((2, 700, H, d), generator=g).to(torch.bfloat16).to(DEV).permute(0, 2, 1, 3)
    ws = sa.alloc_workspace(sa.make_shape(q, block), 0, topk, DEV)
    cq, sq = sa.quant_fp8_pooled(q, block, False, ws)
    ck, sk = sa.quant_fp8_pooled(k, block, True, ws)
    idx, cnt = sa.select_pooled(q, block, topk, ws)
    rq, rsq = sa.quant_fp8(q, block)
    rk, rsk = sa.quant_fp8(k, block)
    ridx, rcnt = sa.select(q, k, block, topk)
    assert cq.stride() == q.stride()
    assert torch.equal(cq, rq) and torch.equal(ck, rk)
    assert torch.equal(sq.view(torch.int32), rsq.view(torch.int32)) and torch.equal(sk.view(torch.int32), rsk.view(torch.int32))
    assert torch.equal(idx, ridx) and torch.equal(cnt, rcnt)


@pytest.mark.parametrize("H,nb,d,window", [(1, 257, 128, 0), (1, 263, 64, 0), (3, 300, 64, 0), (1, 1290, 64, 3), (8, 289, 128, 0), (8, 305, 64, 0)])
def test_few_heads_of_many_blocks(H, nb, d, window):
    """More than 256 key blocks, on either side of the number of query blocks from which a CTA takes 16 of them instead
    of 8 (8 heads of 289 blocks: 152 CTAs of 16): the oracle's lists."""
    g = torch.Generator().manual_seed(nb + d)
    N = nb * 64 - 29
    q, k = ((torch.randn((H, N, d), generator=g) + torch.randn((H, nb, 1, d), generator=g).expand(H, nb, 64, d).reshape(H, -1, d)[:, :N])
            .to(torch.bfloat16) for _ in range(2))
    kw = dict(frame_tokens=1000, window=window) if window else {}
    for topk in (1, nb // 30, nb // 2):
        idx, cnt = sa.select(q[None].to(DEV), k[None].to(DEV), 64, topk, **kw)
        ref_idx, ref_cnt = oracle.select(q, k, 64, topk, **kw)
        assert torch.equal(idx[0].cpu(), ref_idx) and torch.equal(cnt[0].cpu(), ref_cnt)


def test_selections_of_several_threads():
    """Threads with a stream each select at different sizes at the same time: a kernel's limit of dynamic shared memory is one
    for the whole process, and no thread may lower it between another one's setting and launch."""
    g = torch.Generator(device=DEV).manual_seed(9)
    cases = []
    for N, d, block, topk in ((1500, 128, 128, 3), (900, 128, 64, 4), (20000, 128, 64, 9), (6400, 128, 128, 7), (17000, 64, 64, 5), (700, 64, 64, 2)):
        q, k = (torch.randn((1, 2, N, d), generator=g, device=DEV).to(torch.bfloat16) for _ in range(2))
        cases.append((q, k, block, topk, sa.select(q, k, block, topk)))
    torch.cuda.synchronize()
    wrong = []

    def work(first):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for n in range(400):
                    q, k, block, topk, (idx, cnt) = cases[(first + n) % len(cases)]
                    i, c = sa.select(q, k, block, topk)
                    if n % 40 == 0 and not (torch.equal(i, idx) and torch.equal(c, cnt)):
                        wrong.append((first, n))
        except Exception as e:                      # a thread's exception would otherwise end the thread alone
            wrong.append(repr(e))

    threads = [threading.Thread(target=work, args=(j,)) for j in range(len(cases))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not wrong, wrong[:5]
