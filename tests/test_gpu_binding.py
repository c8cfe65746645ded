"""The binding's native marshalling (csrc/binding.cpp) against the same entry points called through ctypes: the same bits, on
strided tensors, for every call it makes."""
import ctypes

import pytest
import torch

import paper_2609_23153_b200 as sa
import workloads

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
H, BLOCK, TOPK = 3, 128, 3
GRID = (3, 15, 20)


def _p(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def _ctypes_call(name, out, *args):
    L = sa.lib()
    rc = getattr(L, "sparkattn_" + name)(*args, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == sa.OK
    return out


@pytest.mark.parametrize("call", ["select", "select_window", "select_padded", "quant", "quant_pooled", "quant_token", "fwd", "fwd_fp8",
                                  "fwd_window", "fwd_padded", "gather", "comp", "fwd_gated"])
def test_native_calls_equal_ctypes_calls(call):
    g = torch.Generator(device=DEV).manual_seed(5)
    q, k, v = (torch.randn((2, 900, H, 128), generator=g, device=DEV).to(torch.bfloat16).permute(0, 2, 1, 3) for _ in range(3))
    if call.endswith("padded"):                 # bricks: a whole number of blocks
        q, k, v = (t[:, :, :896] for t in (q, k, v))
    N = q.shape[2]
    nb = -(-N // BLOCK)
    shape = sa.make_shape(q, BLOCK)
    ref = ctypes.byref(shape)
    ws = torch.zeros(1 << 22, dtype=torch.uint8, device=DEV)
    tail = (_p(ws), ctypes.c_size_t(ws.numel()))
    idx, cnt = torch.empty((2, H, nb, TOPK), dtype=torch.int32, device=DEV), torch.empty((2, H, nb), dtype=torch.int32, device=DEV)
    valid = torch.full((nb,), 100, dtype=torch.int32, device=DEV)
    pq, pk, gate = workloads.compensation_params(workloads.Workload("binding", 3, 2, H, 128, GRID, 128, 0.0), 64, device=DEV)
    axis, freq = workloads.rope_schedule(128, 64)
    grid = (ctypes.c_int32 * 3)(*GRID)
    if call.startswith("select"):
        kw = {"select": {}, "select_window": dict(frame_tokens=300, window=2), "select_padded": dict(block_valid=valid)}[call]
        got = sa.select(q, k, BLOCK, TOPK, **kw)
        mid = {"select": (), "select_window": (300, 2), "select_padded": (_p(valid),)}[call]
        want = _ctypes_call(call, (idx, cnt), ref, _p(q), _p(k), TOPK, *mid, _p(idx), _p(cnt), *tail)
    elif call.startswith("quant"):
        codes, scales = torch.empty_strided(q.shape, q.stride(), dtype=torch.uint8, device=DEV), torch.empty((2, H, nb), device=DEV)
        if call == "quant":
            got = sa.quant_fp8(q, BLOCK)
            want = _ctypes_call("quant_fp8", (codes, scales), ref, _p(q), _p(codes), _p(scales), 0)
        elif call == "quant_token":
            scales = torch.empty((2, H, N), device=DEV)
            got = sa.quant_fp8_per_token(q)
            want = _ctypes_call("quant_fp8_per_token", (codes, scales), ref, _p(q), _p(codes), _p(scales))
        else:
            mine = sa.alloc_workspace(shape, 0, TOPK, DEV)
            pooled = [sa.quant_fp8_pooled(t, BLOCK, side, mine) for t, side in ((q, False), (k, True))]
            got = (*pooled[0], *sa.select_pooled(q, BLOCK, TOPK, mine))
            for t, side in ((k, 1), (q, 0)):
                _ctypes_call("quant_fp8_pooled", None, ref, _p(t), _p(codes), _p(scales), side, *tail)
            want = (codes, scales, *_ctypes_call("select_pooled", (idx, cnt), ref, TOPK, _p(idx), _p(cnt), *tail))
    elif call == "gather":
        index = torch.randint(-1, N, (1100,), generator=g, device=DEV, dtype=torch.int32)
        got = (sa.gather_tokens(q, index),)
        out = torch.empty((2, H, 1100, 128), dtype=torch.bfloat16, device=DEV)
        want = _ctypes_call("gather_tokens", (out,), ref, _p(q), ctypes.byref(sa.make_shape(out, 128)), _p(index), _p(out), *tail)
    else:
        idx, cnt = sa.select(q, k, BLOCK, TOPK)
        out, lse = torch.empty_strided(q.shape, q.stride(), dtype=torch.bfloat16, device=DEV), torch.empty((2, H, N), device=DEV)
        if call in ("comp", "fwd_gated"):
            state = sa.comp_state(k, v, pk, GRID, axis, freq)
        if call == "comp":
            st = torch.empty_like(state)
            _ctypes_call("comp_state", None, ref, _p(k), _p(v), _p(pk), 64, grid, _p(axis), _p(freq), _p(st), *tail)
            got = (state, sa.comp_apply(q, pq, state, gate, v, GRID, axis, freq, eps=1e-5))
            want = _ctypes_call("comp_apply", (st, out), ref, _p(q), _p(pq), 64, grid, _p(axis), _p(freq), _p(st), _p(gate), _p(v),
                                _p(out), ctypes.c_float(1e-5), *tail)
        elif call == "fwd_gated":
            got = sa.fwd_gated(q, k, v, idx, cnt, pq, state, gate, GRID, axis, freq, softmax_scale=0.05, return_lse=True)
            scaled = ctypes.byref(sa.make_shape(q, BLOCK, 0.05))
            want = _ctypes_call("fwd_gated", (out, lse), scaled, _p(q), _p(k), _p(v), _p(idx), _p(cnt), TOPK, _p(pq), 64, grid,
                                _p(axis), _p(freq), _p(state), _p(gate), ctypes.c_float(1e-6), _p(out), _p(lse), *tail)
        else:
            t, sc, dtype, kw = (q, k, v), (None,) * 3, sa.BF16, {}
            if call == "fwd_fp8":
                t, sc = zip(*(sa.quant_fp8(x, BLOCK) for x in t))
                dtype, kw = sa.FP8_E4M3, dict(scales=sc)
            mid = {"fwd_window": (300, 2), "fwd_padded": (_p(valid),)}.get(call, ())
            kw.update({"fwd_window": dict(frame_tokens=300, window=2), "fwd_padded": dict(block_valid=valid)}.get(call, {}))
            got = sa.fwd(*t, idx, cnt, BLOCK, return_lse=True, **kw)
            want = _ctypes_call(call if mid else "fwd", (out, lse), ref, dtype, *map(_p, t), *map(_p, sc), _p(idx), _p(cnt), TOPK, *mid,
                                _p(out), _p(lse), *tail)
    torch.cuda.synchronize()
    assert len(got) == len(want)
    for a, b in zip(got, want):
        assert a.dtype == b.dtype and a.shape == b.shape and a.stride() == b.stride()
        assert torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))
