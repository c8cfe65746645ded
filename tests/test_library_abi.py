"""Host-side checks that need no GPU: the C-ABI library loads, exports every
symbol the public header declares, and rejects bad arguments before touching
the device."""
import ctypes
import os
import re

import pytest
import torch

import paper_2609_23153_b200 as sa

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2609_23153_b200 import build
    build.build()
    return sa.lib()


def test_binding_of_another_torch_or_python_is_rebuilt(lib, monkeypatch, tmp_path):
    """The native marshalling belongs to the torch and the Python that it was built against; nothing in the source tree
    changes when one of them does."""
    from paper_2609_23153_b200 import build
    assert not build.needs_build()
    for module, name in ((torch, "__version__"), (torch.version, "git_version")):
        with monkeypatch.context() as m:
            m.setattr(module, name, "another")
            assert build.needs_build()
    with monkeypatch.context() as m:
        m.setattr(build.sysconfig, "get_config_var", lambda name: "another")
        assert build.needs_build()
    with monkeypatch.context() as m:                          # built before this was recorded
        m.setattr(build, "BINDING_FOR", str(tmp_path / "none"))
        assert build.needs_build()
    assert not build.needs_build()


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "sparkattn.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(sparkattn_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = _declared_symbols()
    assert set(sa.EXPORTS) <= set(names)
    for n in names:
        assert hasattr(lib, n), f"{n} declared in sparkattn.h but not exported"


def test_version_and_status_strings(lib):
    assert lib.sparkattn_version() == sa.VERSION
    seen = set()
    for code in range(0, -9, -1):
        s = sa.status_string(code)
        assert s and s != "unknown status" and s not in seen
        seen.add(s)
    assert sa.status_string(-99) == "unknown status"


def _shape(B=1, H=2, N=2048, d=64, block=64):
    return sa.Shape(ctypes.sizeof(sa.Shape), sa.VERSION, B, H, N, d, block, 0, H * N * d, N * d, d, 0.0, 0)


def test_shape_struct_matches_header_size():
    # 2*u32 + 6*i32 + 3*i64 + f32 + u32 = 64 bytes, no implicit padding
    assert ctypes.sizeof(sa.Shape) == 64


def test_workspace_sizes(lib):
    s = _shape()
    nb = 32
    assert sa.workspace_bytes(s, 1, 16) == 256
    assert sa.workspace_bytes(s, 0, 16) == 256 + 2 * nb * 64 * 4 + 2 * 64 * 32 * 4
    assert sa.workspace_bytes(s, 2, 0) == 256          # the gather call: status header only
    assert sa.workspace_bytes(s, 3, 16) == 0
    bad = _shape(d=96)
    assert sa.workspace_bytes(bad, 0, 16) == 0
    assert sa.arena_bytes(s, sa.BF16, 16) > 4 * 2 * 2048 * 64 * 2
    assert sa.arena_bytes(s, sa.BF16, 0) == 0


def test_argument_errors_are_caught_on_the_host(lib):
    s = _shape()
    fake = ctypes.c_void_p(0x1000)  # never dereferenced: validation fails first
    null = ctypes.c_void_p(0)
    st = ctypes.c_void_p(0)
    r = lib.sparkattn_select(ctypes.byref(s), null, fake, 4, fake, null, fake, 1 << 20, st)
    assert r == sa.E_INVALID_ARG
    r = lib.sparkattn_select(ctypes.byref(s), fake, fake, 0, fake, null, fake, 1 << 20, st)
    assert r == sa.E_INVALID_ARG
    r = lib.sparkattn_select(ctypes.byref(s), fake, fake, 33, fake, null, fake, 1 << 20, st)
    assert r == sa.E_INVALID_ARG
    r = lib.sparkattn_select(ctypes.byref(s), fake, fake, 4, fake, null, fake, 16, st)
    assert r == sa.E_WORKSPACE_TOO_SMALL
    r = lib.sparkattn_select(ctypes.byref(s), ctypes.c_void_p(0x1008), fake, 4, fake, null, fake, 1 << 20, st)
    assert r == sa.E_MISALIGNED
    bad = _shape(d=96)
    assert lib.sparkattn_quant_fp8(ctypes.byref(bad), fake, fake, fake, 0, st) == sa.E_UNSUPPORTED_SHAPE
    assert lib.sparkattn_quant_fp8(ctypes.byref(s), fake, fake, fake, 1, st) == sa.E_INVALID_ARG
    odd = _shape()
    odd.stride_n = 72
    assert lib.sparkattn_quant_fp8(ctypes.byref(odd), fake, fake, fake, 0, st) == sa.E_MISALIGNED
    wrong = _shape()
    wrong.version = 7
    assert lib.sparkattn_quant_fp8(ctypes.byref(wrong), fake, fake, fake, 0, st) == sa.E_INVALID_ARG
    # fwd: FP8 needs scales and the 128/128 shape; kmax in range
    r = lib.sparkattn_fwd(ctypes.byref(s), sa.FP8_E4M3, fake, fake, fake, null, null, null, fake, null, 4, fake,
                          null, fake, 256, st)
    assert r == sa.E_INVALID_ARG
    r = lib.sparkattn_fwd(ctypes.byref(s), sa.FP8_E4M3, fake, fake, fake, fake, fake, fake, fake, null, 4, fake,
                          null, fake, 256, st)
    assert r == sa.E_UNSUPPORTED_SHAPE            # FP8 needs d = 128
    assert sa.workspace_bytes(_shape(d=64, block=64), 1, 4) == 256
    # d = 128 keeps checked copies of the kept lists behind the status words: per item, or per pair of 64-token blocks
    assert sa.workspace_bytes(_shape(d=128, block=128), 1, 4) == 256 + 256 + 2 * 16 * 4 * 4 + 2 * 4
    assert sa.workspace_bytes(_shape(d=128, block=64), 1, 4) == 256 + 256 + 2 * 16 * 8 * 4 + 2 * 4
    assert sa.workspace_bytes(_shape(d=128, block=64), 1, 0) == 0
    assert sa.workspace_bytes(_shape(d=64, block=128), 1, 4) == 0
    r = lib.sparkattn_fwd(ctypes.byref(s), sa.BF16, fake, fake, fake, null, null, null, fake, null, 40, fake,
                          null, fake, 256, st)
    assert r == sa.E_INVALID_ARG
    r = lib.sparkattn_fwd(ctypes.byref(s), 5, fake, fake, fake, null, null, null, fake, null, 4, fake,
                          null, fake, 256, st)
    assert r == sa.E_INVALID_ARG
    r = lib.sparkattn_fwd(ctypes.byref(s), sa.BF16, fake, fake, fake, null, null, null, fake, null, 4, fake,
                          null, fake, 8, st)
    assert r == sa.E_WORKSPACE_TOO_SMALL
    # causal window: frame size and window length must be positive; selection with a window needs kept_cnt
    r = lib.sparkattn_fwd_window(ctypes.byref(s), sa.BF16, fake, fake, fake, null, null, null, fake, null, 4, 0, 1, fake,
                                 null, fake, 256, st)
    assert r == sa.E_INVALID_ARG
    r = lib.sparkattn_fwd_window(ctypes.byref(s), sa.BF16, fake, fake, fake, null, null, null, fake, null, 4, 64, 0, fake,
                                 null, fake, 256, st)
    assert r == sa.E_INVALID_ARG
    r = lib.sparkattn_select_window(ctypes.byref(s), fake, fake, 4, 64, 1, fake, null, fake, 1 << 20, st)
    assert r == sa.E_INVALID_ARG
    r = lib.sparkattn_select_window(ctypes.byref(s), fake, fake, 4, 64, 1, fake, fake, fake, 16, st)
    assert r == sa.E_WORKSPACE_TOO_SMALL
    # compensation branch: d = 128 and rank 64 only; the grid must cover N; rotary tables checked
    s128 = _shape(d=128, block=128)
    grid = (ctypes.c_int32 * 3)(2, 32, 32)
    axis = (ctypes.c_int32 * 32)(*([0] * 32))
    freq = (ctypes.c_float * 32)(*([1.0] * 32))
    r = lib.sparkattn_comp_state(ctypes.byref(s), fake, fake, fake, 64, grid, axis, freq, fake, fake, 1 << 30, st)
    assert r == sa.E_UNSUPPORTED_SHAPE            # d = 64
    r = lib.sparkattn_comp_state(ctypes.byref(s128), fake, fake, fake, 32, grid, axis, freq, fake, fake, 1 << 30, st)
    assert r == sa.E_UNSUPPORTED_SHAPE            # rank 32
    bad_grid = (ctypes.c_int32 * 3)(2, 32, 31)
    r = lib.sparkattn_comp_state(ctypes.byref(s128), fake, fake, fake, 64, bad_grid, axis, freq, fake, fake, 1 << 30, st)
    assert r == sa.E_INVALID_ARG
    axis[5] = 3
    r = lib.sparkattn_comp_state(ctypes.byref(s128), fake, fake, fake, 64, grid, axis, freq, fake, fake, 1 << 30, st)
    assert r == sa.E_INVALID_ARG
    axis[5] = 0
    r = lib.sparkattn_comp_state(ctypes.byref(s128), fake, fake, fake, 64, grid, axis, freq, fake, fake, 256, st)
    assert r == sa.E_WORKSPACE_TOO_SMALL
    r = lib.sparkattn_comp_apply(ctypes.byref(s128), fake, fake, 64, grid, axis, freq, fake, fake, fake, fake,
                                 ctypes.c_float(0.0), fake, 1 << 20, st)
    assert r == sa.E_INVALID_ARG                  # eps must be positive
    assert lib.sparkattn_comp_workspace_bytes(ctypes.byref(s128), bad_grid) == 0
    assert lib.sparkattn_comp_workspace_bytes(ctypes.byref(s128), grid) > 256


def test_fused_quant_pool_entry_points_validate_on_the_host(lib):
    s = _shape()
    fake = ctypes.c_void_p(0x1000)
    null = ctypes.c_void_p(0)
    st = ctypes.c_void_p(0)
    need = sa.workspace_bytes(s, 0, 4)
    assert lib.sparkattn_quant_fp8_pooled(ctypes.byref(s), fake, fake, fake, 2, fake, need, st) == sa.E_INVALID_ARG
    assert lib.sparkattn_quant_fp8_pooled(ctypes.byref(s), fake, fake, fake, 0, null, need, st) == sa.E_INVALID_ARG
    assert lib.sparkattn_quant_fp8_pooled(ctypes.byref(s), fake, fake, fake, 1, fake, need - 1, st) == sa.E_WORKSPACE_TOO_SMALL
    assert lib.sparkattn_quant_fp8_pooled(ctypes.byref(s), fake, fake, fake, 1, ctypes.c_void_p(0x1010), need, st) == sa.E_MISALIGNED
    assert lib.sparkattn_select_pooled(ctypes.byref(s), 0, fake, null, fake, need, st) == sa.E_INVALID_ARG
    assert lib.sparkattn_select_pooled(ctypes.byref(s), 33, fake, null, fake, need, st) == sa.E_INVALID_ARG
    assert lib.sparkattn_select_pooled(ctypes.byref(s), 4, fake, null, fake, 16, st) == sa.E_WORKSPACE_TOO_SMALL
    assert lib.sparkattn_select_pooled(ctypes.byref(_shape(d=96)), 4, fake, null, fake, need, st) == sa.E_UNSUPPORTED_SHAPE


def test_binding_checks_layout():
    q = torch.zeros((1, 2, 128, 64), dtype=torch.bfloat16)
    with pytest.raises(ValueError):
        sa.make_shape(q.transpose(2, 3), 64)
    s = sa.make_shape(q, 64)
    assert (s.B, s.H, s.N, s.d, s.block) == (1, 2, 128, 64, 64)
    assert (s.stride_b, s.stride_h, s.stride_n) == (2 * 128 * 64, 128 * 64, 64)
    # a [B, N, H, d] buffer viewed as [B, H, N, d]
    x = torch.zeros((1, 128, 2, 64), dtype=torch.bfloat16).permute(0, 2, 1, 3)
    s = sa.make_shape(x, 64)
    assert (s.stride_h, s.stride_n) == (64, 128)


def test_missing_library_fails_loudly(monkeypatch, tmp_path):
    monkeypatch.setattr(sa, "_lib", None)
    monkeypatch.setattr(sa, "LIB_PATH", str(tmp_path / "nope.so"))
    with pytest.raises(ImportError):
        sa.lib()


def test_padded_brick_entry_points_validate_on_the_host(lib):
    s128 = _shape(d=128, block=128, N=4096)
    s64 = _shape()
    fake = ctypes.c_void_p(0x1000)
    null = ctypes.c_void_p(0)
    st = ctypes.c_void_p(0)
    grid = (ctypes.c_int32 * 3)(21, 45, 80)
    brick = (ctypes.c_int32 * 3)(3, 5, 8)
    gp, bp = ctypes.cast(grid, ctypes.c_void_p), ctypes.cast(brick, ctypes.c_void_p)
    lib.sparkattn_brick_count.restype = ctypes.c_int64
    assert lib.sparkattn_brick_count(gp, bp) == 7 * 9 * 10
    assert lib.sparkattn_brick_count(null, bp) == 0
    zero = (ctypes.c_int32 * 3)(3, 0, 8)
    assert lib.sparkattn_brick_count(gp, ctypes.cast(zero, ctypes.c_void_p)) == 0
    big = (ctypes.c_int32 * 3)(3, 9, 8)                                   # 216 cells > 128
    assert lib.sparkattn_brick_layout(gp, ctypes.cast(big, ctypes.c_void_p), 128, fake, fake, fake, st) == sa.E_INVALID_ARG
    assert lib.sparkattn_brick_layout(gp, bp, 100, fake, fake, fake, st) == sa.E_INVALID_ARG
    assert lib.sparkattn_brick_layout(gp, bp, 128, null, null, null, st) == sa.E_INVALID_ARG
    # select / fwd on padded bricks: block_valid required, N a multiple of the block, d = 128
    r = lib.sparkattn_select_padded(ctypes.byref(s128), fake, fake, 4, null, fake, null, fake, 1 << 24, st)
    assert r == sa.E_INVALID_ARG
    ragged = _shape(d=128, block=128, N=4000)
    r = lib.sparkattn_select_padded(ctypes.byref(ragged), fake, fake, 4, fake, fake, null, fake, 1 << 24, st)
    assert r == sa.E_INVALID_ARG
    r = lib.sparkattn_select_padded(ctypes.byref(s64), fake, fake, 4, fake, fake, null, fake, 1 << 24, st)
    assert r == sa.E_UNSUPPORTED_SHAPE
    r = lib.sparkattn_fwd_padded(ctypes.byref(s64), sa.BF16, fake, fake, fake, null, null, null, fake, fake, 4, fake, fake,
                                 null, fake, 1 << 24, st)
    assert r == sa.E_UNSUPPORTED_SHAPE
    r = lib.sparkattn_fwd_padded(ctypes.byref(s128), sa.BF16, fake, fake, fake, null, null, null, fake, fake, 4, null, fake,
                                 null, fake, 1 << 24, st)
    assert r == sa.E_INVALID_ARG
    # gather: shapes must agree in B, H, d; buffers must differ; workspace holds the status header
    other = _shape(d=128, block=128, N=4096)
    other.H = s128.H + 1
    assert lib.sparkattn_gather_tokens(ctypes.byref(s128), fake, ctypes.byref(other), fake, ctypes.c_void_p(0x2000), fake, 256, st) == sa.E_INVALID_ARG
    assert lib.sparkattn_gather_tokens(ctypes.byref(s128), fake, ctypes.byref(s128), fake, fake, fake, 256, st) == sa.E_INVALID_ARG
    assert lib.sparkattn_gather_tokens(ctypes.byref(s128), fake, ctypes.byref(s128), fake, ctypes.c_void_p(0x2000), fake, 16, st) == sa.E_WORKSPACE_TOO_SMALL


def test_host_buffer_call_rejects_more_batches_than_head_groups(lib):
    """The host-buffer path runs at most 16 head groups and a group never spans two batch entries: B = 17
    must come back as an error at once (it used to loop for ever while sizing the groups)."""
    fake = ctypes.c_void_p(0x1000)
    st = ctypes.c_void_p(0)
    s = _shape(B=17, H=2, N=256, d=64, block=64)
    r = lib.sparkattn_attention_host(ctypes.byref(s), sa.BF16, fake, fake, fake, 2, fake, ctypes.c_void_p(0), fake, 1 << 40, st)
    assert r == sa.E_UNSUPPORTED_SHAPE
    # 16 batch entries of many heads still form 16 groups (one per batch entry): passes the group sizing
    # and stops at the arena-size check
    s = _shape(B=16, H=40, N=256, d=64, block=64)
    r = lib.sparkattn_attention_host(ctypes.byref(s), sa.BF16, fake, fake, fake, 2, fake, ctypes.c_void_p(0), fake, 256, st)
    assert r == sa.E_WORKSPACE_TOO_SMALL


def test_gated_forward_validates_on_the_host(lib):
    """sparkattn_fwd_gated: every argument check happens before the device is touched."""
    s = _shape(N=2048, d=128, block=128)
    fake = ctypes.c_void_p(0x1000)
    null = ctypes.c_void_p(0)
    st = ctypes.c_void_p(0)
    grid = (ctypes.c_int32 * 3)(2, 32, 32)
    axis = (ctypes.c_int32 * 32)(*([0] * 10 + [1] * 11 + [2] * 11))
    freq = (ctypes.c_float * 32)(*[0.01 * (m + 1) for m in range(32)])
    eps = ctypes.c_float(1e-6)
    need = lib.sparkattn_fwd_gated_workspace_bytes(ctypes.byref(s), 4, grid)
    assert need > sa.workspace_bytes(s, 1, 4)          # the plain forward's workspace plus the rotary table

    def call(shape=s, q=fake, kmax=4, rank=64, g=grid, ax=axis, e=eps, ws=fake, nbytes=need, state=fake):
        return lib.sparkattn_fwd_gated(ctypes.byref(shape), q, fake, fake, fake, null, kmax, fake, rank, g, ax, freq, state,
                                       fake, e, fake, null, ws, nbytes, st)

    assert call(q=null) == sa.E_INVALID_ARG
    assert call(state=null) == sa.E_INVALID_ARG
    assert call(kmax=0) == sa.E_INVALID_ARG
    assert call(kmax=17) == sa.E_INVALID_ARG                          # more than the 16 key blocks
    assert call(e=ctypes.c_float(0.0)) == sa.E_INVALID_ARG
    assert call(g=(ctypes.c_int32 * 3)(2, 32, 31)) == sa.E_INVALID_ARG     # grid does not multiply to N
    assert call(ax=(ctypes.c_int32 * 32)(*([3] * 32))) == sa.E_INVALID_ARG
    assert call(rank=32) == sa.E_UNSUPPORTED_SHAPE
    assert call(shape=_shape(N=2048, d=128, block=64)) == sa.E_UNSUPPORTED_SHAPE
    assert call(shape=_shape(N=2048, d=64, block=128)) == sa.E_UNSUPPORTED_SHAPE
    assert call(q=ctypes.c_void_p(0x1008)) == sa.E_MISALIGNED
    assert call(ws=ctypes.c_void_p(0x1010)) == sa.E_MISALIGNED
    assert call(nbytes=need - 1) == sa.E_WORKSPACE_TOO_SMALL
    assert lib.sparkattn_fwd_gated_workspace_bytes(ctypes.byref(_shape(N=2048, d=128, block=64)), 4, grid) == 0
    assert lib.sparkattn_fwd_gated_workspace_bytes(ctypes.byref(s), 4, (ctypes.c_int32 * 3)(2, 32, 31)) == 0


def test_early_launched_kernels_read_with_ordinary_loads():
    """A kernel that calls pdl_wait may be resident while the kernels before it write what it reads.  A read-only load
    is only defined for data that nothing writes during the kernel's life, so neither __ldg nor a const __restrict__
    parameter may stand in such a kernel or in what it calls."""
    src = os.path.join(ROOT, "paper_2609_23153_b200", "csrc")
    kernels = 0
    for name in sorted(f for f in os.listdir(src) if f.endswith(".cu")):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(src, name)).read())
        if "pdl_wait" not in text:
            continue
        assert "__ldg" not in text, name
        for kernel in re.split(r"\b__global__\b", text)[1:]:
            if "pdl_wait" not in kernel:
                continue
            kernels += 1
            params = kernel[:kernel.index("{")]
            assert not re.search(r"const[^,]*__restrict__", params), (name, params.split("(")[0])
    assert kernels >= 7


def test_only_kernels_inside_a_call_let_the_next_one_in_early():
    """A kernel that ends a call does not know what follows, and the pooling kernel of a selection that is let in while it
    drains is placed unevenly for its whole run.  The pooling quantisation and the state pass may (what they are for says what
    follows), and every other kernel with pdl_trigger is followed by another one of the same call."""
    src = os.path.join(ROOT, "paper_2609_23153_b200", "csrc")
    found = {}
    for name in sorted(f for f in os.listdir(src) if f.endswith(".cu")):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(src, name)).read())
        for kernel in re.split(r"\b__global__\b", text)[1:]:
            if "pdl_trigger" in kernel:
                found[re.search(r"(\w+)\s*\((?=[^()]*(const|int))", kernel[kernel.index("void"):]).group(1)] = name
    assert found == {"rope_table_kernel": "comp.cu", "comp_state_kernel": "comp.cu", "comp_reduce_kernel": "comp.cu", "clear_header_kernel": "fwd.cu",
                     "compact_lists_kernel": "fwd_pipe.cu", "pair_lists_kernel": "fwd_pipe.cu", "head_vmax_kernel": "fwd_pipe.cu",
                     "pool_kernel": "select.cu", "quant_fp8_pool_kernel": "quant.cu"}


def test_failed_rotary_table_launch_is_reported(lib):
    """A grid of no positions is a launch without blocks: the runtime refuses it on the host, with or without a device,
    and the launcher has to hand that on (the gated forward would read a table that nothing wrote)."""
    name = "_ZN9sparkattn17launch_rope_tableERKNS_9RopeTableEP6float2P11CUstream_st"
    launch = getattr(ctypes.CDLL(sa.LIB_PATH), name)
    launch.restype = ctypes.c_int
    launch.argtypes = [ctypes.c_void_p] * 3
    rope = (ctypes.c_int32 * 67)()                            # axis[32], freq[32], T, Hg, Wg
    assert launch(rope, None, None) == sa.E_CUDA


def test_current_stream_without_the_private_name(monkeypatch):
    """The binding takes the current stream's handle through a name that torch may drop; the public way stays."""
    class Stream:
        cuda_stream = 0x1230

    monkeypatch.setattr(torch.cuda, "current_stream", lambda: Stream)
    monkeypatch.setattr(sa, "_raw_stream", None)
    assert sa._stream_ptr(None) == 0x1230
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(sa, "_raw_stream", lambda device: 0x4560 + device)
    assert sa._stream_ptr(None) == 0x4563
    assert sa._stream_ptr(Stream) == 0x1230


def test_binding_refuses_what_it_refused(lib):
    """Errors of the native marshalling, which come before any device work: layouts that differ, a strided last dimension,
    arguments that are no tensors, shapes that the library does not serve, and operands of the compensation branch."""
    q = torch.zeros((1, 2, 256, 128), dtype=torch.bfloat16)
    idx, cnt = torch.zeros((1, 2, 2, 1), dtype=torch.int32), torch.ones((1, 2, 2), dtype=torch.int32)
    pk, axis, freq = torch.zeros((2, 64, 128), dtype=torch.bfloat16), torch.zeros(32, dtype=torch.int32), torch.zeros(32)
    state, gate = torch.zeros((1, 2, 64, 128)), torch.zeros((1, 2, 256))
    other = torch.zeros((1, 256, 2, 128), dtype=torch.bfloat16).transpose(1, 2)      # the same shape, other strides
    turned = q.transpose(2, 3)
    for call in (lambda: sa.select(q, other, 128, 1), lambda: sa.fwd(q, q, other, idx, cnt, 128), lambda: sa.quant_fp8(turned, 128),
                 lambda: sa.select(turned, turned, 128, 1), lambda: sa.gather_tokens(q, cnt), lambda: sa.comp_state(q, other, pk, (1, 1, 256), axis, freq),
                 lambda: sa.comp_state(q, q, pk, (1, 1, 256), axis, freq[:16]), lambda: sa.comp_state(q, q, pk[:1], (1, 1, 256), axis, freq),
                 lambda: sa.comp_apply(q, pk, state[:, :1], gate, q, (1, 1, 256), axis, freq),
                 lambda: sa.fwd_gated(q, q, q, idx, cnt, pk, state, gate.double(), (1, 1, 256), axis, freq),
                 lambda: sa.fwd(q, q, q, idx, cnt, 128, frame_tokens=64, window=1, block_valid=cnt[0, 0])):
        with pytest.raises(ValueError):
            call()
    with pytest.raises(TypeError):
        sa.fwd(q, q, [1.0], idx, cnt, 128)
    for call in (lambda: sa.select(q, q, 96, 1), lambda: sa.fwd(q, q, q, idx, cnt, 96)):
        with pytest.raises(sa.SparkAttnError) as e:
            call()
        assert e.value.status == sa.E_UNSUPPORTED_SHAPE


class _DefaultStream:
    cuda_stream = 0


@pytest.mark.parametrize("block", [0, -1, -128, -(1 << 31)])
def test_binding_leaves_block_sizes_to_the_library(lib, block):
    """A block size below 1 is an unsupported shape like any other that the library does not serve: the binding sizes its
    outputs by the number of blocks, which no such size has."""
    q = torch.zeros((1, 2, 256, 128), dtype=torch.bfloat16)
    idx, cnt = torch.zeros((1, 2, 2, 1), dtype=torch.int32), torch.ones((1, 2, 2), dtype=torch.int32)
    ws = torch.zeros(1 << 16, dtype=torch.uint8)
    kw = dict(stream=_DefaultStream)                 # refused before the stream is used
    for call in (lambda: sa.select(q, q, block, 1, **kw), lambda: sa.select(q, q, block, 1, kept_idx=idx, kept_cnt=cnt, workspace=ws, **kw),
                 lambda: sa.select_pooled(q, block, 1, ws, **kw), lambda: sa.select_pooled(q, block, 1, ws, kept_idx=idx, kept_cnt=cnt, **kw),
                 lambda: sa.fwd(q, q, q, idx, cnt, block, **kw), lambda: sa.fwd(q, q, q, idx, cnt, block, workspace=ws, **kw)):
        with pytest.raises(sa.SparkAttnError) as e:
            call()
        assert e.value.status == sa.E_UNSUPPORTED_SHAPE


@pytest.mark.parametrize("block", [0, -1, -128])
def test_block_quantisation_has_no_hidden_mode(lib, block):
    """quant_fp8 and quant_fp8_pooled scale by token block: a block size that there is none of is refused, whatever
    buffers come with it, and is not taken for the per-token call, which writes N scales per head."""
    x = torch.zeros((1, 2, 256, 128), dtype=torch.bfloat16)
    ws = torch.zeros(1 << 16, dtype=torch.uint8)
    own = dict(codes=torch.full((1, 2, 256, 128), 7, dtype=torch.uint8), scales=torch.full((1, 2, 2), 7.0))
    for kw in ({}, own):
        for call in (lambda: sa.quant_fp8(x, block, stream=_DefaultStream, **kw),
                     lambda: sa.quant_fp8_pooled(x, block, False, ws, stream=_DefaultStream, **kw),
                     lambda: sa.quant_fp8_pooled(x, block, True, ws, stream=_DefaultStream, **kw)):
            with pytest.raises(sa.SparkAttnError) as e:
                call()
            assert e.value.status == sa.E_UNSUPPORTED_SHAPE
    assert torch.all(own["codes"] == 7) and torch.all(own["scales"] == 7)


def test_bench_counts_the_launches_that_the_launchers_make():
    """The benchmark's launch counts take the forward's lines from its source, on both sides of each."""
    import bench
    import workloads
    text = open(os.path.join(ROOT, "paper_2609_23153_b200", "csrc", "fwd_pipe.cu")).read()
    own = int(re.search(r"constexpr int kOwnItems = (\d+);", text).group(1))
    make = lambda H, blocks, d, block, sparsity: workloads.Workload("launches", 1, 1, H, d, (1, blocks, block), block, sparsity)
    for d, block, per_sm, items in ((128, 128, own, 37), (128, 64, own, 37), (64, 64, 1, 37)):
        blocks = 2 * items if (d, block) == (128, 64) else items
        edge = per_sm * 148 // items                          # 4 heads of 37 items fill 148 SMs, 64 of them 16 times over
        assert edge * items == per_sm * 148
        for H, fwd in ((edge, 1), (edge + 1, 2)):
            assert bench.launches_per_step(make(H, blocks, d, block, 0.5), H, 148) == (2, fwd)
            assert bench.launches_per_step(make(H, blocks, d, block, 0.0), H, 148) == (1, fwd)
    assert bench.launches_per_step(workloads.WORKLOADS["wan14b"], 40, 148) == (2, 2)
