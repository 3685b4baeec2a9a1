"""Host-side checks of the C-ABI library that need no GPU: it loads, exports every symbol the
header declares, and rejects bad arguments with the documented status codes before any CUDA call."""
import ctypes as C
import os
import re

import pytest

import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import binding

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    text = open(os.path.join(ROOT, "include", "speckv.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(speckv_[a-z_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported():
    L = speckv.load_library()
    names = _declared()
    assert {"speckv_signals", "speckv_select_gamma", "speckv_verify", "speckv_step",
            "speckv_workspace_size"} <= set(names)
    for n in names:
        assert hasattr(L, n), n


def test_version_and_status_strings():
    assert speckv.version() >= 100
    assert speckv.status_string(0) == "ok"
    assert "workspace" in speckv.status_string(3)


def _cb(**kw):
    b = binding._CBatch()
    b.B, b.gamma_max, b.V, b.dtype = 4, 8, 128256, binding.BF16
    b.draft_logits = 0x1000
    b.draft_stride_b, b.draft_stride_pos = 8 * 128256, 128256
    b.temperature_scalar = 1.0
    for k, v in kw.items():
        setattr(b, k, v)
    return b


def test_workspace_size_and_argument_checks_without_a_gpu():
    L = speckv.load_library()
    n = C.c_size_t(0)
    assert L.speckv_workspace_size(C.byref(_cb()), C.byref(n)) == binding.OK and n.value >= 256
    small = n.value
    assert L.speckv_workspace_size(C.byref(_cb(B=64)), C.byref(n)) == binding.OK and n.value > small
    assert L.speckv_workspace_size(C.byref(_cb(V=0)), C.byref(n)) == binding.ERR_INVALID_ARG
    assert L.speckv_workspace_size(C.byref(_cb(gamma_max=17)), C.byref(n)) == binding.ERR_UNSUPPORTED
    assert L.speckv_workspace_size(C.byref(_cb()), None) == binding.ERR_INVALID_ARG
    # signals: NULL logits, bad dtype, bad strides, missing / misaligned / short workspace
    call = lambda b, ws, nb: L.speckv_signals(C.byref(b), None, None, None, None, ws, nb, None)
    assert call(_cb(draft_logits=None), 0x100, 1 << 30) == binding.ERR_INVALID_ARG
    assert call(_cb(dtype=7), 0x100, 1 << 30) == binding.ERR_UNSUPPORTED
    assert call(_cb(draft_stride_pos=100), 0x100, 1 << 30) == binding.ERR_INVALID_ARG
    assert call(_cb(), None, 1 << 30) == binding.ERR_INVALID_ARG
    assert call(_cb(), 0x101, 1 << 30) == binding.ERR_INVALID_ARG
    assert call(_cb(), 0x100, 16) == binding.ERR_WORKSPACE
    assert call(_cb(B=-1), 0x100, 1 << 30) == binding.ERR_INVALID_ARG
    # flags: the value 2 (no kernel behind it any more) and unknown bits are refused before anything is launched
    assert call(_cb(flags=2), 0x100, 1 << 30) == binding.ERR_INVALID_ARG
    assert call(_cb(flags=8), 0x100, 1 << 30) == binding.ERR_INVALID_ARG
    assert call(_cb(B=0), None, 0) == binding.OK          # empty batch: nothing to do
    # verify needs target, tokens and uniforms
    assert L.speckv_verify(C.byref(_cb()), 0x100, 0x100, None, 0x100, 1 << 30, None) == binding.ERR_INVALID_ARG
    # controller checks
    m = binding._CMlp()
    assert L.speckv_select_gamma(4, 0x100, None, C.byref(m), None, 0x100, None) == binding.ERR_INVALID_ARG
    m.n_in, m.n_hidden, m.n_out = 5, 64, 4
    m.W1 = m.b1 = m.W2 = m.b2 = 0x100
    assert L.speckv_select_gamma(4, 0x100, None, C.byref(m), None, 0x100, None) == binding.ERR_UNSUPPORTED


def test_shard_calls_refuse_buffers_off_the_grid_of_their_records():
    # the kernels read and write these in words of 16 bytes (states, row records) and 8 (token logits)
    L = speckv.load_library()
    b = _cb(V=4000, draft_stride_b=8 * 4000, draft_stride_pos=4000, target_logits=0x1000, target_stride_b=9 * 4000,
            target_stride_pos=4000, draft_tokens=0x1000, uniforms=0x1000)
    ok, big = 0x1000, 1 << 30
    bad = binding.ERR_INVALID_ARG
    for off in (4, 8):
        assert L.speckv_shard_sweep(C.byref(b), 0, ok + off, ok, 0x100, big, None) == bad
        assert L.speckv_shard_draw_sums(C.byref(b), ok + off, ok, 0x100, big, None) == bad
        assert L.speckv_shard_draw_pick(C.byref(b), 0, 0, 2, ok + off, ok, ok, 0x100, big, None) == bad
    assert L.speckv_shard_sweep(C.byref(b), 0, ok, ok + 4, 0x100, big, None) == bad


def test_sampling_workspace_does_not_outgrow_the_buffers_in_use():
    # a buffer of the size that was asked for when the sums were kept per 256 elements (44 bytes and 12 per chunk of each
    # position) goes on being accepted, whatever the vocabulary; a size for more rows serves fewer
    L = speckv.load_library()
    n = C.c_size_t(0)
    up = lambda x: -(-x // 256) * 256
    for dtype in (binding.F32, binding.BF16):
        for V in [*range(1, 600, 7), 1000, 2304, 4096, 8191, 20000, 31738, 31999, 32000, 32001, 32641, 33000, 50257, 65536, 151936, 1 << 24]:
            for B, G in ((1, 1), (3, 4), (64, 8), (1000, 16)):
                assert L.speckv_sample_workspace_size(C.byref(_cb(B=B, gamma_max=G, V=V, dtype=dtype)), C.byref(n)) == binding.OK
                pos, chunks = B * G, -(-V // 256)
                before = sum(up(x) for x in ((2 * B + pos) * 4, pos * 32, pos * 512, pos * chunks * 4, pos * chunks * 8))
                assert n.value <= before, (dtype, V, B, G, n.value, before)


def test_binding_refuses_cpu_tensors():
    import torch
    with pytest.raises(ValueError, match="CUDA"):
        speckv.speckv_signals(speckv.Batch(draft_logits=torch.zeros(1, 2, 16)))
