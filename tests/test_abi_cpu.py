"""CPU-side checks of the boundary: the library builds, loads and exports every symbol the public
header declares; the schedule the library exports agrees with the printed table.  No compute calls."""
import os
import re

import numpy as np
import pytest

import synth_inputs as si
from paper_2512_16483_b200 import build as fbuild
from paper_2512_16483_b200 import schedule

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    text = open(os.path.join(ROOT, "include", "fvar.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(fvar_[a-z0-9_]+)\s*\(", text)))


def test_library_builds_loads_and_exports_every_declared_symbol():
    fbuild.build()
    from paper_2512_16483_b200 import binding
    lib = binding.load_library()
    names = _declared()
    assert len(names) >= 20
    for n in names:
        assert hasattr(lib, n), n
    assert sorted(binding.EXPORTED) == names


def test_library_loads_without_its_call_layer(monkeypatch):
    """The call layer is built against torch.  Where it does not load, the error names the reason, and what needs no
    tensors works."""
    import sys
    from paper_2512_16483_b200 import binding
    fbuild.build()
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_calls", None)
    monkeypatch.delattr("paper_2512_16483_b200._calls", raising=False)
    monkeypatch.setitem(sys.modules, "paper_2512_16483_b200._calls", None)       # its import fails
    assert schedule.rank_from_keep_ratio(169, 0.5) == 85
    assert hasattr(binding.load_library(), "fvar_scale_step")
    with pytest.raises(ImportError) as e:
        binding._native()
    assert str(e.value.__cause__) in str(e.value) and "torch" in str(e.value)
    monkeypatch.setattr(fbuild, "CALLS", fbuild.CALLS + ".missing")
    with pytest.raises(FileNotFoundError, match="not built"):
        binding._native()


def test_call_layer_of_another_torch_is_stale(monkeypatch):
    """After torch or Python is replaced the sources are no newer than the call layer, which has to be built anew all the same."""
    fbuild.build()
    assert not fbuild._calls_stale() and not fbuild._lib_stale()
    assert fbuild.calls_built_for() == fbuild._built_for()
    built = []
    monkeypatch.setattr(fbuild, "_built_for", lambda: "fvar call layer for torch 0.0, Python 0.0")
    monkeypatch.setattr(fbuild, "_compile_calls", lambda: built.append("calls"))
    monkeypatch.setattr(fbuild, "_build_lib", lambda: built.append("library"))
    fbuild.build()
    assert built == ["calls"]


def test_workspace_bytes_and_bad_shapes_without_gpu():
    import ctypes as ct
    from paper_2512_16483_b200 import binding
    lib = binding.load_library()
    hw = (ct.c_int * 4)(2, 2, 3, 3)
    cfg = binding._Cfg(2, 1, 128, 2, 64, 256, 2, ct.cast(hw, ct.POINTER(ct.c_int)), 2, 0, 0, 0, 1e-6)
    n = lib.fvar_workspace_bytes(ct.byref(cfg))
    assert n > 0 and n % 1024 == 0
    cfg.head_dim = 32                                    # unsupported head size
    assert lib.fvar_workspace_bytes(ct.byref(cfg)) == 0
    cfg.head_dim, cfg.blocks_per_group = 64, 3           # 2 blocks do not split into groups of 3
    assert lib.fvar_workspace_bytes(ct.byref(cfg)) == 0
    ctx = ct.c_void_p(None)
    w = binding._Weights()
    st = lib.fvar_init(ct.byref(w), ct.byref(cfg), None, 0, None, ct.byref(ctx))
    assert st == binding.EINVAL and not ctx.value
    assert b"shape" in lib.fvar_last_error(None)
    assert lib.fvar_kv_append(None, 0) == binding.EINVAL


@pytest.mark.parametrize("call,args,vary", [
    ("fvar_row_scores", (64, 1, 4, 8, 64, None), {0: 16}),
    ("fvar_row_keys", (64, 64, 1, 4, 8, 64, None), {0: 16}),
    ("fvar_ln_modulate", (64, 4, 8, 4, 64, 64, 8, 1e-6, 64, None), {0: 16, 4: 16, 5: 16, 8: 8}),
    ("fvar_gemm_bf16", (64, 64, 64, 4, 64, 8, 64, None), {2: 16, 6: 16}),
    ("fvar_gemm_bf16_form", (64, 64, 64, 4, 8, 8, 3, 0, 64, None), {2: 16, 8: 16}),
    ("fvar_gemm_bf16_wt", (64, 64, 64, 4, 64, 8, 0, 64, None), {2: 16, 7: 16}),
    ("fvar_attention", (64, 64, 64, 1, 1, 4, 64, 4, 8, 64, None), {9: 16}),
    ("fvar_cfg_combine", (64, 2, 8, 1.0, 64, None), {0: 16, 4: 16}),
    ("fvar_rtr_fill", (64, 1, 2, 2, 4, 4, 8, 64, 64, None), {0: 16, 8: 16}),
    ("fvar_select_rows_static", (64, 1, 4, 8, 2, 64, 64, None), {0: 16}),
])
def test_kernel_calls_refuse_addresses_off_their_vector_grid(call, args, vary):
    """The kernels move 8 or 16 bytes at a time; a buffer off that grid has to come back as FVAR_EINVAL, before anything
    is launched.  (The addresses here are numbers, not memory: only refused calls are made.)"""
    from paper_2512_16483_b200 import binding
    fn = getattr(binding.load_library(), call)
    for pos, grid in vary.items():
        for off in (2, 4, 8):
            if off % grid:
                bad = list(args)
                bad[pos] += off
                assert fn(*bad) == binding.EINVAL, (call, pos, off)
                assert b"aligned" in binding.load_library().fvar_last_error(None) or call == "fvar_cfg_combine"
    if call == "fvar_ln_modulate":                       # rows of shift and scale off the grid
        assert fn(*args[:6], 6, *args[7:]) == binding.EINVAL


@pytest.mark.parametrize("C,F", [(1024, 4096), (1920, 7680), (2048, 8192)])
def test_free_width_tiles_make_no_more_chunks_than_they_have_to(C, F):
    """A tile of 16 more rows than a multiple of 32 is taken where it makes no more chunks than the next multiple of 32;
    208, the widest with six pipeline stages, and 176 over short sums may.  Pairs of 128 features are faster than 112 rows."""
    from helpers import PLAN_FLEX, PLAN_PAIR, gemm_plan
    for N, K in ((3 * C, C), (C, C), (F, C), (C, F)):
        for R in list(range(33, 1100)) + list(range(1100, 8193, 7)) + [2048, 4096]:
            form, w = gemm_plan(R, N, K)
            if form == PLAN_FLEX:
                assert w % 16 == 0 and 64 <= w <= 256
                if w % 32 and not (w == 208 or (w == 176 and K <= 2048)):
                    assert -(-R // w) == -(-R // (w + 16)), (R, N, K, w)
                if w == 112:                         # where pairs of 128 features would need another round of the chip
                    assert -(-R // 256) * -(-N // 128) > 74 >= -(-R // w) * -(-N // 256), (R, N, K)
    for R in (2048, 4096):                           # full pairs of 256 rows
        assert gemm_plan(R, 2048, 2048)[0] == PLAN_PAIR and gemm_plan(R, 2048, 8192)[0] == PLAN_PAIR


def test_schedule_matches_printed_table():
    rows = []
    with open(os.path.join(ROOT, "tests", "golden", "rank_ratio_alpha096.txt")) as f:
        for line in f:
            if line.strip() and not line.startswith("#"):
                rows.append(tuple(float(v) for v in line.split()))
    assert tuple(rows) == schedule.rank_ratio_table()
    assert schedule.infinity_group_ranks(40) == [26, 218, 336, 400, 410, 317, 251, 306]
    assert schedule.infinity_group_ranks(64) == [16, 111, 170, 135, 115, 59, 78, 113]
    assert schedule.infinity_stage_modes(True) == [0] * 10 + [1, 2, 2]
    assert schedule.infinity_stage_modes(False) == [0] * 10 + [1, 1, 1]
    assert schedule.cache_rows(si.INFINITY_SCALES)[-1] == 10521 and schedule.cache_rows(si.VAR_SCALES)[-1] == 680
    assert schedule.rank_from_keep_ratio(169, 0.5) == 85 and schedule.rank_from_keep_ratio(100, 0.001) == 1
    assert schedule.infinity_schedule(True)[0] == list(si.INFINITY_SCALES)
    assert schedule.rank_from_table_ratio(1600, 2048, 0.016) == 26 and schedule.rank_from_table_ratio(4096, 2048, 0.083) == 170
    assert schedule.infinity_group_ranks(48, 2048, 4) == [schedule.infinity_group_ranks(48)[c] for c in (1, 3, 5, 7)]


def test_bf16_rounding_of_the_input_generator():
    x = np.array([1.0, 1.00390625, 1.005859375, -2.5, 3.0e38, 1e-40], dtype=np.float32)
    r = si.round_to_bf16(x)
    assert r[0] == 1.0 and r[1] == 1.0 and r[2] == np.float32(1.0078125)     # ties to even, then up
    assert np.all((r.view(np.uint32) & 0xFFFF) == 0)
    assert np.array_equal(si.bf16_bits_to_f32(si.bf16_bits(r)), r)
