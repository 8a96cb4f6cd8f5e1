"""Host-only checks of the C-ABI boundary: the library loads, exports every symbol the
header declares, struct layouts agree, and host-detectable errors return a status before
any CUDA work (so these run without a GPU)."""
import ctypes
import os
import re

import pytest
import torch

from paper_2609_34814_b200 import binding as wb
from paper_2609_34814_b200 import build as wbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    wbuild.build()
    return wb.load()


def test_exports_match_header(lib):
    header = open(os.path.join(ROOT, "include", "waveal.h")).read()
    declared = set(re.findall(r"\b(waveal_[a-z0-9_]+)\s*\(", header))
    assert declared == set(wb.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), name


def test_struct_layouts():
    assert ctypes.sizeof(wb.PlanDesc) == 80
    assert ctypes.sizeof(wb.PlanOut) == 64
    assert ctypes.sizeof(wb.AttnDesc) == 96
    assert wb.PlanDesc.seed.offset == 24 and wb.PlanDesc.min_nnz.offset == 72
    assert wb.AttnDesc.q_stride.offset == 24 and wb.AttnDesc.order_heads_interleaved.offset == 88


def test_defaults_and_workspace_query(lib):
    d = wb.plan_desc_default()
    assert (d.svd_iters, d.mode, d.l2_fit_num, d.l2_fit_den, d.min_density_ppm, d.local_num, d.local_den) == \
        (5, wb.AUTO, 9, 16, 10000, 1, 2)
    with pytest.raises(wb.WavealError) as e:
        wb.plan_workspace_bytes(d)                       # heads etc. still 0
    assert e.value.status == wb.ERR_INVALID_ARG and "positive" in str(e.value)
    d.heads, d.n_q_blocks, d.n_kv_blocks = 2, 100, 130
    n = wb.plan_workspace_bytes(d)
    assert n >= 2 * 100 * 3 * 8 + 2 * 130 * 2 * 8
    d.n_q_blocks = 1 << 20
    with pytest.raises(wb.WavealError) as e:
        wb.plan_workspace_bytes(d)
    assert e.value.status == wb.ERR_UNSUPPORTED
    d.n_q_blocks, d.mode = 100, 9
    with pytest.raises(wb.WavealError):
        wb.plan_workspace_bytes(d)
    for mode in (9 | wb.PLAN_CLEAR_STATUS, 64, -1):
        d.mode = mode
        with pytest.raises(wb.WavealError):
            wb.plan_workspace_bytes(d)
    d.mode = wb.STAGE1_ONLY | wb.PLAN_CLEAR_STATUS
    assert wb.plan_workspace_bytes(d) == n
    assert lib.waveal_plan_csr(ctypes.byref(d), 0x1000, 0x2000, 0x3000, n, ctypes.byref(wb.PlanOut(row_order=0x4000)),
                               None) == wb.ERR_INVALID_ARG and "mode" in wb.last_error()


def test_plan_host_errors_before_any_launch(lib):
    d = wb.plan_desc_default(heads=1, n_q_blocks=4, n_kv_blocks=4)
    out = wb.PlanOut()
    assert lib.waveal_plan_bitmap(ctypes.byref(d), None, None, 0, ctypes.byref(out), None) == wb.ERR_INVALID_ARG
    assert lib.waveal_plan_bitmap(ctypes.byref(d), 0x1000, 0x2000, 1 << 20, ctypes.byref(out), None) == wb.ERR_INVALID_ARG
    assert "row_order" in wb.last_error()
    out.row_order = 0x3000
    assert lib.waveal_plan_bitmap(ctypes.byref(d), 0x1000, 0x2000, 16, ctypes.byref(out), None) == wb.ERR_WORKSPACE
    assert lib.waveal_plan_bitmap(ctypes.byref(d), 0x1000, 0x2010, 1 << 20, ctypes.byref(out), None) == wb.ERR_INVALID_ARG
    assert lib.waveal_plan_csr(ctypes.byref(d), None, None, 0x2000, 1 << 20, ctypes.byref(out), None) == wb.ERR_INVALID_ARG
    assert lib.waveal_bitmap_to_csr(0, 4, 4, 0x1000, 0x2000, None, 0, 0x3000, 64, None) == wb.ERR_INVALID_ARG
    assert lib.waveal_bitmap_to_csr(1, 4, 4, 0x1000, 0x2000, None, 0, 0x3000, 4, None) == wb.ERR_WORKSPACE


def test_attention_host_errors_before_any_launch(lib):
    d = wb.AttnDesc()
    d.heads, d.seq_q, d.seq_kv, d.head_dim, d.block_q, d.block_kv = 2, 256, 256, 128, 128, 128
    for s in (d.q_stride, d.k_stride, d.v_stride, d.o_stride):
        s[0], s[1] = 256 * 128, 128
    n = ctypes.c_size_t()
    assert lib.waveal_bsattn_workspace_bytes(ctypes.byref(d), ctypes.byref(n)) == wb.OK
    assert n.value == 256                                # counters + 8 + 32 bytes per (head, query block), in units of 256
    d.heads, d.seq_q = 40, 75600
    assert lib.waveal_bsattn_workspace_bytes(ctypes.byref(d), ctypes.byref(n)) == wb.OK
    tasks = 40 * 591
    assert n.value == ((32 + 8 * tasks + 31) // 32 * 32 + 32 * tasks + 255) // 256 * 256
    d.heads, d.seq_q = 2, 256
    call = lambda q=0x1000, ws=0x9000, wsb=256, scale=0.0: lib.waveal_bsattn_fwd(
        ctypes.byref(d), q, 0x2000, 0x3000, 0x4000, None, 0x5000, 0x6000, None, ctypes.c_float(scale), ws, wsb,
        None, None)
    assert call(q=None) == wb.ERR_INVALID_ARG
    assert call(q=0x1004) == wb.ERR_INVALID_ARG and "aligned" in wb.last_error()
    assert call(ws=None) == wb.ERR_WORKSPACE
    assert call(wsb=8) == wb.ERR_WORKSPACE
    assert call(scale=float("nan")) == wb.ERR_INVALID_ARG
    d.head_dim = 96
    assert call() == wb.ERR_UNSUPPORTED
    d.head_dim, d.block_q = 128, 64
    assert call() == wb.ERR_UNSUPPORTED                  # block_q != block_kv
    d.block_q = 128
    d.q_stride[1] = 100
    assert call() == wb.ERR_INVALID_ARG
    assert wb.status_string(wb.ERR_TIMEOUT) == "device-side wait timed out"


@pytest.mark.parametrize("lists", [False, True])
def test_a_plan_s_status_words_are_cleared_by_the_call(monkeypatch, lists):
    """Not when they are first looked at: that could be inside a graph capture or on another stream."""
    handed, modes = [], []

    class Lib:
        def waveal_plan_bitmap(self, desc, bits, ws, n, out, stream):
            handed.append(out._obj.dev_status)
            modes.append(desc._obj.mode)
            if desc._obj.mode & wb.PLAN_CLEAR_STATUS:
                ctypes.memset(out._obj.dev_status, 0, 16)
            return wb.OK

        def waveal_plan_csr(self, desc, ptr, idx, ws, n, out, stream):
            handed.append(out._obj.dev_status)
            return wb.OK

    monkeypatch.setattr(wb, "load", lambda: Lib())
    monkeypatch.setattr(wb, "_stream", lambda s: None)
    desc = wb.PlanDesc(heads=3, n_q_blocks=5, n_kv_blocks=70, mode=wb.STAGE2_ONLY | wb.RING_CUT_LARGEST_GAP)
    ws = torch.empty((64,), dtype=torch.uint8)
    if lists:
        res = wb.plan_csr(desc, torch.zeros((16,), dtype=torch.int32), torch.zeros((1,), dtype=torch.int32), workspace=ws)
    else:
        res = wb.plan_bitmap(desc, torch.zeros((3, 5, 2), dtype=torch.int64), workspace=ws)
    assert handed[0] is not None and ctypes.string_at(handed[0], 16) == bytes(16)          # (before anyone looks)
    assert res.dev_status.tolist() == [0] * 4 and res.dev_status.dtype == torch.int32
    assert handed == [res.dev_status.data_ptr()] and desc.mode == wb.STAGE2_ONLY | wb.RING_CUT_LARGEST_GAP
    assert modes == ([] if lists else [desc.mode | wb.PLAN_CLEAR_STATUS])
    for name in ("row_order", "row_nnz", "skip_flags"):      # (they share an allocation)
        getattr(res, name).fill_(77)
    assert res.dev_status.tolist() == [0] * 4 and (res.row_order == 77).all() and (res.row_nnz == 77).all()


def test_missing_library_fails_loudly(monkeypatch, tmp_path):
    monkeypatch.setattr(wb, "_lib", None)
    monkeypatch.setattr(wb, "LIB_PATH", str(tmp_path / "nope.so"))
    with pytest.raises(RuntimeError, match="no CPU fallback"):
        wb.load()


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("heads,seq_q", [(1, 64), (1, 20000), (8, 20480), (32, 98304), (40, 75600)])
def test_attention_workspace_is_the_sum_of_its_listed_parts(lib, block, heads, seq_q):
    d = wb.AttnDesc(heads=heads, seq_q=seq_q, seq_kv=seq_q, head_dim=128, block_q=block, block_kv=block)
    for name in ("q_stride", "k_stride", "v_stride", "o_stride"):
        getattr(d, name)[0], getattr(d, name)[1] = seq_q * 128, 128
    tasks = heads * -(-seq_q // block)
    assert wb.bsattn_workspace_bytes(d) == -(-(-(-(32 + 8 * tasks) // 32) * 32 + 32 * tasks) // 256) * 256
