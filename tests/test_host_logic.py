"""Host logic: the accounting the benchmark reports against the App. C model,
the seeded input generators, and the binding's views of the cache."""
import contextlib

import pytest
import torch

import workloads
from oracle import cost_model as cm
from paper_2608_21229_gb300 import accounting as acc
from paper_2608_21229_gb300 import refcache as rcb


@pytest.mark.parametrize("w", [workloads.TINY, workloads.EDIT_512_2REF, workloads.EDIT_1024_5REF]
                         + list(workloads.SWEEP_1024), ids=lambda w: w.name)
def test_accounting_equals_app_c_model(w):
    r = w.requests[0]
    s = r.n_lt + r.n_x
    assert acc.prefill_units(w.requests) == cm.c_pre(r.n_r, r.n_st)
    assert acc.step_units(w.requests) == cm.c_step(r.n_r, s)
    assert 40 * acc.full_units(w.requests) == cm.c_full(r.n_r, s, 40)
    assert acc.modelled_ratio(w.requests, 40) == pytest.approx(cm.speedup(r.n_r, r.n_st, s, 40), rel=1e-12)
    assert acc.flops(1, 24, 128) == cm.flops_per_unit(128) * 24
    assert acc.prefill_units(w.requests) - acc.prefill_units(
        [workloads.Request(0, r.n_lt, r.n_x, r.n_r)]) == cm.anchor_overhead(r.n_r, r.n_st)


def test_headline_step_flops():
    w = workloads.EDIT_1024_5REF
    f = acc.flops(acc.step_units(w.requests), w.num_heads, w.head_dim)
    assert f == 4 * 128 * 24 * 4608 * (4608 + 20480)
    assert acc.cache_bytes(w.requests, 24, 128) == 2 * 20480 * 24 * 128 * 2


def test_generators_are_deterministic_and_distinct():
    a = workloads.randn_bf16((64, 2, 8), 0, "x")
    b = workloads.randn_bf16((64, 2, 8), 0, "x")
    c = workloads.randn_bf16((64, 2, 8), 0, "y")
    assert a.dtype == torch.bfloat16 and torch.equal(a, b) and not torch.equal(a, c)
    assert abs(float(workloads.randn_bf16((4096, 64), 1, "z").float().std()) - 1.0) < 0.02


def test_workload_shapes():
    w = workloads.RAGGED_4REQ
    assert w.batch == 4 and [r.n_r // 1024 if r.n_x == 1024 else r.n_r // 4096 for r in w.requests] == [1, 3, 5, 8]
    assert w.cu_live[-1] == sum(r.n_lt + r.n_x for r in w.requests)
    q, k, v = workloads.static_qkv(workloads.TINY)
    assert q.shape == (288, 4, 64)


def test_bench_clock_ceilings():
    """The bench line's two clock-based figures: the tensor pipe's ceiling
    (8192 dense bf16 FLOPs per clock per SM) and the exponential floor (one
    ex2 per visible pair at a given rate per clock per SM), at a given clock."""
    import bench

    n = bench.nominal_at_clock(1000.0, 2000.0, 152)
    assert n["tflops"] == pytest.approx(8192 * 152 * 2.0e9 / 1e12) and n["frac"] == pytest.approx(1000.0 / n["tflops"])
    assert bench.nominal_at_clock(1000.0, None, 152) is None
    w = workloads.EDIT_1024_5REF
    exps = acc.step_units(w.requests) * w.num_heads
    f = bench.exp_floor(exps, 1e-3, 2000.0, 152, 32.0)
    assert f["floor_ms"] == pytest.approx(exps / (32 * 152 * 2.0e9) * 1e3)
    assert f["frac_of_step"] == pytest.approx(f["floor_ms"] / 1.0)
    assert bench.exp_floor(exps, 1e-3, 2000.0, 152, 16.0)["floor_ms"] == pytest.approx(2 * f["floor_ms"])
    assert bench.exp_floor(exps, 1e-3, None, 152, 32.0) is None


def test_guard_report_finds_planted_writes():
    """The canary check of tests/test_gpu_canary.py: bytes changed in either
    guard and elements left unwritten are counted (planted on the CPU)."""
    import numpy as np
    import parity_utils as pu

    g, n, pat = 64, 40, 0xA5
    full = np.full(g + n + g, pat, dtype=np.uint8)
    full[g:g + n] = 1                      # every element written
    assert pu.guard_report(full, g, n, 4, pat) == (0, 0, 0)
    full[g - 1] = 0                        # one byte before the buffer
    full[g + n + 5] = 7                    # and one after
    full[g + 8:g + 12] = pat               # one 4-byte element never written
    assert pu.guard_report(full, g, n, 4, pat) == (1, 1, 1)
    full[g + 12] = pat                     # a partly matching element is written
    assert pu.guard_report(full, g, n, 4, pat)[2] == 1
    assert pu.guard_report(full, g, n, 2, pat)[2] == 2


class _KvLibrary:
    """refcache_kv_ptr of a cache of 3 layers with 5 rows, 2 heads of 64, 256 bytes into its memory."""

    def __init__(self, base):
        self.base = base

    def refcache_kv_ptr(self, h, layer, k, v, rows):
        if h is None or not 0 <= layer < 3:
            return rcb.ERR_INVALID_ARG
        n = 5 * 2 * 64 * 2
        k._obj.value, v._obj.value, rows._obj.value = self.base + 256 + 2 * n * layer, self.base + 256 + 2 * n * layer + n, 5
        return rcb.OK

    def refcache_last_error(self, buf, n):
        return 0

    def refcache_destroy(self, h):
        pass


@pytest.mark.parametrize("use", [contextlib.nullcontext, torch.no_grad, torch.inference_mode])
@pytest.mark.parametrize("first", [contextlib.nullcontext, torch.no_grad, torch.inference_mode])
def test_slot_views_can_be_written_whatever_mode_they_were_first_asked_for_in(monkeypatch, first, use):
    c = rcb.RefCache.__new__(rcb.RefCache)
    c.seg, c.num_layers, c.h = rcb.Segments(2, 64, [0, 1], [0, 5], [0]), 3, rcb.ctypes.c_void_p(1)
    c.mem = torch.zeros(256 + 3 * 2 * 1280, dtype=torch.uint8)
    monkeypatch.setattr(rcb, "load", lambda: _KvLibrary(c.mem.data_ptr()))
    try:
        with first():
            c.kv(1)
        x = torch.arange(5 * 2 * 64).view(5, 2, 64).to(torch.bfloat16)
        with use():
            for layer in (2, 0, 1, 2):
                for i, slot in enumerate(c.kv(layer)):
                    assert slot.shape == (5, 2, 64) and slot.data_ptr() == c.mem.data_ptr() + 256 + 1280 * (2 * layer + i)
                    slot.copy_((x + layer + i).requires_grad_())
                    assert torch.equal(c.kv(layer)[i], x + layer + i)
        for bad in (-1, 3):
            with pytest.raises(rcb.RefCacheError):
                c.kv(bad)
    finally:
        c.h = None  # closed (and nothing for the library to free)
    with pytest.raises(rcb.RefCacheError):
        c.kv(0)
