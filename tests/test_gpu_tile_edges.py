"""Key ranges that end inside a key tile, with far higher scores just past the
end: the tile holds rows of the next request there, and none of them may enter
the row maximum (which the kernels take from the loads of whole 32-column
chunks).  A maximum that included one would exceed the row's own by more than
2^100 and every visible weight would vanish.  Bars as in the parity tests."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from paper_2608_21229_gb300 import refcache as rcb

import parity_utils as pu
import test_gpu_fp8 as fp8

pytestmark = pytest.mark.gpu

#: (live keys, reference keys) of the first request: below, at and above the
#: edges of 32-column chunks and of 128- and 192-key tiles
LENGTHS = [(1, 193), (31, 192), (32, 191), (33, 129), (96, 97), (127, 128), (128, 127), (129, 33), (191, 32), (192, 31), (193, 1)]
GAIN = 30.0  # the second request's keys: its scores have 30 times the first's spread


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    rcb.load()
    oracle.build()
    yield
    rcb.set_kernel("tcgen05")


def _workload(n_x, n_r, head_dim):
    w = workloads.Workload(f"edges_{n_x}_{n_r}", 2, head_dim,
                           (workloads.Request(0, 0, n_x, n_r), workloads.Request(0, 0, 200, 200)), 31)
    static, live = list(workloads.static_qkv(w)), list(workloads.live_qkv(w))
    for t, first in ((static[1], n_r), (live[1], n_x)):
        t[first:] = (t[first:].float() * GAIN).to(torch.bfloat16)
    return w, tuple(static), tuple(live)


@pytest.mark.parametrize("kernel", ["tcgen05", "tcgen05_k128"])
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("lengths", LENGTHS, ids=str)
def test_keys_past_the_end_do_not_enter_the_maximum(kernel, head_dim, lengths):
    w, static, live = _workload(*lengths, head_dim)
    pu.full_compare(pu.GpuRun(w, kernel=kernel, static=static, live=live))


@pytest.mark.parametrize("lengths", LENGTHS, ids=str)
def test_keys_past_the_end_do_not_enter_the_maximum_e4m3(monkeypatch, lengths):
    w, static, live = _workload(*lengths, 128)
    rcb.set_kernel("tcgen05")
    monkeypatch.setattr(workloads, "live_qkv", lambda *a, **k: live)
    fp8.check_step(fp8.Fp8Run(w, static=static), np.arange(2), statistical=False)


#: items of one to four key tiles after one another (an item's first S is issued
#: inside the item before it, whose last tiles it follows), repeated so that the
#: ring of items wraps several times on every CTA pair
SHORT = [(1, 1), (200, 1), (64, 300), (193, 5), (17, 130), (400, 385), (5, 64), (256, 190), (130, 500), (3, 2)]


@pytest.mark.parametrize("kernel", ["tcgen05", "tcgen05_k128"])
@pytest.mark.parametrize("head_dim", [64, 128])
def test_short_items_after_one_another(kernel, head_dim):
    reqs = tuple(workloads.Request(i % 3, 0, *SHORT[i % len(SHORT)]) for i in range(90))
    pu.full_compare(pu.GpuRun(workloads.Workload("short_items", 7, head_dim, reqs, 32), kernel=kernel))


def test_short_items_after_one_another_e4m3():
    reqs = tuple(workloads.Request(i % 3, 0, *SHORT[i % len(SHORT)]) for i in range(60))
    rcb.set_kernel("tcgen05")
    fp8.check_step(fp8.Fp8Run(workloads.Workload("short_items_fp8", 7, 128, reqs, 33)), np.arange(7), rows_per_request=8,
                   statistical=False)


@pytest.mark.parametrize("head_dim", [64, 128])
def test_short_items_in_static_order(head_dim):
    """full_attention_noalloc hands items out in a fixed order: the same bytes as the work counter's."""
    cu = np.concatenate([[0], np.cumsum([1 + (i * 37) % 420 for i in range(120)])]).tolist()
    q, k, v = (torch.randn(cu[-1], 5, head_dim, device="cuda", generator=torch.Generator("cuda").manual_seed(s)).to(torch.bfloat16)
               for s in (1, 2, 3))
    outs = []
    for call in (rcb.full_attention, rcb.full_attention_noalloc):
        o, lse = torch.empty_like(q), torch.empty(cu[-1], 5, device="cuda")
        call(cu, q, k, v, o, lse)
        assert rcb.status() == rcb.OK, rcb.last_error()
        outs.append((o, lse))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


@pytest.mark.parametrize("batch", [1, 31, 32, 33])
def test_full_attention_lists(batch):
    """Work lists that travel as a kernel parameter (up to 32 requests, empty ones not counted) and in memory:
    the same bytes as full_attention_noalloc's, whose list is in memory."""
    lens = [0 if i % 5 == 3 else 1 + (i * 97) % 700 for i in range(batch)] + [0, 0]
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    q, k, v = (torch.randn(cu[-1], 3, 128, device="cuda", generator=torch.Generator("cuda").manual_seed(s)).to(torch.bfloat16)
               for s in (4, 5, 6))
    outs = []
    for call in (rcb.full_attention, rcb.full_attention, rcb.full_attention_noalloc):  # two in a row: the counter is reset
        o, lse = torch.full_like(q, float("nan")), torch.full((cu[-1], 3), float("nan"), device="cuda")
        call(cu, q, k, v, o, lse)
        outs.append((o, lse))
    assert rcb.status() == rcb.OK, rcb.last_error()
    for o, lse in outs[:2]:
        assert torch.equal(o, outs[2][0]) and torch.equal(lse, outs[2][1])


#: cached rows of a request at the edges of the cache write's groups of eight rows
#: and of its 128-row tiles
ROWS = (1, 7, 8, 9, 63, 64, 65, 120, 121, 127, 128, 129, 249, 256)


@pytest.mark.parametrize("heads", [1, 5])
@pytest.mark.parametrize("mode", ["beyond", "beyond_alt"])
def test_e4m3_cache_write_at_the_edges_of_row_groups(mode, heads):
    reqs = tuple(workloads.Request(i % 2, 0, 1, n) for i, n in enumerate(ROWS))
    w = workloads.Workload("quant_edges", heads, 128, reqs, 35)
    static = list(workloads.static_qkv(w))
    for i, t in enumerate(static[1:]):  # columns of one head at other scales, one tile of zeros
        t[:, 0, 8 * i:8 * i + 3] *= 300.0
        t[w.cu_static[3]:w.cu_static[4]] = 0
    rcb.set_kernel("tcgen05")
    fp8.check_cache(fp8.Fp8Run(w, mode=mode, static=tuple(static)), np.arange(heads))


@pytest.mark.parametrize("batch", [1, 2, 31, 32, 33, 34, 1024, 1025, 1100])
def test_cache_write_finds_the_segment_of_every_piece(batch):
    """The bf16 cache write of many requests, some without cached rows: the slots hold the rows' bytes."""
    heads, dim = 3, 64  # rows of 384 bytes: segments of one piece, and of several with a short last one
    lens = [0 if i % 7 == 5 else 1 + (i * 53) % 29 for i in range(batch)]
    reqs = tuple(workloads.Request(i % 2, 0, 1, n) for i, n in enumerate(lens))
    w = workloads.Workload("segments", heads, dim, reqs, 36)
    seg = rcb.Segments.from_workload(w)
    cache = rcb.RefCache(seg)
    for t in cache.kv(0):
        t.fill_(float("nan"))
    q, k, v = (torch.randn(seg.static_rows, heads, dim, device="cuda", generator=torch.Generator("cuda").manual_seed(s)).to(torch.bfloat16)
               for s in (7, 8, 9))
    cache.build(0, q, k, v, torch.empty_like(q))
    assert rcb.status() == rcb.OK, rcb.last_error()
    rows = np.concatenate([np.arange(s + r.n_st, s + r.n_static) for s, r in zip(w.cu_static, reqs)])
    rows = torch.from_numpy(rows).cuda()
    for slot, t in zip(cache.kv(0), (k, v)):
        assert torch.equal(slot.view(torch.int16), t[rows].view(torch.int16))
