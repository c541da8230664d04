"""Steps with split items (parts through the workspace, merged behind the
attention kernel), both head dims and cache types, both forms of the merge, two
to eight parts and tasks that end inside the merge's blocks of 32 rows: the
outputs against the oracle, and guard bytes around them."""
import math

import numpy as np
import pytest
import torch

import oracle
import workloads
from paper_2608_21229_gb300 import refcache as rcb

import parity_utils as pu
import split_workloads
import test_gpu_fp8 as fp8
from test_gpu_canary import Guarded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    rcb.load()
    oracle.build()
    rcb.set_kernel("tcgen05")
    yield
    rcb.set_kernel("tcgen05")


def _guarded_step(cache, live):
    """One step into guarded buffers: (O, LSE)."""
    seg = cache.seg
    o = Guarded((seg.live_rows, seg.num_heads, seg.head_dim), torch.bfloat16)
    lse = Guarded((seg.live_rows, seg.num_heads), torch.float32)
    cache.step(0, *live, o.t, lse.t)
    torch.cuda.synchronize()
    assert rcb.status() == rcb.OK, rcb.last_error()
    o.check("O")
    lse.check("LSE")
    return o.t, lse.t


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("case", range(len(split_workloads.NAMES)), ids=split_workloads.NAMES)
def test_split_step(case, dim):
    w = split_workloads.cases(dim)[case][0]
    static, live = workloads.static_qkv(w), workloads.live_qkv(w)
    cache = rcb.RefCache(rcb.Segments.from_workload(w))
    assert cache.launches("step") == 2  # the attention and the merge
    cache.build(0, *(t.cuda() for t in static), torch.empty_like(static[0], device="cuda"))
    o, lse = _guarded_step(cache, [t.cuda() for t in live])
    o, lse = pu.f64(o), pu.f64(lse)
    rng = np.random.default_rng(case)
    for b, r in enumerate(w.requests):
        pairs = None
        if w.num_heads > 12:  # every row, of three heads each
            pairs = np.array([(i, h) for i in range(r.n_live) for h in rng.integers(0, w.num_heads, 3)], np.int32)
        ref_o, ref_l = pu.oracle_live_request(w, "beyond", b, static, live, 1.0 / math.sqrt(dim), pairs)
        g_o, g_l = o[w.cu_live[b]:w.cu_live[b] + r.n_live], lse[w.cu_live[b]:w.cu_live[b] + r.n_live]
        if pairs is not None:
            g_o, g_l = g_o[pairs[:, 0], pairs[:, 1]], g_l[pairs[:, 0], pairs[:, 1]]
        pu.check_close(g_o, ref_o, g_l, ref_l, f"request {b}")


@pytest.mark.parametrize("case", range(len(split_workloads.NAMES)), ids=split_workloads.NAMES)
def test_split_step_e4m3(case):
    w = split_workloads.cases(128)[case][0]
    run = fp8.Fp8Run(w)
    assert run.cache.launches("step") == 2
    o, lse = _guarded_step(run.cache, [t.cuda() for t in run.live])
    assert torch.equal(o.cpu().view(torch.int16), run.o_live.cpu().view(torch.int16))
    assert torch.equal(lse.cpu().view(torch.int32), run.lse_live.cpu().view(torch.int32))
    heads = list(range(w.num_heads)) if w.num_heads <= 12 else [0, 1, 21, 43]
    fp8.check_step(run, heads=heads, rows_per_request=48, seed=case)
