"""The library's host side without a GPU: its CUDA runtime calls go to
host-memory stand-ins (tests/c/host_cudart.c), in a child process."""
import json
import os
import subprocess
import sys

import pytest

from paper_2608_21229_gb300 import build as cbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, json, sys
sys.path.insert(0, {root!r})
from paper_2608_21229_gb300 import refcache as rc
cudart = ctypes.CDLL(None)
cudart.host_cudart_calls.restype = ctypes.c_char_p
cudart.host_cudart_live.restype = ctypes.c_longlong
cudart.host_cudart_list.restype = cudart.host_cudart_copy_dst.restype = ctypes.c_void_p
cudart.host_cudart_copy_bytes.restype = ctypes.c_size_t
L = rc.load()


def segments(heads, dim, reqs):
    # reqs: (anchor, instruction, target, reference) rows of each request
    cu_l, cu_s = [0], [0]
    for n_st, n_lt, n_x, n_r in reqs:
        cu_l.append(cu_l[-1] + n_lt + n_x)
        cu_s.append(cu_s[-1] + n_st + n_r)
    return rc.Segments(heads, dim, cu_l, cu_s, [r[0] for r in reqs], [r[1] for r in reqs])


def create(heads, dim, reqs, flags=0, fail_at=-1):
    seg, h = segments(heads, dim, reqs), ctypes.c_void_p()
    cudart.host_cudart_reset(fail_at)
    code = L.refcache_create(ctypes.byref(h), 1, flags, ctypes.byref(seg.c), None, 0)
    out = dict(code=code, calls=cudart.host_cudart_calls().decode(), live=cudart.host_cudart_live())
    if code == 0:
        out["step_launches"] = L.refcache_call_launches(h, 1)
        # after the memset: the build's items, the step's, its merge jobs, the in-slot build's tasks, each if there are any
        lists = []
        for i in range(out["calls"].index("s") + 1, out["calls"].rindex("m") + 1):
            words = (ctypes.c_int32 * (cudart.host_cudart_copy_bytes(i) // 4)).from_address(cudart.host_cudart_copy_dst(i))
            lists.append([list(words[k:k + 8]) for k in range(0, len(words), 8)])
        if out["step_launches"] == 2:
            out["jobs"] = lists.pop(2)  # q_row0, q_rows, head, part0, nparts
        out["tasks"] = sum(lists, [])  # q_row0, q_rows, a_row0, a_len, b_row0, b_len, head, part
        L.refcache_destroy(h)
    out["live_after"] = cudart.host_cudart_live()
    return out


{body}
"""


@pytest.fixture(scope="module")
def run_child(tmp_path_factory):
    shim = str(tmp_path_factory.mktemp("cudart") / "host_cudart.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", shim, os.path.join(ROOT, "tests", "c", "host_cudart.c")],
                   check=True)
    cbuild.build()

    def run(body):
        r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, body=body)], capture_output=True, text=True,
                           timeout=300, env=dict(os.environ, LD_PRELOAD=shim))
        assert r.returncode == 0, r.stderr
        return json.loads(r.stdout.splitlines()[-1])

    return run


@pytest.mark.parametrize("flags", [0, 0x100])
def test_create_returns_only_after_its_lists_are_on_the_device(run_child, flags):
    """A host-to-device copy from pageable memory may return before it has
    reached the device, and a non-blocking stream is not ordered behind it: a
    launch reads its work list before it waits for anything, so the device is
    synchronised after the last upload."""
    out = run_child(f"print(json.dumps(create(24, 128, [(64, 256, 1024, 20480)], {flags})))")
    assert out["code"] == 0 and out["live_after"] == 0
    calls = out["calls"]
    last = max(calls.rindex("m"), calls.rindex("s"))
    assert "d" in calls[last:], calls


def test_create_gives_back_its_memory_when_a_call_fails(run_child):
    out = run_child("""
ok = create(24, 128, [(64, 256, 1024, 20480)])
print(json.dumps([create(24, 128, [(64, 256, 1024, 20480)], 0, i) for i in range(len(ok["calls"].rstrip("d")) + 1)]))""")
    assert len(out) >= 5
    for r in out:
        assert r["code"] != 0 and r["live_after"] == 0, r


@pytest.mark.parametrize("dim", [64, 128])
def test_lists_that_are_read_early_lie_in_the_librarys_own_memory(run_child, dim):
    """The pair kernel reads a cache's work list before it waits for the kernel
    before it, which may be one of the caller's that restores the cache memory it
    owns: the list must not lie there."""
    out = run_child(f"""
seg, h, mem = segments(24, {dim}, [(64, 256, 1024, 2048), (3, 5, 70, 300)]), ctypes.c_void_p(), ctypes.c_void_p()
n = L.refcache_bytes(1, 0, ctypes.byref(seg.c))
assert cudart.cudaMalloc(ctypes.byref(mem), ctypes.c_size_t(n)) == 0
assert L.refcache_create(ctypes.byref(h), 1, 0, ctypes.byref(seg.c), mem, n) == 0
t = ctypes.c_void_p(1 << 20)
calls = [L.refcache_build(h, 0, t, t, t, t, None, 0.1, None), L.step_attention(h, 0, t, t, t, t, None, 0.1, None),
         L.refcache_build_in_slot(h, 0, t, t, t, t, None, 0.1, None)]
lists = [cudart.host_cudart_list(i) for i in range(cudart.host_cudart_launches())]
print(json.dumps(dict(calls=calls, mem=[mem.value, n], lists=[x for x in lists if x])))""")
    assert out["calls"] == [0, 0, 0] and len(out["lists"]) == 3
    lo, n = out["mem"]
    assert not any(lo <= x < lo + n for x in out["lists"])


@pytest.mark.parametrize("dim", [64, 128])
def test_workloads_of_the_split_tests_are_split_as_they_say(run_child, dim):
    import split_workloads

    cases = split_workloads.cases(dim)
    reqs = [(w.num_heads, [(r.n_st, r.n_lt, r.n_x, r.n_r) for r in w.requests]) for w, _, _ in cases]
    for flags, want in ((0, 1), (0x100, 2)) if dim == 128 else ((0, 1),):
        out = run_child(f"print(json.dumps([create(h, {dim}, r, {flags}) for h, r in {reqs}]))")
        for c, o in zip(cases, out):
            assert o["code"] == 0 and o["step_launches"] == 2, c[0].name
            assert sorted({j[4] for j in o["jobs"]}) == c[want], c[0].name
    # both forms of the merge: 16 blocks a job (8 at head dim 64), two of which fit on each of 152 SMs
    jobs = [len(o["jobs"]) * 8 * dim // 64 for o in out]
    assert min(jobs) <= 304 < max(jobs)


def test_a_cache_too_large_to_build_can_still_be_planned(run_child):
    """refcache_bytes is arithmetic: it answers for any rows that fit 32 bits."""
    out = run_child("""
seg = segments(8192, 128, [(0, 0, 1, 2147483000)])
print(json.dumps([L.refcache_bytes(1, 0, ctypes.byref(seg.c)), L.refcache_bytes(2, 0, ctypes.byref(seg.c))]))""")
    layer = 2 * 2147483000 * 8192 * 128 * 2
    assert out[1] - out[0] == layer and 0 < out[0] - layer < 1 << 31


def test_a_refused_build_launches_nothing(run_child):
    """An E4M3 cache of more 128-row tiles than its cache write's grid takes (65535): the build says so before
    it has launched the prefill."""
    out = run_child("""
seg, h = segments(1, 128, [(0, 0, 1, 1)] * 65536), ctypes.c_void_p()
assert L.refcache_create(ctypes.byref(h), 1, 0x100, ctypes.byref(seg.c), None, 0) == 0
t = ctypes.c_void_p(1 << 20)
code = L.refcache_build(h, 0, t, t, t, t, None, 0.1, None)
print(json.dumps([code, rc.last_error(), cudart.host_cudart_launches(), L.refcache_layer_built(h, 0)]))""")
    assert out[0] == -4 and out[2] == 0 and out[3] == 0 and "quantize_cache_kernel" in out[1], out


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_every_item_has_rows_and_keys(run_child, mode):
    """The pair kernel walks an item's key tiles without asking whether it has any: requests with empty blocks, in
    every mask mode and cache type, and with parts, make no item without."""
    lens = [0, 1, 5, 200, 1100]
    reqs = [(a if mode != 2 else 0, b, c, d) for a in (0, 3) for b in lens[:3] for c in lens for d in lens]
    big = [(0, 7, 230, 8300), (0, 0, 0, 0), (0 if mode == 2 else 4, 0, 1, 0)]
    out = run_child(f"""
outs = [create(2, 128, r, {mode} | f) for r in ({reqs}, {big}) for f in (0, 0x100)]
print(json.dumps([dict(code=o["code"], jobs=len(o.get("jobs", [])), tasks=o["tasks"]) for o in outs]))""")
    assert all(o["code"] == 0 and o["tasks"] for o in out) and any(o["jobs"] for o in out)
    for o in out:
        assert all(1 <= t[1] <= 256 and min(t[3], t[5]) >= 0 and t[3] + t[5] >= 1 for t in o["tasks"])
