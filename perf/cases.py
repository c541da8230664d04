"""The calls whose time this library is judged by, as a user's program makes them.

A case is one call of one layer: the static prefill with its cache write
(``build``, or ``build_in_slot`` where the caller projected the reference K/V
straight into the cache), one denoising step over the cache (``step``), or the
full recompute that a program without a cache runs (``full``).  ``reqs`` lists
the batch's requests as ``n_st,n_lt,n_x,n_r`` (anchor, instruction, target and
reference tokens), ``;`` between requests; a 1024x1024 image is 4096 tokens, a
512x512 one 1024.  Tensors are packed ``[tokens, heads, dim]`` bf16.
"""
import math

import torch

from paper_2608_21229_gb300 import refcache as rc

#: The largest listed case's work, which a drawn case stays below.
MOST_FLOPS = 5.0e12


def _case(name, kind, heads, dim, reqs, cache="bf16", mask="beyond", lse=False, gain=1.0):
    c = {"kind": kind, "heads": heads, "dim": dim, "reqs": reqs, "cache": cache, "mask": mask, "lse": lse, "gain": gain}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a toy model's step, all launch and latency
        _case("step_tiny_d64", "step", 4, 64, "32,64,256,256", lse=True),
        # editing a 512x512 image with two references: a small interactive step and its prefill
        _case("step_512_2ref", "step", 24, 128, "64,256,1024,2048"),
        _case("build_512_2ref", "build", 24, 128, "64,256,1024,2048", gain=2.5),
        # editing a 1024x1024 image with one reference, the commonest request: sharper scores, log-sum-exp kept
        _case("step_1024_1ref", "step", 24, 128, "128,512,4096,4096", lse=True, gain=2.5),
        _case("build_1024_1ref", "build", 24, 128, "128,512,4096,4096", lse=True),
        # five references at 1024x1024: 40 steps for each prefill
        _case("step_1024_5ref", "step", 24, 128, "128,512,4096,20480"),
        _case("build_1024_5ref", "build", 24, 128, "128,512,4096,20480"),
        # the same with the cache in E4M3 (twice the references in the same memory), and a prefill that writes one
        _case("step_1024_5ref_e4m3", "step", 24, 128, "128,512,4096,20480", cache="fp8"),
        _case("build_1024_2ref_e4m3", "build", 24, 128, "128,512,4096,8192", cache="fp8"),
        # a serving batch of four users' requests, 512x512 and 1024x1024, one to eight references
        _case("step_ragged_4req", "step", 24, 128,
              "64,256,1024,1024;128,512,4096,12288;96,384,1024,5120;128,512,4096,32768", gain=2.5),
        # head dim 64 with the same hidden size, three requests of odd lengths, reference K/V projected in place
        _case("build_in_slot_odd_d64", "build_in_slot", 48, 64, "77,301,1537,2049;13,40,777,1021;128,511,4095,6143", lse=True),
        # the recompute of every row that a program without a cache pays on each step
        _case("full_1024_1ref", "full", 24, 128, "0,512,4096,4096"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(["step", "step", "step", "build", "build", "build_in_slot", "full"])
        dim = rng.choice([128, 128, 128, 64])
        heads = _log_int(rng, 4, 48)
        cache = "fp8" if kind in ("step", "build") and dim == 128 and rng.random() < 0.3 else "bf16"
        mask = rng.choice(["beyond", "beyond", "beyond", "beyond_alt", "isolated"]) if kind != "full" else "beyond"
        reqs = []
        for _ in range(rng.choice([1, 1, 2, 3, 5])):
            n_st = 0 if mask == "isolated" else rng.randint(0, 128)
            reqs.append((n_st, rng.randint(0, 512), _log_int(rng, 200, 4608), _log_int(rng, 200, 24576)))
        c = _case("", kind, heads, dim, ";".join(",".join(str(n) for n in r) for r in reqs), cache, mask,
                  rng.random() < 0.5, rng.choice([1.0, 2.5]))
        # a pass at head dim 64 takes about twice the time of one at 128 for the same work
        if work(c)["flops"] * (128 // dim) <= 0.6 * MOST_FLOPS:
            return c


def _reqs(case):
    return [tuple(int(n) for n in r.split(",")) for r in case["reqs"].split(";")]


def _cu(lens):
    out = [0]
    for n in lens:
        out.append(out[-1] + n)
    return out


def _randn(gen, rows, case, gain=1.0):
    x = torch.randn(rows, case["heads"], case["dim"], generator=gen, device="cuda", dtype=torch.float32)
    return (x * gain).to(torch.bfloat16)


def _inputs(case, seed):
    """Seeded q, k, v of the static rows [ST; R] and of the live rows [LT; X] (full: of the whole sequences).
    Unit-variance bf16; ``gain`` sharpens the scores as learned query scales do."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    reqs, g = _reqs(case), case["gain"]
    live = sum(r[1] + r[2] + (r[3] if case["kind"] == "full" else 0) for r in reqs)
    x = {"live": tuple(_randn(gen, live, case, k) for k in (g, 1.0, 1.0))}
    if case["kind"] != "full":
        x["static"] = tuple(_randn(gen, sum(r[0] + r[3] for r in reqs), case, k) for k in (g, 1.0, 1.0))
    return x


def _anchor_rows(reqs):
    """The anchors' rows of the packed static tensors."""
    rows, s = [], 0
    for r in reqs:
        rows.append(torch.arange(s, s + r[0], device="cuda"))
        s += r[0] + r[3]
    return torch.cat(rows)


def _cached_rows(case, reqs):
    rows, s = [], 0
    for r in reqs:
        n = r[0] + r[3]
        rows.append(torch.arange(s if case["mask"] == "beyond_alt" else s + r[0], s + n, device="cuda"))
        s += n
    return torch.cat(rows)


def prepare(case, seed):
    """The tensors and, but for ``full``, the cache that a program holds before the call."""
    x, reqs, kind = _inputs(case, seed), _reqs(case), case["kind"]
    st = {"case": case, "x": x}
    rows = x["live"][0] if kind in ("step", "full") else x["static"][0]
    st["o"] = torch.empty_like(rows)
    st["lse"] = torch.empty(rows.shape[0], rows.shape[1], dtype=torch.float32, device="cuda") if case["lse"] else None
    if kind == "full":
        st["cu"] = _cu([r[1] + r[2] + r[3] for r in reqs])
        return st
    seg = rc.Segments(case["heads"], case["dim"], _cu([r[1] + r[2] for r in reqs]), _cu([r[0] + r[3] for r in reqs]),
                      [r[0] for r in reqs], [r[1] for r in reqs])
    cache = st["cache"] = rc.RefCache(seg, num_layers=1, mask_mode=case["mask"], cache_dtype=case["cache"])
    q, k, v = x["static"]
    if kind == "step":
        cache.build(0, q, k, v, torch.empty_like(q))
        del x["static"]
    elif kind == "build_in_slot":
        for slot, t in zip(cache.kv(0), (k, v)):
            slot.copy_(t[_cached_rows(case, reqs)])
        a = _anchor_rows(reqs)
        st["anchors"] = (k[a].contiguous(), v[a].contiguous()) if len(a) and case["mask"] != "beyond_alt" else (None, None)
    return st


def run(st):
    kind, o, lse = st["case"]["kind"], st["o"], st["lse"]
    if kind == "full":
        rc.full_attention(st["cu"], *st["x"]["live"], o, lse)
    elif kind == "step":
        st["cache"].step(0, *st["x"]["live"], o, lse)
    elif kind == "build":
        st["cache"].build(0, *st["x"]["static"], o, lse)
    else:
        st["cache"].build_in_slot(0, st["x"]["static"][0], *st["anchors"], o, lse)
    out = {"o": o}
    if lse is not None:
        out["lse"] = lse
    if kind == "build":  # what the call left in the cache
        out["cache"] = list(st["cache"].kv(0) if st["case"]["cache"] == "bf16" else st["cache"].fp8(0))
    return out


def _pairs_and_rows(case):
    """Visible (query, key) pairs of one head, query rows, keys read once and rows written to the cache."""
    pairs = rows = keys = cached = 0
    for n_st, n_lt, n_x, n_r in _reqs(case):
        live, static = n_lt + n_x, n_st + n_r
        kept = static if case["mask"] == "beyond_alt" else n_r
        if case["kind"] == "full":
            n = live + n_r
            pairs, rows, keys = pairs + n * n, rows + n, keys + n
        elif case["kind"] == "step":
            pairs, rows, keys, cached = pairs + live * (live + kept), rows + live, keys + live, cached + kept
        else:
            pairs += n_st * n_st + n_r * static if case["mask"] == "beyond_alt" else static * static
            rows, keys = rows + static, keys + static
            cached += kept if case["kind"] == "build" else 0
    return pairs, rows, keys, cached


def work(case):
    pairs, rows, keys, cached = _pairs_and_rows(case)
    h, d = case["heads"], case["dim"]
    size = 2 if case["cache"] == "bf16" else 1
    return {"bytes": h * d * (2 * 2 * rows + 2 * 2 * keys + 2 * size * cached) + (4 * h * rows if case["lse"] else 0),
            "flops": 4 * d * h * pairs}


def tolerance(case):
    """Softmax weights and outputs are rounded to bf16 (sums in fp32): two correct orders of the work differ by a
    rounding of each.  Steps on an E4M3 cache round their weights to E4M3 (up to 2^-4 each), which depends on the
    running maximum."""
    if case["cache"] == "fp8" and case["kind"] == "step":
        return {"rel": 0.03, "max": 0.3}
    return {"rel": 8e-3, "max": 0.06}


# ---------------------------------------------------------------- the same in 64 bits
def _e4m3(x, amax):
    """x [..., n] as E4M3 codes under one scale amax / 448 (fp32 arithmetic), back in 64 bits."""
    inv = torch.where(amax > 0, 448.0 / amax, torch.zeros_like(amax))
    code = (x.float() * inv).clamp(-448, 448).to(torch.float8_e4m3fn)
    return code.double() * (amax / 448.0).double()


def _e4m3_rows(x):
    return _e4m3(x, x.float().abs().amax(-1, keepdim=True))


def _e4m3_tiles(x):
    """Cached rows [rows, dim] of one head: one scale per 128 rows."""
    return torch.cat([_e4m3(t, t.float().abs().amax().view(1, 1)) for t in x.split(128)]) if len(x) else x.double()


def _attend(q, keys, scale):
    """Softmax attention of one head in 64 bits: ``keys`` is a list of (queries for these keys, K, V)."""
    o, lse = [], []
    for r in range(0, len(q), 2048):
        s = torch.cat([qq[r:r + 2048].double() @ k.double().T for qq, k, _ in keys], 1) * scale
        m = s.amax(1, keepdim=True)
        p = torch.exp(s - m)
        l = p.sum(1, keepdim=True)
        o.append((p / l) @ torch.cat([v.double() for _, _, v in keys]))
        lse.append((m + l.log()).squeeze(1))
    return torch.cat(o), torch.cat(lse)


def exact(case, seed):
    if work(case)["flops"] > 8e12:
        return None
    x, kind, dim = _inputs(case, seed), case["kind"], case["dim"]
    scale = 1.0 / math.sqrt(dim)
    q, k, v = x["live"] if kind in ("step", "full") else x["static"]
    o = torch.zeros(q.shape, dtype=torch.float64, device="cuda")
    lse = torch.zeros(q.shape[:2], dtype=torch.float64, device="cuda")
    l0 = s0 = 0
    for n_st, n_lt, n_x, n_r in _reqs(case):
        live, static = n_lt + n_x + (n_r if kind == "full" else 0), n_st + n_r
        kept = slice(s0 if case["mask"] == "beyond_alt" else s0 + n_st, s0 + static)
        for h in range(case["heads"]):
            if kind in ("step", "full"):
                a = slice(l0, l0 + live)
                keys = [(q[a, h], k[a, h], v[a, h])]
                if kind == "step":
                    kc, vc = x["static"][1][kept, h], x["static"][2][kept, h]
                    keys.append((q[a, h], kc, vc) if case["cache"] == "bf16" else
                                (_e4m3_rows(q[a, h]), _e4m3_tiles(kc), _e4m3_tiles(vc)))
                parts = [(a, keys)]
            elif case["mask"] == "beyond_alt":
                a, b, c = slice(s0, s0 + n_st), slice(s0 + n_st, s0 + static), slice(s0, s0 + static)
                parts = [(r, [(q[r, h], k[w, h], v[w, h])]) for r, w in ((a, a), (b, c)) if r.stop > r.start]
            else:
                a = slice(s0, s0 + static)
                parts = [(a, [(q[a, h], k[a, h], v[a, h])])]
            for r, keys in parts:
                o[r, h], lse[r, h] = _attend(q[r, h], keys, scale)
        l0, s0 = l0 + live, s0 + static
    out = {"o": o}
    if case["lse"]:
        out["lse"] = lse
    if kind == "build":
        rows = _cached_rows(case, _reqs(case))
        out["cache"] = [k[rows].double(), v[rows].double()] if case["cache"] == "bf16" else [None, None, None]
    return out
