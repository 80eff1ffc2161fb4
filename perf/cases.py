"""Timed cases of the resource-routed attention path, through the package's public calls.

A case is one thing that a serving program has one attention layer do:

  encode  new resources arrive and are encoded into the cache
  turn    a batch of requests composes cached resources (compaction) and prefills its
          conversation tokens; `copy` = the route rows are materialised, else the prefill
          reads them from the cache through the index list; `pages` = the routes' pages
          for the decode that follows are materialised too
  later   a later turn of running conversations: new tokens over routes and earlier turns
  decode  one token for every running sequence; `copy` = resource rows in pages of their
          own, else read from the cache through the index list
  whole   encode, compaction and prefill in the exact fp32 arithmetic

Lengths follow from the case alone (`mix` seeds them), so that the work of a case is known;
tensors, keep masks and routes follow from the seed.  Activations and cached rows are N(0,1),
as normalised projections are; about 30 % of a resource's tokens are kept, as field spans of
4-32 tokens, and a KV group sees a quarter of a request's resources.
"""
import functools
import math

import numpy as np
import torch

from paper_2608_19662_b200 import PACKED, PAGED, ReCache
from paper_2608_19662_b200 import workloads as wl

KEPT = 0.30            # share of a resource's tokens that the span masks keep
ROUTED = 0.25          # share of a request's resources that a KV group sees
MAX_POS = 131072       # rows of the rotary table: the longest context served
THETA = {"bf16": 1.0e6, "f32": 1.0e4}
PAGE = wl.PAGE_TOKENS


def _case(kind, name=None, hq=32, g=8, d=128, dtype="bf16", **sizes):
    case = {"kind": kind, "hq": hq, "g": g, "d": d, "dtype": dtype, **sizes}
    return {"name": name, **case} if name else case


def listed():
    return [
        # a single tool is added while requests are served: the smallest encode, where launches count
        _case("encode", "encode-one-tool", n_res=1, lo=200, hi=800, mix=1),
        # a pool of ordinary tools is encoded once and cached
        _case("encode", "encode-pool", n_res=64, lo=150, hi=1200, mix=3),
        # a long tool set arrives at once: the largest call
        _case("encode", "encode-long-tool-set", n_res=64, lo=1000, hi=2000, mix=5),
        # first turn of one user over a handful of tools: what the time to first token waits for
        _case("turn", "turn-one-request", batch=1, res=8, lo=200, hi=800, tq_lo=512, tq_hi=512, copy=True, pages=False, mix=2),
        # a batch of first turns over a shared pool; its decode pages are laid out in the same pass
        _case("turn", "turn-batch", batch=16, res=8, lo=150, hi=1200, tq_lo=256, tq_hi=1024, copy=True, pages=True, mix=3),
        # one long turn over a long tool set
        _case("turn", "turn-long-tool-set", batch=1, res=64, lo=1000, hi=2000, tq_lo=2048, tq_hi=2048, copy=True, pages=False, mix=5),
        # a batch of short turns whose route rows are never copied
        _case("turn", "turn-zero-copy", batch=8, res=16, lo=700, hi=1300, tq_lo=256, tq_hi=256, copy=False, pages=False, mix=6),
        # short user turns in running conversations, on the shape with two query heads per KV head
        _case("later", "later-turn", hq=16, batch=8, res=16, lo=500, hi=700, tq_lo=17, tq_hi=250, hist_lo=300, hist_hi=2048, mix=7),
        # the steady decode of a full server
        _case("decode", "decode-batch-64", batch=64, res=16, lo=500, hi=700, hist_lo=2048, hist_hi=2048, copy=True, mix=4),
        # one user alone: a decode step of tens of microseconds
        _case("decode", "decode-one-sequence", batch=1, res=16, lo=500, hi=700, hist_lo=1500, hist_hi=3000, copy=True, mix=8),
        # decode without materialised resource pages, ragged histories
        _case("decode", "decode-zero-copy", batch=16, res=16, lo=500, hi=700, hist_lo=300, hist_hi=4000, copy=False, mix=9),
        # the whole path in exact fp32 arithmetic, as it is run where bf16 results are checked
        _case("whole", "whole-fp32", hq=4, g=2, d=64, dtype="f32", n_res=6, lo=17, hi=400, tq_lo=160, tq_hi=160, mix=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _span(rng, lo, hi):
    """A range of lengths inside [lo, hi]."""
    a, b = _log(rng, lo, hi), _log(rng, lo, hi)
    return min(a, b), max(a, b)


def draw(rng):
    kind = rng.choice(["encode", "encode", "encode", "turn", "turn", "turn", "turn", "later", "decode", "decode", "decode", "whole"])
    mix = rng.randrange(1 << 16)
    hq = rng.choice([16, 32, 32, 32, 64])
    if kind == "encode":
        lo, hi = _span(rng, 60, 2000)
        square = (lo * lo + lo * hi + hi * hi) / 3            # mean of a length's square: the cost of a resource
        n = min(_log(rng, 1, 64), int(64 * 2.3e6 * 32 / (square * hq)))
        return _case("encode", hq=hq, n_res=n, lo=lo, hi=hi, mix=mix)
    if kind == "turn":
        batch, copy = _log(rng, 1, 16), rng.random() < 0.6
        lo, hi = _span(rng, 100, 1500)
        tq_lo, tq_hi = _span(rng, 32, 2048 if batch <= 2 else 1024)
        return _case("turn", hq=hq, batch=batch, res=_log(rng, 4, 64 if batch == 1 else 16), lo=lo, hi=hi, tq_lo=tq_lo, tq_hi=tq_hi,
                     copy=copy, pages=copy and rng.random() < 0.5, mix=mix)
    if kind == "later":
        tq_lo, tq_hi = _span(rng, 9, 400)
        h_lo, h_hi = _span(rng, 100, 4000)
        return _case("later", hq=hq, batch=_log(rng, 1, 32), res=_log(rng, 4, 16), lo=200, hi=800, tq_lo=tq_lo, tq_hi=tq_hi, hist_lo=h_lo,
                     hist_hi=h_hi, mix=mix)
    if kind == "decode":
        h_lo, h_hi = _span(rng, 64, 4096)
        return _case("decode", hq=hq, batch=_log(rng, 1, 64), res=_log(rng, 4, 16), lo=200, hi=800, hist_lo=h_lo, hist_hi=h_hi,
                     copy=rng.random() < 0.6, mix=mix)
    hq, g, d = rng.choice([(4, 2, 64), (8, 2, 64), (8, 2, 128)])
    lo, hi = _span(rng, 17, 500)
    tq = _log(rng, 32, 256)
    return _case("whole", hq=hq, g=g, d=d, dtype="f32", n_res=rng.randrange(2, 9), lo=lo, hi=hi, tq_lo=tq, tq_hi=tq, mix=mix)


# ---------------------------------------------------------------- sizes of a case --
def _lengths(case):
    """(resource lengths [requests][resources], query tokens [requests], history rows [requests])."""
    rng = np.random.default_rng([case["mix"], 19662])
    batch = case.get("batch", 1)
    res = rng.integers(case["lo"], case["hi"] + 1, (batch, case.get("res", case.get("n_res")))).astype(np.int32)
    tq = rng.integers(case.get("tq_lo", 1), case.get("tq_hi", 1) + 1, batch).astype(np.int32)
    hist = rng.integers(case.get("hist_lo", 0), case.get("hist_hi", 0) + 1, batch).astype(np.int32)
    return res, tq, hist


def _visible(n_res):
    return max(1, int(math.floor(ROUTED * n_res + 0.5)))


def work(case):
    res, tq, hist = (x.astype(np.int64) for x in _lengths(case))
    hq, g, d = case["hq"], case["g"], case["d"]
    row = d * (2 if case["dtype"] == "bf16" else 4)       # bytes of one key or value row
    s = hq // g
    route = res.mean(1) * _visible(res.shape[1]) * KEPT   # rows a route exposes, on average
    n_bytes = flops = 0.0
    if case["kind"] in ("encode", "whole"):
        t = int(res.sum())
        n_bytes += t * (2 * hq + 4 * g) * row              # q in, o out; k, v in and into the cache
        flops += 4 * d * hq * float((res * (res + 1) // 2).sum())
    if case["kind"] in ("turn", "later", "whole"):
        pairs = (tq * (route + hist) + tq * (tq + 1) / 2).sum()
        flops += 4 * d * hq * float(pairs)
        n_bytes += float(tq.sum()) * (2 * hq + 4 * g) * row + float(route.sum()) * g * 2 * row
        if case["kind"] == "later":
            n_bytes += float(hist.sum()) * g * 2 * row
        else:
            copies = (1 if case.get("copy", True) else 0) + (1 if case.get("pages") else 0)
            n_bytes += float(res.sum()) + float(route.sum()) * g * (4 + copies * 2 * row)
    if case["kind"] == "decode":
        rows = float((route + hist).sum()) * g
        n_bytes += rows * 2 * row + len(tq) * (2 * hq + 4 * g) * row
        flops += 4 * d * s * rows
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    # four times what the outputs differ by from the same pass in fp64: rel 3.6e-7, max 3e-6 in fp32;
    # rel 2.3e-3, max 2.3e-2 with bf16 inputs, probabilities and results
    if case["dtype"] == "f32":
        return {"rel": 1.5e-6, "max": 1.2e-5}
    return {"rel": 1e-2, "max": 1e-1}


# ------------------------------------------------------------------------ inputs --
@functools.lru_cache(maxsize=8)
def _context(hq, g, d, dtype):
    """The attention shape's context: made once by a program, like the model's weights."""
    return ReCache(hq, g, d, THETA[dtype], dtype, max_pos=MAX_POS, page_tokens=PAGE, device=torch.cuda.current_device())


class _Draw:
    """Seeded tensors on the device, and index arrays from the same seed."""

    def __init__(self, seed, dtype):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(int(seed))
        self.np = np.random.default_rng([int(seed), 1])
        self.dtype = torch.bfloat16 if dtype == "bf16" else torch.float32

    def normal(self, *shape):
        return torch.randn(shape, generator=self.gen, dtype=self.dtype, device="cuda")

    @staticmethod
    def ints(a, dtype=np.int32):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype)).cuda()


def _offsets(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)


def _routes(case, dr, res):
    """Keep mask over the pool and visibility of every listed resource, and the rows each route gets."""
    g, batch, n = case["g"], res.shape[0], res.shape[1]
    masks = wl.keep_mask_spans(dr.np, res.reshape(-1))
    vis = np.concatenate([wl.routes_random(dr.np, g, n, ROUTED) for _ in range(batch)], axis=1)
    kept = np.array([int(m.sum()) for m in masks], np.int64)
    rows = (vis.astype(np.int64) * kept).reshape(g, batch, n).sum(2).T.reshape(-1)      # route = request * g + group
    return np.concatenate(masks), vis, rows


def _most_rows(res):
    """Rows that a route of each request can hold at most: what buffers are sized for, the kept share being the device's to know."""
    return np.sort(res, axis=1)[:, -_visible(res.shape[1]):].sum(1).astype(np.int64)


def _compaction(case, dr, res):
    """Arguments and outputs of compact_routes for requests that list `res`, packed one after the other in the pool."""
    st = {}
    keep, vis, _ = _routes(case, dr, res)
    routes, capacity = res.shape[0] * case["g"], int(_most_rows(res).sum()) * case["g"]
    flat = res.reshape(-1)
    st["keep"], st["vis"] = dr.ints(keep, np.uint8), dr.ints(vis, np.uint8)
    st["res_off"] = dr.ints(np.arange(res.shape[0] + 1) * res.shape[1])
    st["res_slot"], st["res_len"] = dr.ints(_offsets(flat)[:-1]), dr.ints(flat)
    st["route_cu"] = torch.zeros(routes + 1, dtype=torch.int32, device="cuda")
    st["route_idx"] = torch.zeros(capacity, dtype=torch.int32, device="cuda")
    return st, routes, capacity


def _prepare_encode(case, dr, res):
    flat = res.reshape(-1)
    t, hq, g, d = int(flat.sum()), case["hq"], case["g"], case["d"]
    return dict(q=dr.normal(t, hq, d), k=dr.normal(t, g, d), v=dr.normal(t, g, d), cu=dr.ints(_offsets(flat)), max_len=int(flat.max()),
                slot=dr.ints(_offsets(flat)[:-1]), k_cache=torch.zeros((g, t, d), dtype=dr.dtype, device="cuda"),
                v_cache=torch.zeros((g, t, d), dtype=dr.dtype, device="cuda"))


def _prepare_queries(case, dr, res, tq, before):
    n, hq, g, d = int(tq.sum()), case["hq"], case["g"], case["d"]
    return dict(cq=dr.normal(n, hq, d), ck=dr.normal(n, g, d), cv=dr.normal(n, g, d), cu_q=dr.ints(_offsets(tq)),
                q_pos0=dr.ints(res.sum(1) + before), max_q=int(tq.max()))


def _prepare_turn(case, dr, res, tq):
    g, d, pool = case["g"], case["d"], int(res.sum())
    st, routes, capacity = _compaction(case, dr, res)
    st.update(_prepare_queries(case, dr, res, tq, 0))
    if case["kind"] == "turn":
        st["k_cache"], st["v_cache"] = dr.normal(g, pool, d), dr.normal(g, pool, d)
    st["copy"] = case.get("copy", True)
    if st["copy"]:
        st["k_route"], st["v_route"] = (torch.zeros((capacity, d), dtype=dr.dtype, device="cuda") for _ in range(2))
    if case.get("pages"):
        n_pages = (_most_rows(res) + PAGE - 1) // PAGE
        total = int(n_pages.sum()) * g
        st["free"] = dr.ints(dr.np.permutation(total))
        st["k_pages"], st["v_pages"] = (torch.zeros((total, PAGE, d), dtype=dr.dtype, device="cuda") for _ in range(2))
        st["page_table"] = torch.zeros((routes, int(n_pages.max())), dtype=torch.int32, device="cuda")
        st["route_len"] = torch.zeros(routes, dtype=torch.int32, device="cuda")
    return st


def _prepare_later(case, dr, res, tq, hist):
    g, d = case["g"], case["d"]
    _, _, rows = _routes(case, dr, res)
    st = _prepare_queries(case, dr, res, tq, hist)
    st["k_route"], st["v_route"] = dr.normal(int(rows.sum()), d), dr.normal(int(rows.sum()), d)
    st["route_cu"] = dr.ints(_offsets(rows))
    room = (hist + tq + PAGE - 1) // PAGE * PAGE          # page-aligned regions: the same memory serves the decode
    st["conv_slot"], st["hist_len"] = dr.ints(_offsets(room)[:-1]), dr.ints(hist)
    st["k_conv"], st["v_conv"] = dr.normal(g, int(room.sum()), d), dr.normal(g, int(room.sum()), d)
    return st


def _prepare_decode(case, dr, res, hist):
    hq, g, d, batch = case["hq"], case["g"], case["d"], res.shape[0]
    st = dict(q=dr.normal(batch, hq, d), k_new=dr.normal(batch, g, d), v_new=dr.normal(batch, g, d), q_pos=dr.ints(res.sum(1) + hist - 1),
              hist_len=dr.ints(np.repeat(hist, g)), copy=case["copy"])
    keep, vis, rows = _routes(case, dr, res)
    room, hist_pages = np.repeat((_most_rows(res) + PAGE - 1) // PAGE, g), np.repeat((hist + PAGE - 1) // PAGE, g)
    res_pages = (rows + PAGE - 1) // PAGE
    st["max_res_pages"] = int(room.max())

    def table(counts, ids, width):
        out = np.full((len(counts), int(width)), -1, np.int32)
        out[np.arange(out.shape[1])[None, :] < counts[:, None]] = ids
        return dr.ints(out)

    n_hist = int(hist_pages.sum())
    ids = dr.np.permutation(n_hist + (int(room.sum()) if case["copy"] else 0)).astype(np.int32)
    st["hist_table"] = table(hist_pages, ids[:n_hist], hist_pages.max())
    if case["copy"]:
        st["res_table"], st["res_rows"] = table(res_pages, ids[n_hist:][:int(res_pages.sum())], room.max()), dr.ints(rows)
    else:
        flat = res.reshape(-1)
        slot = _offsets(flat)[:-1]
        kept = [np.flatnonzero(keep[a:a + n]).astype(np.int32) + a for a, n in zip(slot, flat)]
        n = res.shape[1]
        idx = [kept[b * n + r] for b in range(batch) for kg in range(g) for r in range(n) if vis[kg, b * n + r]]
        st["route_idx"], st["route_cu"] = dr.ints(np.concatenate(idx)), dr.ints(_offsets(rows))
        st["k_cache"], st["v_cache"] = dr.normal(g, int(flat.sum()), d), dr.normal(g, int(flat.sum()), d)
    st["k_pages"], st["v_pages"] = dr.normal(len(ids), PAGE, d), dr.normal(len(ids), PAGE, d)
    return st


def prepare(case, seed):
    dr = _Draw(seed, case["dtype"])
    res, tq, hist = _lengths(case)
    st = {"kind": case["kind"], "rc": _context(case["hq"], case["g"], case["d"], case["dtype"])}
    if case["kind"] == "encode":
        st.update(_prepare_encode(case, dr, res))
    elif case["kind"] == "turn":
        st.update(_prepare_turn(case, dr, res, tq))
    elif case["kind"] == "later":
        st.update(_prepare_later(case, dr, res, tq, hist))
    elif case["kind"] == "decode":
        st.update(_prepare_decode(case, dr, res, hist))
    else:
        st.update(_prepare_encode(case, dr, res))
        st.update(_prepare_turn(case, dr, res, tq))
    return st


# -------------------------------------------------------------------------- passes --
def _encode(st):
    out = st["rc"].encode_resources(st["q"], st["k"], st["v"], st["cu"], st["max_len"], st["slot"], st["k_cache"], st["v_cache"])
    return {"o": out, "k_cache": st["k_cache"], "v_cache": st["v_cache"]}


def _turn(st):
    rc = st["rc"]
    lists = (st["keep"], st["res_off"], st["res_slot"], st["res_len"], st["vis"])
    queries = (st["cq"], st["ck"], st["cv"], st["cu_q"], st["q_pos0"], st["max_q"])
    done = {"route_cu": st["route_cu"], "route_idx": st["route_idx"]}
    if st["copy"]:
        rc.compact_routes(st["k_cache"], st["v_cache"], *lists, PACKED, st["route_cu"], st["route_idx"], st["k_route"], st["v_route"])
        done["o"], done["k_conv"], done["v_conv"] = rc.attend_prefill(*queries, st["k_route"], st["v_route"], st["route_cu"])
        done["k_route"], done["v_route"] = st["k_route"], st["v_route"]
    else:
        rc.compact_routes(st["k_cache"], st["v_cache"], *lists, PACKED, st["route_cu"], st["route_idx"], None, None)
        done["o"], done["k_conv"], done["v_conv"] = rc.attend_prefill_gather(*queries, st["k_cache"], st["v_cache"], st["route_idx"],
                                                                             st["route_cu"])
    if "page_table" in st:
        rc.compact_routes(st["k_cache"], st["v_cache"], *lists, PAGED, st["route_cu"], st["route_idx"], st["k_pages"], st["v_pages"],
                          route_len=st["route_len"], page_table=st["page_table"], free_pages=st["free"])
        done.update({name: st[name] for name in ("k_pages", "v_pages", "page_table", "route_len")})
    return done


def _later(st):
    out = st["rc"].attend_prefill_history(st["cq"], st["ck"], st["cv"], st["cu_q"], st["q_pos0"], st["max_q"], st["k_route"], st["v_route"],
                                          st["route_cu"], st["k_conv"], st["v_conv"], st["conv_slot"], st["hist_len"])
    return {"o": out, "k_conv": st["k_conv"], "v_conv": st["v_conv"]}


def _decode(st):
    rc = st["rc"]
    if st["copy"]:
        out = rc.attend_decode(st["q"], st["q_pos"], st["k_pages"], st["v_pages"], st["res_table"], st["res_rows"], st["hist_table"],
                               st["hist_len"], k_new=st["k_new"], v_new=st["v_new"])
    else:
        out = rc.attend_decode_gather(st["q"], st["q_pos"], st["k_cache"], st["v_cache"], st["route_idx"], st["route_cu"],
                                      st["max_res_pages"], st["k_pages"], st["v_pages"], st["hist_table"], st["hist_len"],
                                      k_new=st["k_new"], v_new=st["v_new"])
    return {"o": out, "k_pages": st["k_pages"], "v_pages": st["v_pages"]}


def _whole(st):
    return {"encode": _encode(st), "turn": _turn(st)}


_PASS = {"encode": _encode, "turn": _turn, "later": _later, "decode": _decode, "whole": _whole}


def run(state):
    return _PASS[state["kind"]](state)
