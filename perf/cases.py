"""The work a user of this library has it do, as cases that can be timed and compared.

A case names one public entry point and the sizes of the pages it works on; the page structures
follow from the case alone, every tensor value from the seed. Sizes are those of the repository's
own workloads (inputs.py, bench.py and the tests): 16 query heads over 2 KV heads of 128 dims in
16-token bf16 blocks, prefixes of 1024 to 4096 tokens, 8 layout tokens per branch, log-normal
private histories.

  decode    one attention layer of a decode step over the paged cache (engine.DecodePlan.run, or
            padoc_branch_decode_attn_e4m3 for the FP8 cache)
  prefill   one attention layer of the packed training / prefill forward (engine.PrefillPlan.run)
  backward  its gradients (engine.PrefillBwdPlan.run)
  chunk     branch prefill over the paged cache (engine.ChunkPrefillPlan.run)
  fill      a batch's K/V written to the FP8 cache: whole blocks, then one appended row per stream
  loop      Algorithm 1 from admission to the last EOS (engine.MaskedParallelLoop)
"""
import math

import numpy as np
import torch

from paper_2608_06146_gb300 import engine
from paper_2608_06146_gb300 import padoc_attn as pa
from paper_2608_06146_gb300.inputs import LoopTokenSource, PageSpec

DEV = "cuda"
D = 128          # head dim
BS = 16          # tokens per cache block
GROUP = 8        # query heads per KV head


def _case(name, kind, pages, prefix, branches, private, cap, shape, *, kv_heads=2, kv="bf16", layout=False,
          forks="ordered", done=0):
    """prefix, branches: (least, most) per page; private: median of the branch lengths; done: private
    rows a chunk's branch has in the cache before the chunk; shape: seed of the page structures."""
    return {"name": name, "kind": kind, "pages": pages, "prefix_min": prefix[0], "prefix_max": prefix[1],
            "branches_min": branches[0], "branches_max": branches[1], "private": private, "cap": cap, "shape": shape,
            "kv_heads": kv_heads, "kv": kv, "layout": layout, "forks": forks, "done": done}


def listed():
    return [
        # one user's page: the latency of a single decode step of 16 branches
        _case("decode_page", "decode", 1, (2048, 2048), (16, 16), 96, 256, 1),
        # the serving batch: 32 concurrent pages, about 20 live branches each
        _case("decode_serving", "decode", 32, (1024, 4096), (10, 30), 96, 2048, 3),
        # table- and formula-heavy pages, many branches each, the layout streams decoding along
        _case("decode_dense", "decode", 40, (4096, 4096), (56, 64), 64, 1024, 2, layout=True),
        # the serving batch over the FP8 cache, and one page over it
        _case("decode_fp8_serving", "decode", 32, (1024, 4096), (10, 30), 96, 2048, 3, kv="e4m3"),
        _case("decode_fp8_page", "decode", 1, (2048, 2048), (16, 16), 96, 256, 1, kv="e4m3"),
        # training or prefilling a single page of odd length, and a packed batch of about 32k tokens
        _case("prefill_page", "prefill", 1, (2001, 2001), (20, 20), 56, 512, 5),
        _case("prefill_packed", "prefill", 8, (1024, 3072), (8, 48), 50, 1024, 4),
        # the training backward of the same, its branches in reading order and shuffled
        _case("backward_page", "backward", 1, (2001, 2001), (20, 20), 56, 512, 5, forks="shuffled"),
        _case("backward_packed", "backward", 8, (1024, 3072), (8, 48), 50, 1024, 4),
        # branches resumed in the middle and prefilled over pages already in the cache
        _case("chunk_batch", "chunk", 12, (1024, 4096), (10, 30), 96, 2048, 3, done=21),
        # a batch's prefixes and histories written to the FP8 cache
        _case("fill_fp8", "fill", 32, (1024, 4096), (10, 30), 96, 2048, 3, kv="e4m3"),
        # four pages decoded from admission to their last EOS
        _case("loop_pages", "loop", 4, (1024, 2048), (8, 16), 48, 128, 6),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["decode", "decode", "decode", "prefill", "prefill", "backward", "backward", "chunk", "fill", "loop"])
    shape = rng.randrange(1 << 30)
    kvh = rng.choice([1, 2, 2, 2])
    lo = rng.randint(500, 3000)
    prefix = (lo, rng.randint(lo, 4096))
    forks = rng.choice(["ordered", "shuffled"])
    b = rng.randint(1, 30)
    c = _case("", kind, 1, prefix, (b, b + rng.randint(0, 10)), rng.randint(20, 120), rng.randint(200, 2048), shape,
              kv_heads=kvh, forks=forks)
    del c["name"]
    if kind == "decode":
        c["pages"] = log_int(1, 40)
        c["kv"] = rng.choice(["bf16", "e4m3"])
        c["layout"] = rng.random() < 0.4
        if rng.random() < 0.3:
            c["branches_min"], c["branches_max"] = 33, rng.randint(34, 64)
    elif kind in ("prefill", "backward"):
        c["pages"] = log_int(1, 7 if kind == "prefill" else 3)
        c["prefix_min"] = min(c["prefix_min"], 2500)
        c["prefix_max"] = max(c["prefix_min"], min(c["prefix_max"], 3072 if kind == "prefill" else 2500))
        c["private"], c["cap"] = rng.randint(10, 50), 1024
    elif kind == "chunk":
        c["pages"] = log_int(1, 6)
        c["branches_max"] = min(c["branches_max"], 25)
        c["branches_min"] = min(c["branches_min"], 20)
        c["private"], c["done"] = rng.randint(20, 96), rng.choice([0, 0, 5, 40])
    elif kind == "fill":
        c["pages"], c["kv"] = log_int(1, 32), "e4m3"
        c["branches_max"] = min(c["branches_max"], 30)
        c["branches_min"] = min(c["branches_min"], 30)
    else:
        c["pages"], c["private"], c["cap"] = rng.randint(1, 3), rng.randint(10, 48), 128
        c["branches_min"], c["branches_max"] = 1 + b // 4, 1 + b // 2
        c["prefix_max"] = max(c["prefix_min"], min(c["prefix_max"], 2048))
    return c


# ------------------------------------------------------------------------------------------------
# Structures and values
# ------------------------------------------------------------------------------------------------

def _pages(case):
    rng = np.random.default_rng(case["shape"])
    sigma = 0.75 if case["kind"] in ("prefill", "backward") else 1.0
    pages = []
    for _ in range(case["pages"]):
        p = int(rng.integers(case["prefix_min"], case["prefix_max"] + 1))
        n = int(rng.integers(case["branches_min"], case["branches_max"] + 1))
        lens = np.clip(np.round(case["private"] * np.exp(sigma * rng.standard_normal(n))), 1, case["cap"]).astype(int)
        forks = 8 * (1 + np.arange(n))
        if case["forks"] == "shuffled":
            forks = rng.permutation(forks)
        pages.append(PageSpec(p, 8 * n, [int(x) for x in forks], [int(x) for x in lens]))
    return pages


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.bfloat16)


def _streams(case, pages):
    """(page, shared rows seen, private rows) of every stream, page by page."""
    out = []
    for i, pg in enumerate(pages):
        out += [(i, pg.prefix_len + f, n) for f, n in zip(pg.fork_offset, pg.branch_len)]
        if case["layout"]:
            out.append((i, pg.stream_len, 0))
    return out


def _tables(case, pages, seed):
    """Block tables of the pages' shared rows and the streams' private rows over a pool in random order."""
    streams = _streams(case, pages)
    need = [-(-pg.stream_len // BS) for pg in pages] + [-(-n // BS) for _, _, n in streams]
    ids = np.random.default_rng(seed).permutation(sum(need)).astype(np.int32)
    page_table = np.full((len(pages), max(need[:len(pages)])), -1, np.int32)
    stream_table = np.full((len(streams), max(max(need[len(pages):]), 1)), -1, np.int32)
    at = 0
    for i, n in enumerate(need):
        row = page_table[i] if i < len(pages) else stream_table[i - len(pages)]
        row[:n] = ids[at:at + n]
        at += n
    return page_table, stream_table, max(len(ids), 1)


def _bf16_pool(case, blocks, seed):
    g = _gen(seed)
    shape = (blocks, case["kv_heads"], BS, D)
    return _randn(g, *shape), _randn(g, *shape)


def _scaled(case, x):
    """Codes and scales of an FP8 cache holding x: per (block, KV head) scale = amax / 448."""
    scale = x.float().abs().amax(dim=(2, 3)) / 448.0
    codes = (x.float() / scale[:, :, None, None]).to(torch.float8_e4m3fn).view(torch.uint8)
    return codes, scale


def _up(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _chunks(case, pages):
    """One chunk per branch: its rows past the first `done` (all of a branch no longer than that)."""
    out = []
    for i, pg in enumerate(pages):
        for f, n in zip(pg.fork_offset, pg.branch_len):
            a = case["done"] if n > case["done"] else 0
            out.append((i, pg.prefix_len + f, a, n - a))
    return out


# ------------------------------------------------------------------------------------------------
# The cases' passes
# ------------------------------------------------------------------------------------------------

def prepare(case, seed):
    pages, hkv = _pages(case), case["kv_heads"]
    hq, scale, kind = GROUP * hkv, 1.0 / math.sqrt(D), case["kind"]
    s = {"case": case, "scale": scale}
    if kind in ("decode", "chunk"):
        page_table, stream_table, blocks = _tables(case, pages, seed)
        k, v = _bf16_pool(case, blocks, seed)
        s["page_table"] = _up(page_table)
        if kind == "decode":
            s["plan"] = engine.DecodePlan(pages, hq, hkv, D, DEV, layout_streams=case["layout"])
            s["stream_table"] = _up(stream_table)
            rows = s["plan"].num_streams
        else:
            page_len = np.array([pg.stream_len for pg in pages], np.int32)
            s["plan"] = engine.ChunkPrefillPlan(page_len, _chunks(case, pages), stream_table, hq, hkv, D, DEV)
            rows = s["plan"].num_tokens
        if case["kv"] == "e4m3":
            s["pool"] = pa.E4M3Pool(blocks, hkv, D, DEV)
            for x, codes, scales in ((k, s["pool"].k_codes, s["pool"].k_scales), (v, s["pool"].v_codes, s["pool"].v_scales)):
                c, f = _scaled(case, x)
                codes.copy_(c)
                scales.copy_(f)
        else:
            s["k"], s["v"] = k, v
        s["q"] = _randn(_gen(seed + 1000003), rows, hq, D)
        s["out"], s["lse"] = torch.empty_like(s["q"]), torch.empty(rows, hq, device=DEV)
    elif kind in ("prefill", "backward"):
        t = sum(pg.packed_len for pg in pages)
        g = _gen(seed)
        s["q"], s["k"], s["v"] = _randn(g, t, hq, D), _randn(g, t, hkv, D), _randn(g, t, hkv, D)
        s["out"], s["lse"] = torch.empty_like(s["q"]), torch.empty(t, hq, device=DEV)
        s["plan"] = engine.PrefillPlan(pages, torch.bfloat16, D, DEV)
        if kind == "backward":
            s["plan"].run(s["q"], s["k"], s["v"], scale, s["out"], s["lse"])
            s["plan"] = engine.PrefillBwdPlan(pages, torch.bfloat16, D, hq, DEV)
            s["dout"] = _randn(g, t, hq, D)
            s["dq"], s["dk"], s["dv"] = torch.empty_like(s["q"]), torch.empty_like(s["k"]), torch.empty_like(s["v"])
    elif kind == "fill":
        page_table, stream_table, blocks = _tables(case, pages, seed)
        s["k"], s["v"] = _bf16_pool(case, blocks, seed)
        s["pool"] = pa.E4M3Pool(blocks, hkv, D, DEV)
        s["dst"] = _up(np.random.default_rng(seed + 1).permutation(blocks).astype(np.int32))
        streams, slots = _streams(case, pages), []
        for i, (_, _, n) in enumerate(streams):     # each stream's newest row
            slots.append(int(stream_table[i, (n - 1) // BS]) * BS + (n - 1) % BS)
        s["slots"] = _up(np.array(slots, np.int32))
        g = _gen(seed + 1000003)
        s["k_new"], s["v_new"] = _randn(g, len(slots), hkv, D), _randn(g, len(slots), hkv, D)
    else:
        t = sum(pg.packed_len for pg in pages)
        g = _gen(seed)
        s["q"], s["k"], s["v"] = _randn(g, t, hq, D), _randn(g, t, hkv, D), _randn(g, t, hkv, D)
        need = sum(-(-pg.stream_len // BS) + sum(-(-n // BS) for n in pg.branch_len) for pg in pages)
        order = np.random.default_rng(seed).permutation(need + 8).astype(np.int32)
        s["loop"] = engine.MaskedParallelLoop(need + 8, hq, hkv, D, torch.bfloat16, DEV, block_order=order)
        s["admit"], s["steps"], s["rows"], s["ids"] = _record(pages)
        cap = len(pages) + sum(pg.num_branches for pg in pages)
        s["out"] = torch.zeros(len(s["rows"]) + cap, hq, D, device=DEV, dtype=torch.bfloat16)
        s["lse"] = torch.zeros(len(s["rows"]) + cap, hq, device=DEV)
        s["cap"], s["first_id"], s["row_of"] = cap, 0, np.zeros(16 * s["ids"], np.int32)
    return s


def _record(pages):
    """What the decoder makes of the pages, as it will be replayed: each page's admission, each step's
    (stream ids, source rows, forks, EOS), and all decoded rows in order."""
    src = LoopTokenSource(pages)
    mpd = pa.Mpd(sum(-(-pg.stream_len // BS) + sum(-(-n // BS) for n in pg.branch_len) for pg in pages) + 8, BS)
    admit, steps, rows, ids = [], [], [], 0
    for p in range(len(pages)):
        plen, nf, eos, prow = src.admission(p)
        _, _, new = mpd.add_page(plen, nf, eos)
        src.admitted(p, new)
        admit.append((plen, nf, eos, prow))
        ids = max(ids, int(new.max()) + 1)
    while mpd.status()[1]:
        live, _ = mpd.begin_step()
        r = src.rows(live).astype(np.int32)
        nf, eos = src.events(live)
        new = mpd.end_step(nf, eos)
        src.forked(live, nf, new)
        ids = max([ids] + [int(x) + 1 for x in new])
        steps.append((live.astype(np.int64), r, nf, eos))
        rows.append(r)
    mpd.close()
    return admit, steps, np.concatenate(rows), ids


def run(state):
    s, kind = state, state["case"]["kind"]
    if kind == "decode" and s["case"]["kv"] == "e4m3":
        p = s["plan"]
        pa.padoc_branch_decode_attn_e4m3(s["pool"], p.info, p.plan_dev, s["page_table"], s["stream_table"], s["q"],
                                         s["scale"], s["out"], s["lse"], p.workspace)
    elif kind == "decode":
        s["plan"].run(s["k"], s["v"], s["page_table"], s["stream_table"], s["q"], s["scale"], s["out"], s["lse"])
    elif kind == "chunk":
        s["plan"].run(s["k"], s["v"], s["page_table"], s["q"], s["scale"], s["out"], s["lse"])
    elif kind == "prefill":
        s["plan"].run(s["q"], s["k"], s["v"], s["scale"], s["out"], s["lse"])
    elif kind == "backward":
        s["plan"].run(s["q"], s["k"], s["v"], s["out"], s["dout"], s["lse"], s["scale"], s["dq"], s["dk"], s["dv"])
        return [s["dq"], s["dk"], s["dv"]]
    elif kind == "fill":
        pa.padoc_quantize_kv_blocks(s["pool"], s["k"], s["v"], s["dst"])
        pa.padoc_append_inputs_e4m3(s["pool"], s["k_new"], s["v_new"], s["slots"])
        p = s["pool"]
        return [p.k_codes, p.v_codes, p.k_scales, p.v_scales]
    else:
        return _run_loop(s)
    return [s["out"], s["lse"]]


def _run_loop(s):
    loop, base, at = s["loop"], s["first_id"], 0
    if base + s["ids"] > s["row_of"].size:
        s["row_of"] = np.zeros(2 * s["row_of"].size, np.int32)
    for plen, nf, eos, prow in s["admit"]:
        loop.add_page(plen, nf, eos, s["k"], s["v"], prow)
    row_of = s["row_of"]
    for live, rows, nf, eos in s["steps"]:
        row_of[base + live] = rows
        n, _ = loop.run_step(s["k"], s["v"], s["q"], row_of, s["scale"], s["out"][at:at + s["cap"]],
                             s["lse"][at:at + s["cap"]])
        loop.end_step(nf, eos)
        at += n
    s["first_id"] = base + s["ids"]
    return [s["out"][:at], s["lse"][:at]]


# ------------------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------------------

def _decode_work(case, pages, streams):
    """Each page's visible shared rows once, all private rows once, queries in, outputs out."""
    hkv, hq = case["kv_heads"], GROUP * case["kv_heads"]
    shared = {}
    for p, cut, _ in streams:
        shared[p] = max(shared.get(p, 0), cut)
    kv = sum(shared.values()) + sum(n for _, _, n in streams)
    row = 2 * hkv * (D * 2 if case["kv"] == "bf16" else D + 4 / BS)
    pairs = sum(cut + n for _, cut, n in streams)
    return {"bytes": kv * row + len(streams) * hq * (4 * D + 4), "flops": pairs * hq * 4 * D}


def _pairs(pages):
    """Visible (query, key) pairs of the packed pages."""
    n = 0
    for pg in pages:
        n += pg.stream_len * (pg.stream_len + 1) // 2
        n += sum(b * (pg.prefix_len + f) + b * (b + 1) // 2 for f, b in zip(pg.fork_offset, pg.branch_len))
    return n


def work(case):
    pages, hkv, hq = _pages(case), case["kv_heads"], GROUP * case["kv_heads"]
    t = sum(pg.packed_len for pg in pages)
    kind = case["kind"]
    if kind == "decode":
        return _decode_work(case, pages, _streams(case, pages))
    if kind == "prefill":
        return {"bytes": t * D * 2 * (2 * hq + 2 * hkv) + t * hq * 4, "flops": _pairs(pages) * hq * 4 * D}
    if kind == "backward":
        return {"bytes": t * D * 2 * (4 * hq + 4 * hkv) + t * hq * 4, "flops": _pairs(pages) * hq * 10 * D}
    if kind == "chunk":
        ch = _chunks(case, pages)
        q = sum(n for _, _, _, n in ch)
        kv = sum(max(cut for p, cut, _, _ in ch if p == i) for i in range(len(pages)) if pages[i].num_branches)
        kv += sum(a + n for _, _, a, n in ch)
        pairs = sum(n * (cut + a) + n * (n + 1) // 2 for _, cut, a, n in ch)
        return {"bytes": kv * 4 * hkv * D + q * hq * (4 * D + 4), "flops": pairs * hq * 4 * D}
    if kind == "fill":
        streams = _streams(case, pages)
        blocks = sum(-(-pg.stream_len // BS) for pg in pages) + sum(-(-n // BS) for _, _, n in streams)
        return {"bytes": blocks * hkv * 2 * (BS * D * 3 + 4) + len(streams) * hkv * 2 * D * 3, "flops": 0}
    nbytes = flops = 0
    src = _record(pages)
    lay = np.concatenate([np.concatenate([np.full(pg.stream_len, -1), np.repeat(np.arange(pg.num_branches), pg.branch_len)])
                          for pg in pages])
    start = np.concatenate([[0], np.cumsum([pg.packed_len for pg in pages])])
    for _, rows, _, _ in src[1]:
        page = np.searchsorted(start, rows, side="right") - 1
        pos = rows - start[page]
        streams = []
        for p, j, k in zip(page, pos, lay[rows]):
            pg = pages[p]
            if k < 0:
                streams.append((int(p), int(j) + 1, 0))
            else:
                first = pg.stream_len + sum(pg.branch_len[:k])
                streams.append((int(p), pg.prefix_len + pg.fork_offset[k], int(j - first) + 1))
        w = _decode_work(case, pages, streams)
        nbytes += w["bytes"] + len(streams) * 4 * D * hkv
        flops += w["flops"]
    nbytes += sum(pg.prefix_len for pg in pages) * 8 * D * hkv
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------------------------
# The results in 64 bits
# ------------------------------------------------------------------------------------------------

def _mask(pg):
    """Visible keys of every packed token of a page, [T][T]."""
    t = torch.arange(pg.packed_len, device=DEV)
    m = torch.zeros(pg.packed_len, pg.packed_len, dtype=torch.bool, device=DEV)
    causal = t[None, :] <= t[:, None]
    n = pg.stream_len
    m[:n, :n] = causal[:n, :n]
    for f, b in zip(pg.fork_offset, pg.branch_len):
        m[n:n + b, :pg.prefix_len + f] = True
        m[n:n + b, n:n + b] = causal[n:n + b, n:n + b]
        n += b
    return m


def _attend(q, k, v, m, scale, need_p=False):
    """q [T][8][d] of one KV head's group, k, v [K][d], m [T][K], in 64 bits: (out, lse[, P])."""
    x = torch.einsum("thd,kd->htk", q, k).mul_(scale).masked_fill_(~m[None], -math.inf)
    lse = torch.logsumexp(x, -1)
    p = x.sub_(lse[..., None]).exp_()
    out = torch.einsum("htk,kd->thd", p, v)
    return (out, lse.T, p) if need_p else (out, lse.T)


def exact(case, seed):
    pages, hkv, kind = _pages(case), case["kv_heads"], case["kind"]
    s = prepare(case, seed)
    scale = s["scale"]
    if kind == "fill":
        def scales(x, new):
            f = torch.zeros(x.shape[0], hkv, dtype=torch.float64, device=DEV)
            f[s["dst"].long()] = x.double().abs().amax(dim=(2, 3)) / 448.0
            b = s["slots"].long() // BS
            fresh = (s["slots"] % BS == 0)[:, None]
            f[b] = torch.maximum(torch.where(fresh, torch.zeros_like(f[b]), f[b]), new.double().abs().amax(-1) / 448.0)
            return f
        return [None, None, scales(s["k"], s["k_new"]), scales(s["v"], s["v_new"])]
    if kind in ("prefill", "backward", "loop"):
        q, k, v = s["q"].double(), s["k"].double(), s["v"].double()
        out, lse = torch.empty_like(q), torch.empty(q.shape[:2], dtype=torch.float64, device=DEV)
        dq, dk, dv = torch.empty_like(q), torch.empty_like(k), torch.empty_like(v)
        at = 0
        for pg in pages:
            r, m = slice(at, at + pg.packed_len), _mask(pg)
            for g in range(hkv):
                h = slice(GROUP * g, GROUP * g + GROUP)
                if kind != "backward":
                    out[r, h], lse[r, h] = _attend(q[r, h], k[r, g], v[r, g], m, scale)
                    continue
                o, _, p = _attend(q[r, h], k[r, g], v[r, g], m, scale, True)
                do = s["dout"][r, h].double()
                dv[r, g] = torch.einsum("htk,thd->kd", p, do)
                dp = torch.einsum("thd,kd->htk", do, v[r, g])
                ds = p.mul_(dp.sub_((do * o).sum(-1).T[..., None])).mul_(scale)
                dq[r, h] = torch.einsum("htk,kd->thd", ds, k[r, g])
                dk[r, g] = torch.einsum("htk,thd->kd", ds, q[r, h])
            at += pg.packed_len
        if kind == "backward":
            return [dq, dk, dv]
        if kind == "loop":
            rows = torch.from_numpy(s["rows"]).long().to(DEV)
            return [out[rows], lse[rows]]
        return [out, lse]
    # over the paged cache: the rows of a list of blocks, in order, [rows][Hkv][d] in 64 bits
    if case["kv"] == "e4m3":
        p = s["pool"]
        pools = [c.view(torch.float8_e4m3fn).float().double() * f.double()[:, :, None, None]
                 for c, f in ((p.k_codes, p.k_scales), (p.v_codes, p.v_scales))]
    else:
        pools = [s["k"], s["v"]]
    page_table, stream_table, _ = _tables(case, pages, seed)

    def gather(ids, n):
        b = torch.from_numpy(ids[:-(-n // BS)]).long().to(DEV)
        return [x[b].double().transpose(1, 2).reshape(-1, hkv, D)[:n] for x in pools]

    # (page, shared rows seen, private rows before the first token, tokens, block row) per query run
    if kind == "chunk":
        runs = [(p, cut, a, n, i) for i, (p, cut, a, n) in enumerate(_chunks(case, pages))]
    else:
        runs = [(p, cut, n - 1, 1, i) for i, (p, cut, n) in enumerate(_streams(case, pages))]
    q = s["q"].double()
    out, lse = torch.empty_like(q), torch.empty(q.shape[:2], dtype=torch.float64, device=DEV)
    at, shared_of, shared = 0, None, None
    for p, cut, a, n, i in runs:
        if p != shared_of:
            shared_of, shared = p, gather(page_table[p], pages[p].stream_len)
        own = gather(stream_table[i], max(a + n, 0))
        k, v = (torch.cat([x[:cut], y]) for x, y in zip(shared, own))
        m = torch.ones(n, k.shape[0], dtype=torch.bool, device=DEV)
        if own[0].shape[0]:
            m[:, cut:] = (torch.arange(a + n, device=DEV)[None] <= a + torch.arange(n, device=DEV)[:, None])
        for g in range(hkv):
            h = slice(GROUP * g, GROUP * g + GROUP)
            out[at:at + n, h], lse[at:at + n, h] = _attend(q[at:at + n, h], k[:, g], v[:, g], m, scale)
        at += n
    return [out, lse]
