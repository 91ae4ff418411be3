"""What a user of this framework has it do, for timing: decode steps of every kind, and the calls around them.

A case is a dict of plain values: its `kind` names the entry points that a pass goes through, the rest are the
sizes and options of the context (`paper_2602_03152_b200.binding.Fasa`).  Kinds:

  step      append one token per sequence and decode it (`append_decode_step`), the call of a generation loop
  calls     `fc_score`, `topk`, `sparse_decode_attn` one after another, for programs that keep the scores
  block     a block of query tokens (speculative decoding): roll back to the accepted length, append the
            block's rows (`kv_append`), then `decode_step_batched`
  dense     `full_decode_attn`, for layers that stay dense
  prompt    a new request in a slot: length to zero, `kv_append` of the prompt's rows
  offload   `m_decode_step`: keys split, non-dominant channels and values in page-locked host memory
  calib     `calib_accumulate` of one batch of samples

Sequences of a "step" grow by a token per pass, as they do in generation; max_len leaves them room.
Inputs follow `synth` (log-normal channel scales, outlier channels, RoPE at true positions).
"""
import math

import torch

from paper_2602_03152_b200 import binding, synth

DEFAULTS = dict(n_dom=16, budget=256, n_sink=0, n_recent=0, pairing=0, group_reduce=0, sel_heads=0,
                page_size=0, q_len=1, rows=0)


def case(kind, batch, q_heads, kv_heads, max_len, len_lo, len_hi, **options):
    return dict(DEFAULTS, kind=kind, batch=batch, n_q_heads=q_heads, n_kv_heads=kv_heads, max_len=max_len,
                len_lo=len_lo, len_hi=len_hi, **options)


def listed():
    return [
        # the smallest: one KV head's cache of 4 K tokens, three small launches
        dict(case("calls", 1, 4, 1, 4096, 4096, 4096, n_dom=8), name="calls_1head_4k"),
        # one user at a Llama-3-8B-like layer, with sinks and a recent window
        dict(case("step", 1, 32, 8, 32768, 19000, 19000, n_sink=4, n_recent=64), name="step_b1_32k"),
        # a small server batch at the same layer
        dict(case("step", 8, 32, 8, 65536, 57000, 57000), name="step_b8_64k"),
        # the largest: long contexts of different lengths
        dict(case("step", 16, 32, 8, 131072, 65536, 126000, budget=1024), name="step_b16_128k_ragged"),
        # long chain-of-thought decoding at a Qwen2.5-7B-like layer: groups of 7 heads, budget 18.9 % of the length
        dict(case("step", 32, 28, 4, 16384, 9000, 9000, budget=-189), name="step_b32_g7_longcot"),
        # a serving engine's paged caches, 64-token pages in any order
        dict(case("step", 12, 32, 8, 32768, 3001, 28001, budget=512, page_size=64), name="step_b12_paged"),
        # the paper's own reading: an index set per query head
        dict(case("step", 4, 32, 8, 65536, 30011, 56003, sel_heads=1), name="step_b4_set_per_head"),
        # five-token blocks of speculative decoding
        dict(case("block", 8, 32, 8, 65536, 40000, 65000, budget=512, q_len=5), name="block_b8_q5_64k"),
        # a dense layer beside the sparse ones
        dict(case("dense", 4, 32, 8, 65536, 20003, 60007), name="dense_b4_64k"),
        # four prompts enter the caches
        dict(case("prompt", 4, 32, 8, 8192, 0, 0, rows=3001), name="prompt_b4_3001"),
        # caches in host memory, forced rows resident on the GPU
        dict(case("offload", 2, 32, 8, 32768, 20001, 30001, n_sink=4, n_recent=64), name="offload_b2_32k"),
        # offline calibration of the dominant chunks, 32 samples
        dict(case("calib", 1, 32, 8, 32768, 24001, 24001), name="calib_b1_32k"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges: mostly decode steps, at most as large as the largest listed ones."""
    kind = rng.choice(["step"] * 6 + ["calls", "block", "dense", "prompt", "offload", "calib"])
    q_heads, kv_heads = rng.choice([(32, 8), (32, 8), (28, 4), (16, 8), (40, 8)])
    options = dict(n_dom=rng.choice([4, 8, 12, 16, 16, 16, 24, 32, 64]), budget=rng.choice([64, 128, 256, 512, 1024, 2048, -189]))
    if rng.random() < 0.3:
        options.update(n_sink=4, n_recent=64)
    if kind == "calib":
        options.update(budget=rng.choice([128, 256, 512]))
        hi = _log(rng, 2048, 24000)
        return case(kind, 1, q_heads, kv_heads, hi + rng.randrange(512), hi // 2, hi, **options)
    if kind == "prompt":
        rows = _log(rng, 64, 4096)
        return case(kind, _log(rng, 1, min(16, 16384 // rows)), q_heads, kv_heads, 8192, 0, 0, rows=rows, **options)
    if kind == "offload":
        options.update(n_dom=rng.choice([8, 16, 32]), budget=rng.choice([128, 256, 512]))
        hi = _log(rng, 4096, 30000)
        return case(kind, rng.choice([1, 2]), q_heads, kv_heads, hi + 8192, hi * 2 // 3, hi, **options)
    batch = _log(rng, 1, 32)
    hi = _log(rng, 2048, 120000)
    cap = {"calls": 1 << 20, "step": 1 << 20, "block": 1 << 19, "dense": 1 << 18}[kind]      # tokens of all sequences
    if options["n_dom"] > 16:
        cap = cap * 16 // options["n_dom"]
    if kind == "step" and rng.random() < 0.15:
        options.update(sel_heads=1)
        cap //= 4
    elif kind == "step" and rng.random() < 0.2:
        options.update(page_size=rng.choice([16, 64, 256]))
    if kind == "block":
        options.update(q_len=rng.randint(2, 8), budget=rng.choice([128, 256, 512]))
    if kind == "calls":
        options.update(pairing=rng.choice([0, 1]), group_reduce=rng.choice([0, 1]))
    hi = max(1024, min(hi, cap // batch))
    lo = rng.randint(hi // 2, hi)
    max_len = hi + max(4096, hi // 8)
    if options.get("page_size"):
        max_len = -(-max_len // options["page_size"]) * options["page_size"]
    c = case(kind, batch, q_heads, kv_heads, max_len, lo, hi, **options)
    while work(c)["bytes"] > 8e8 and c["batch"] > 1:
        c["batch"] -= max(1, c["batch"] // 8)
    return c


def _workload(c, seed, **over):
    w = synth.Workload("case", seed, c["batch"], c["n_q_heads"], c["n_kv_heads"], c["max_len"], c["len_lo"], c["len_hi"],
                       c["n_dom"], c["budget"], c["n_sink"], c["n_recent"], pairing=c["pairing"],
                       group_reduce=c["group_reduce"], sel_heads=c["sel_heads"])
    return w.replace(**over) if over else w


def _n_sel_max(c, length):
    k = c["budget"] if c["budget"] > 0 else (-c["budget"] * length + 999) // 1000
    return min(c["max_len"], k + c["n_sink"] + c["n_recent"])


def _paged(cache, page, table):
    """The pool [n_pages, kv heads, page, 128] that holds a contiguous cache behind the block table."""
    B, H, L, d = cache.shape
    pool = torch.empty((B * (L // page), H, page, d), dtype=cache.dtype, device=cache.device)
    pool[table.reshape(-1).long()] = cache.view(B, H, L // page, page, d).transpose(1, 2).reshape(-1, H, page, d)
    return pool


def prepare(c, seed):
    dev, kind = torch.device("cuda"), c["kind"]
    if kind == "prompt":
        w = _workload(c, seed, max_len=c["rows"], len_lo=c["rows"], len_hi=c["rows"])
        t = synth.make_inputs(w, dev)
        f = binding.Fasa.from_workload(_workload(c, seed), t["dom"])
        shape = (c["batch"], c["n_kv_heads"], c["max_len"], 128)
        return dict(kind=kind, f=f, k_new=t["k"], v_new=t["v"], k=torch.zeros(shape, dtype=torch.bfloat16, device=dev),
                    v=torch.zeros(shape, dtype=torch.bfloat16, device=dev), proxy=f.alloc_proxy(),
                    lens=torch.zeros(c["batch"], dtype=torch.int32, device=dev))
    w = _workload(c, seed)
    t = synth.make_inputs(w, dev)
    new = synth.make_step_inputs(w, 0, dev)
    page = c["page_size"]
    f = binding.Fasa(w.batch, w.n_q_heads, w.n_kv_heads, w.max_len, t["dom"], rope_pairing=w.pairing,
                     group_reduce=w.group_reduce, n_sink=w.n_sink, n_recent=w.n_recent, select_heads=w.sel_heads,
                     page_size=page, n_pages=w.batch * (w.max_len // page) if page else 0)
    s = dict(kind=kind, f=f, q=t["q"], k=t["k"], v=t["v"], lens=t["seq_lens"], budget=w.budget)
    if kind == "calib":
        s.update(top_k=w.budget if w.budget > 0 else 256,
                 counts=torch.zeros((w.n_q_heads, 64), dtype=torch.int64, device=dev),
                 used=torch.zeros(w.n_q_heads, dtype=torch.int64, device=dev))
        s.update(ws=torch.empty(f.calib_workspace_bytes(s["top_k"]), dtype=torch.uint8, device=dev))
        return s
    # a generation loop bounds its selections at the length that it will have reached a few thousand tokens on
    n_sel_max = _n_sel_max(c, min(w.max_len, c["len_hi"] + 4096))
    rows = (w.batch, c["q_len"]) if kind == "block" else (w.batch,)
    s.update(idx=torch.zeros(rows + (f.n_sets, n_sel_max), dtype=torch.int32, device=dev),
             n_sel=torch.zeros(rows + (f.n_sets,), dtype=torch.int32, device=dev),
             out=torch.zeros(rows + (w.n_q_heads, 128), dtype=torch.float32, device=dev),
             lse=torch.zeros(rows + (w.n_q_heads,), dtype=torch.float32, device=dev), ws=f.alloc_workspace(n_sel_max))
    if kind == "dense":
        return s
    if page:
        g = torch.Generator(device=dev).manual_seed(seed)
        table = torch.randperm(w.batch * (w.max_len // page), generator=g, device=dev).to(torch.int32).view(w.batch, -1)
        f.set_block_table(table)
        s.update(k=_paged(s["k"], page, table), v=_paged(s["v"], page, table), table=table)
    s.update(proxy=f.alloc_proxy(), k_new=new["k_new"], v_new=new["v_new"])
    f.proxy_build(s["k"], s["proxy"], s["lens"])
    if kind in ("calls", "block"):
        s.update(scores=torch.zeros(rows + (f.n_sets, w.max_len), dtype=torch.float32, device=dev))
    if kind == "block":
        T = c["q_len"]
        blocks = [synth.make_step_inputs(w, i, dev) for i in range(T)]
        s.update(q=torch.stack([x["q"] for x in blocks], 1), accepted=s["lens"].clone(),
                 k_new=torch.cat([x["k_new"] for x in blocks], 2), v_new=torch.cat([x["v_new"] for x in blocks], 2))
    if kind == "offload":
        k_nondom, v_host = f.alloc_host_nondom(), f.alloc_host_cache()
        f.m_split(s["k"], k_nondom, s["lens"])
        v_host.copy_(s["v"])
        s.update(k=k_nondom, v=v_host)
        if w.n_sink + w.n_recent:
            s.update(resident=f.alloc_resident())
            f.m_resident_build(k_nondom, v_host, s["proxy"], s["lens"])
    return s


def run(s):
    f, kind = s["f"], s["kind"]
    if kind == "step":
        f.append_decode_step(s["q"], s["k_new"], s["v_new"], s["k"], s["v"], s["proxy"], s["lens"], s["budget"], None,
                             s["idx"], s["n_sel"], s["out"], s["ws"])
        return [s[n] for n in ("out", "idx", "n_sel", "lens", "k", "v", "proxy")]
    if kind == "calls":
        f.fc_score(s["q"], s["proxy"], s["lens"], s["scores"])
        f.topk(s["scores"], s["lens"], s["budget"], s["idx"], s["n_sel"], s["ws"])
        f.sparse_decode_attn(s["q"], s["k"], s["v"], s["idx"], s["n_sel"], s["out"], s["ws"], s["lse"])
        return [s[n] for n in ("out", "lse", "idx", "n_sel", "scores")]
    if kind == "block":
        s["lens"].copy_(s["accepted"])
        f.kv_append(s["k"], s["v"], s["proxy"], s["lens"], s["k_new"], s["v_new"])
        f.decode_step_batched(s["q"], s["k"], s["v"], s["proxy"], s["lens"], s["budget"], s["scores"], s["idx"],
                              s["n_sel"], s["out"], s["ws"])
        return [s[n] for n in ("out", "idx", "n_sel", "scores", "lens", "k", "v", "proxy")]
    if kind == "dense":
        f.full_decode_attn(s["q"], s["k"], s["v"], s["lens"], s["out"], s["ws"], s["lse"])
        return [s["out"], s["lse"]]
    if kind == "prompt":
        s["lens"].zero_()
        f.kv_append(s["k"], s["v"], s["proxy"], s["lens"], s["k_new"], s["v_new"])
        return [s[n] for n in ("k", "v", "proxy", "lens")]
    if kind == "offload":
        f.m_decode_step(s["q"], s["k"], s["v"], s["proxy"], s["lens"], s["budget"], None, s["idx"], s["n_sel"], s["out"],
                        s["ws"], None, s["k_new"], s["v_new"])
        return [s[n] for n in ("out", "idx", "n_sel", "lens", "k", "v", "proxy")]
    f.calib_accumulate(s["q"], s["k"], s["lens"], s["top_k"], s["counts"], s["used"], s["ws"])
    return [s["counts"], s["used"]]


def work(c):
    """Bytes and operations of one pass at the mean length: the proxy once per KV head, the K and V rows of every
    index set, scores and lists where they are results, queries, outputs and appended rows."""
    B, Hq, Hkv, T, F = c["batch"], c["n_q_heads"], c["n_kv_heads"], c["q_len"], c["n_dom"]
    L = (c["len_lo"] + c["len_hi"]) / 2
    sets = Hq // c["sel_heads"] if c["sel_heads"] else Hkv
    if c["kind"] == "prompt":
        return {"bytes": B * Hkv * c["rows"] * (4 * 256 + 4 * F), "flops": 0}
    if c["kind"] == "calib":
        return {"bytes": B * Hkv * L * 256 + B * Hq * (256 + 64 * 8), "flops": B * Hq * L * 256}
    if c["kind"] == "dense":
        return {"bytes": B * Hkv * L * 512 + B * Hq * (256 + 516), "flops": B * Hq * L * 512}
    n = min(L, _n_sel_max(c, int(L)))
    by = B * Hkv * L * 4 * F + B * T * sets * n * (512 + 4) + B * T * Hq * (256 + 512)
    if c["kind"] in ("calls", "block"):
        by += B * T * sets * L * 4
    if c["kind"] != "calls":
        by += B * T * Hkv * (4 * 256 + 4 * F)
    return {"bytes": by, "flops": B * T * Hq * (L * 4 * F + n * 512)}


def tolerance(c):
    """Attention outputs against double precision on the same rows: 3e-7 to 2e-6 measured (the probabilities of the
    tensor-core path carry 17 bits), single values off by up to 5e-5 of the root mean square.  Two scores that differ
    in their last bit may swap at the edge of one list, which shifts part of that list."""
    if c["kind"] in ("prompt", "calib"):
        return "exact"
    return {"rel": 1e-5, "max": 2e-4, "differ": 0.01}
