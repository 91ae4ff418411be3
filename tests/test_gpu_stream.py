"""The score stream and the selections that follow it, where the shapes of its launches change."""
import pytest
import torch

from paper_2602_03152_b200 import binding, synth

from gpu_harness import SENTINEL, Run

pytestmark = pytest.mark.gpu

C = synth.CONFIGS


def _device_us(call, n=20, reps=9):
    """Median device time of a call among n of them, captured once."""
    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(n):
            call()
    times = []
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) / n * 1e3)
    return sorted(times)[reps // 2]


def test_short_sequences_in_a_long_cache_are_scored_as_in_a_short_one():
    # What the stream takes goes by the lengths, not by max_len: 4000 tokens of 16 sequences in caches of 4096 and of
    # 65536: 8.2 and 10.2 us.  (Shares of max_len put all of a sequence on two CTAs while the others read where nothing is: 21.3.)
    us = {}
    for max_len in (4096, 65536):
        B, T, H = 16, 3, 8
        f = binding.Fasa(B, 4 * H, H, max_len, torch.arange(16, dtype=torch.int32).repeat(H, 1))
        proxy = f.alloc_proxy()
        q = torch.ones((B, T, 4 * H, 128), dtype=torch.bfloat16, device="cuda")
        lens = torch.full((B,), 4000, dtype=torch.int32, device="cuda")
        scores = torch.empty((B, T, H, max_len), dtype=torch.float32, device="cuda")
        us[max_len] = _device_us(lambda: f.fc_score_batched(q, proxy, lens, scores))
        del proxy, scores
    assert us[65536] <= 1.8 * us[4096], us


@pytest.mark.parametrize("B,H,max_len,n,launches", [
    (34, 8, 8704, 256, 1),      # 272 clusters of one CTA, two to an SM: one round that leaves nothing to even out
    (34, 8, 8704, 128, 2),
    (18, 8, 17408, 512, 1),     # 144 clusters of two
    (18, 8, 17408, 256, 2),
    (20, 8, 8704, 512, 2),      # 160 clusters of one: some SMs with two CTAs, others with one
    (20, 8, 8704, 1024, 1),
    (48, 8, 8704, 1024, 1),     # rounds of clusters of one
    (48, 8, 4352, 512, 2),
])
def test_default_sets_take_two_launches_only_where_they_gain(B, H, max_len, n, launches):
    f = binding.Fasa(B, 4 * H, H, max_len, torch.arange(16, dtype=torch.int32).repeat(H, 1))
    k = torch.zeros((B, H, max_len, 128), dtype=torch.bfloat16, device="cuda")
    q = torch.ones((B, 4 * H, 128), dtype=torch.bfloat16, device="cuda")
    idx, n_sel = torch.empty((B, H, n), dtype=torch.int32, device="cuda"), torch.empty((B, H), dtype=torch.int32, device="cuda")
    lens = torch.full((B,), max_len // 2, dtype=torch.int32, device="cuda")
    n0 = f.launch_count()
    f.decode_step(q, k, k, f.alloc_proxy(), lens, n, None, idx, n_sel, torch.empty((B, 4 * H, 128), device="cuda"), f.alloc_workspace(n))
    assert f.launch_count() - n0 == launches


def test_workspace_of_a_page_pool_goes_by_what_it_holds():
    # sequences of up to 32 K, 24 of them, in a pool of a quarter of that: partial results alone, not 4 bytes to a position
    B, H, max_len, page, T, n = 24, 8, 32768, 64, 3, 256
    dom = torch.arange(16, dtype=torch.int32).repeat(H, 1)
    f = [binding.Fasa(B, 4 * H, H, max_len, dom, page_size=page, n_pages=p) for p in (B * max_len // page // 4, B * max_len // page)]
    rows = B * H * max_len * 4
    small, large = (x.workspace_bytes(n) for x in f)
    assert small < 2 * B * 4 * H * 130 * 4 * (max_len // 2048) < rows and large >= rows
    # and what it does without changes no result
    pages = f[0].n_pages
    g = torch.Generator(device="cuda").manual_seed(3)
    k, v = ((0.5 * torch.randn((pages, H, page, 128), generator=g, device="cuda")).to(torch.bfloat16) for _ in range(2))
    q = torch.randn((B, T, 4 * H, 128), generator=g, device="cuda").to(torch.bfloat16)
    lens = torch.randint(5000, max_len // 4, (B,), generator=g, device="cuda").to(torch.int32)
    table = torch.zeros((B, max_len // page), dtype=torch.int32, device="cuda")
    table[:, :max_len // 4 // page] = torch.randperm(pages, generator=g, device="cuda").to(torch.int32).view(B, -1)
    got = []
    for x in f:
        x.set_block_table(table)
        proxy = x.alloc_proxy()
        kk, vv = k, v
        if x.n_pages > pages:
            kk, vv = (torch.cat([y, torch.zeros((x.n_pages - pages, H, page, 128), dtype=torch.bfloat16, device="cuda")]) for y in (k, v))
        x.proxy_build(kk, proxy, lens)
        ws = x.alloc_workspace(n)
        o = [torch.zeros((B, T, H, max_len), device="cuda"), torch.zeros((B, T, H, n), dtype=torch.int32, device="cuda"),
             torch.zeros((B, T, H), dtype=torch.int32, device="cuda"), torch.zeros((B, T, 4 * H, 128), device="cuda")]
        s = [torch.zeros((B, H, max_len), device="cuda"), torch.zeros((B, H, n), dtype=torch.int32, device="cuda"),
             torch.zeros((B, H), dtype=torch.int32, device="cuda"), torch.zeros((B, 4 * H, 128), device="cuda")]
        x.decode_step_batched(q, kk, vv, proxy, lens, n, *o, ws)
        x.decode_step(q[:, 0].contiguous(), kk, vv, proxy, lens, n, *s, ws)
        torch.cuda.synchronize()
        assert x.device_status() == 0
        got.append(o + s)
        del kk, vv, proxy
    for i, (a, b) in enumerate(zip(*got)):
        assert torch.equal(a, b) if i % 4 < 3 else float((a - b).abs().max()) <= 1e-5


def _score_bounds(r, q, t, T):
    """Scores of query t in fp64 and the sums of the products' magnitudes, [batch][kv heads][max_len]."""
    w = r.w
    B, H, G = w.batch, w.n_kv_heads, w.group
    ref = torch.empty((B, H, w.max_len), dtype=torch.float64, device="cuda")
    mag = torch.empty_like(ref)
    c0 = r.dom.long() if w.pairing == 0 else 2 * r.dom.long()
    chan = torch.cat([c0, c0 + (64 if w.pairing == 0 else 1)], dim=1).cuda()          # [kv heads][2 F]
    for b in range(B):
        for h in range(H):
            kk = r.k[b, h][:, chan[h]].double()
            qq = q[b, t, h * G:(h + 1) * G][:, chan[h]].double()
            s, m = kk @ qq.T, kk.abs() @ qq.abs().T
            ref[b, h] = s.max(1).values if w.group_reduce else s.sum(1)
            mag[b, h] = m.max(1).values if w.group_reduce else m.sum(1)
    return ref, mag


# Blocks whose warps take several iterations (a share of 3 to 12), ending anywhere in one; the number of rows and max_len decide
# the thread block of the selection that takes the stream's maxima: 1024, 512 or 256 threads.
@pytest.mark.parametrize("kw,T,page", [
    (dict(batch=24, n_q_heads=16, n_dom=8, max_len=4001, budget=256, n_sink=3, n_recent=13), 3, 0),    # 576 rows, misaligned: eight listed positions to a thread of 256
    (dict(batch=24, n_q_heads=32, n_dom=16, max_len=4000, budget=100), 5, 0),                          # groups of 8, chunks of 32 at 256 threads
    (dict(batch=24, n_q_heads=16, n_dom=16, max_len=4096, budget=300, n_sink=40), 8, 64),
    (dict(batch=20, n_q_heads=48, n_dom=32, max_len=4000, budget=64, group_reduce=1), 2, 0),           # three pairs of heads, max
    (dict(batch=20, n_q_heads=56, n_dom=28, max_len=4096, budget=64), 4, 16),                          # four pairs, seven chunks, pages of one tile
    (dict(batch=20, n_q_heads=64, n_dom=64, max_len=4000, budget=3), 3, 0),                            # one tile in registers; groups of 32
    (dict(batch=24, n_q_heads=24, n_dom=64, max_len=3999, budget=200, n_recent=70), 2, 0),             # odd group
    (dict(batch=24, n_q_heads=8, n_dom=4, max_len=8000, budget=500, pairing=1), 2, 0),                 # one head to a set
    (dict(batch=2, n_q_heads=16, n_kv_heads=4, n_dom=16, max_len=20003, budget=700, n_sink=5, n_recent=9), 5, 0),   # 40 rows: 1024 threads
    (dict(batch=6, n_q_heads=28, n_kv_heads=4, n_dom=8, max_len=20000, budget=512), 6, 0),             # 144 rows
    (dict(batch=1, n_q_heads=32, n_dom=16, max_len=66003, budget=512, n_sink=4, n_recent=64), 5, 0),   # beyond 65536: groups of 32
    (dict(batch=5, n_q_heads=32, n_dom=16, max_len=66000, budget=800), 4, 0),                          # 160 rows
])
def test_blocks_whose_warps_take_several_iterations(kw, T, page):
    base = dict(n_kv_heads=8, len_lo=kw["max_len"] // 3, len_hi=kw["max_len"], n_sink=0, n_recent=0)
    w = C["c1"].replace(**dict(base, **kw))
    t = synth.make_inputs(w.replace(rope=False), "cuda")
    t["seq_lens"][0], t["seq_lens"][-1] = w.max_len, T + 1
    r = Run(w, t)
    f, k, v = r.fasa, r.k, r.v
    B, Hs = w.batch, w.n_sets
    if page:
        n = w.max_len // page
        f = binding.Fasa(B, w.n_q_heads, w.n_kv_heads, w.max_len, r.dom, rope_pairing=w.pairing, group_reduce=w.group_reduce,
                         n_sink=w.n_sink, n_recent=w.n_recent, page_size=page, n_pages=B * n)
        table = torch.randperm(B * n, generator=torch.Generator(device="cuda").manual_seed(5), device="cuda").to(torch.int32).view(B, n)
        f.set_block_table(table)
        pool = [torch.empty((B * n, w.n_kv_heads, page, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        for p, c in zip(pool, (r.k, r.v)):
            p[table.reshape(-1).long()] = c.view(B, w.n_kv_heads, n, page, 128).transpose(1, 2).reshape(-1, w.n_kv_heads, page, 128)
        k, v = pool
    proxy = f.alloc_proxy()
    f.proxy_build(k, proxy, r.seq_lens)
    q = torch.stack([synth.make_step_inputs(w, i, "cuda")["q"] for i in range(T)], dim=1).contiguous()
    scores = torch.full((B, T, Hs, w.max_len), SENTINEL, dtype=torch.float32, device="cuda")
    o = [torch.full((B, T, Hs, r.n_sel_max), -7, dtype=torch.int32, device="cuda"), torch.full((B, T, Hs), -7, dtype=torch.int32, device="cuda"),
         torch.full((B, T, w.n_q_heads, 128), SENTINEL, dtype=torch.float32, device="cuda")]
    o2 = [x.clone() for x in o]
    ws = f.alloc_workspace(r.n_sel_max)
    f.decode_step_batched(q, k, v, proxy, r.seq_lens, w.budget, scores, *o, ws)
    for i in range(T):
        lens = (r.seq_lens - (T - 1 - i)).clamp(min=0)
        seen = torch.arange(w.max_len, device="cuda") < lens.view(B, 1, 1)
        ref, mag = _score_bounds(r, q, i, T)
        assert torch.all((scores[:, i] == SENTINEL) == ~seen.expand(B, Hs, -1))
        # (a sum of at most 2 F bf16 products to a head, then of the heads, each addition rounded in fp32: 136 roundings of 2^-24)
        assert torch.all(((scores[:, i].double() - ref).abs() <= 1e-5 * mag) | ~seen)
    # the selection without the stream's maxima, and its attention, from the same scores
    f.topk_batched(scores, r.seq_lens, w.budget, *o2[:2])
    f.sparse_decode_attn_batched(q, k, v, *o2[:2], o2[2], ws)
    for x, y in zip(o, o2):
        assert torch.equal(x, y)
    assert f.device_status() == 0


# Where a thread takes a listed group of eight: 1024, 512 and 256 threads, rows that are aligned or not, groups that the forced
# positions cut.
@pytest.mark.parametrize("B,H,L,k", [(4, 8, 20003, 1500), (4, 8, 20004, 1500), (20, 8, 9001, 700), (20, 8, 9004, 700), (40, 8, 5001, 300), (40, 8, 5004, 300)])
@pytest.mark.parametrize("n_sink,n_recent", [(0, 0), (3, 13)])
def test_listed_groups_of_rows_that_are_not_aligned(B, H, L, k, n_sink, n_recent):
    g = torch.Generator(device="cuda").manual_seed(L)
    scores = torch.randn((B, H, L), generator=g, device="cuda")
    f = binding.Fasa(B, H, H, L, torch.arange(4, dtype=torch.int32).repeat(H, 1), n_sink=n_sink, n_recent=n_recent)
    f.set_step_mode(2)
    lens = torch.randint(12 * k + 100, L + 1, (B,), generator=g, device="cuda").to(torch.int32)
    lens[0], lens[1] = L, L - 1
    n = k + n_sink + n_recent
    idx, n_sel = torch.empty((B, H, n), dtype=torch.int32, device="cuda"), torch.empty((B, H), dtype=torch.int32, device="cuda")
    f.topk(scores, lens, k, idx, n_sel)
    at = torch.arange(L, device="cuda").view(1, 1, L)
    end = lens.view(B, 1, 1)
    forced = (at < end) & ((at < n_sink) | (at >= end - n_recent))
    key = torch.where(at < end, torch.where(forced, torch.inf, scores), -torch.inf)
    ref = torch.sort(torch.sort(key, dim=2, descending=True, stable=True).indices[:, :, :n], dim=2).values.to(torch.int32)
    assert torch.equal(idx, ref) and torch.all(n_sel == n)


def test_few_sets_of_long_rows_leave_the_selection_to_clusters():
    # 16 sets of 35 K in caches of 142 K, 512 of each: a step that selects whole rows with one CTA each takes 55 us, the cluster
    # kernel's selection and the attention of its lists 39
    B, H, max_len, n = 2, 8, 142710, 512
    g = torch.Generator(device="cuda").manual_seed(9)
    f = binding.Fasa(B, 4 * H, H, max_len, torch.arange(8, dtype=torch.int32).repeat(H, 1))
    k, v = (torch.randn((B, H, max_len, 128), generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    q = torch.randn((B, 4 * H, 128), generator=g, device="cuda", dtype=torch.bfloat16)
    lens = torch.tensor([35000, 34000], dtype=torch.int32, device="cuda")
    proxy, ws = f.alloc_proxy(), f.alloc_workspace(n)
    f.proxy_build(k, proxy, lens)
    idx, n_sel = torch.empty((B, H, n), dtype=torch.int32, device="cuda"), torch.empty((B, H), dtype=torch.int32, device="cuda")
    out = torch.empty((B, 4 * H, 128), device="cuda")
    step = _device_us(lambda: f.decode_step(q, k, v, proxy, lens, n, None, idx, n_sel, out, ws))

    def apart():
        f.select_step(q, k, v, proxy, lens, n, None, idx, n_sel)
        f.sparse_decode_attn(q, k, v, idx, n_sel, out, ws)
    apart = _device_us(apart)
    assert step <= 1.2 * apart, (step, apart)


@pytest.mark.parametrize("rows,L,budgets", [
    ((4, 8), 65536, (255, 256)),            # a cluster each from here on
    ((5, 8), 50001, (255, 256)),            # where rows are not aligned
    ((9, 8), 40001, (2047, 2048)),
    ((6, 8), 66001, (255, 256)),
    ((4, 8), 66000, (64, 128)),
    ((8, 8), 40000, (2047, 2048)),
    ((9, 8), 40000, (4095, 4096)),
    ((9, 8), 66000, (2047, 2048)),
])
@pytest.mark.parametrize("outliers", [0, 1])
def test_topk_where_the_route_of_its_rows_changes(rows, L, budgets, outliers):
    B, H = rows
    g = torch.Generator(device="cuda").manual_seed(L + B)
    scores = torch.randn((B, H, L), generator=g, device="cuda")
    if outliers:                            # one in 500 far above the others
        scores[torch.rand(scores.shape, generator=g, device="cuda") < 0.002] *= 30
    f = binding.Fasa(B, H, H, L, torch.arange(4, dtype=torch.int32).repeat(H, 1))
    lens = torch.full((B,), L, dtype=torch.int32, device="cuda")
    order = torch.sort(scores, dim=2, descending=True, stable=True).indices
    for k in budgets:
        ref = torch.sort(order[:, :, :k], dim=2).values.to(torch.int32)
        for mode in (1, 2):
            f.set_step_mode(mode)
            idx, n_sel = torch.empty((B, H, k), dtype=torch.int32, device="cuda"), torch.empty((B, H), dtype=torch.int32, device="cuda")
            f.topk(scores, lens, k, idx, n_sel)
            assert torch.equal(idx, ref) and torch.all(n_sel == k)
