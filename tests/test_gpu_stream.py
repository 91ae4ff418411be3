"""The score stream and the selections that follow it, where the shapes of its launches change."""
import pytest
import torch

from paper_2602_03152_b200 import binding

pytestmark = pytest.mark.gpu


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
