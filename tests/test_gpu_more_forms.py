"""Forms of the scoring calls beside one contiguous prompt in one call: key shards, batches, 8-bit keys, streams.  Against the
general path or the same prompts one by one; a logit's error is that of test_gpu_kernel_edges, a log-sum-exp's no larger."""
import pytest
import torch

from test_gpu_kernel_edges import SPAN, make

pytestmark = pytest.mark.gpu


def out(L, Hq, m, n):
    return torch.full((n,), -1.0, device="cuda"), torch.full((L, Hq, m), -1.0, device="cuda")


def scratch(size):
    return torch.empty(size, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("L,Hq,Hkv,d,m,n", [
    (16, 32, 8, 64, 8, 4001), (16, 32, 8, 64, 8, 60001), (16, 32, 8, 64, 8, 100100),      # groups of 8, 67 and 132 CTAs; 4, 7, 6 tiles
    (12, 16, 8, 128, 8, 60001), (8, 32, 8, 64, 8, 9 * SPAN - 300), (6, 24, 8, 128, 8, 20011), (8, 16, 4, 64, 16, 30001),
    (4, 8, 2, 128, 8, 9 * SPAN - 50), (4, 4, 2, 64, 16, 5 * SPAN - 50), (4, 2, 2, 64, 16, 10 * SPAN - 50)])     # maxima in tensor memory
def test_shards_through_many_rounds_of_every_ring(L, Hq, Hkv, d, m, n):
    """One visit alone: stages are freed by the sum warps (first call), or waited for without a sum pass (second)."""
    import paper_2603_02631_b200 as spf
    q, k = make(L, Hq, Hkv, d, m, n)
    importance, lse = out(L, Hq, m, n)
    want_i, want_l = out(L, Hq, m, n)
    p, w = spf.PromptBuffers(q, k, importance, lse), spf.PromptBuffers(q, k, want_i, want_l)
    ws, status = scratch(spf.spf_score_workspace_bytes([p])), torch.zeros(1, dtype=torch.int32, device="cuda")
    spf.spf_score_shard_lse(w, ws)
    for _ in range(2):
        spf.spf_score_shard_lse_ex(p, ws, status)
        torch.testing.assert_close(lse, want_l, rtol=0, atol=1e-4)
    spf.spf_score_shard_apply(w, want_l, ws)
    spf.spf_score_shard_apply_ex(p, want_l, ws, status)
    torch.testing.assert_close(importance, want_i, rtol=2e-4, atol=0)
    assert int(status) == 0


@pytest.mark.parametrize("L,Hq,Hkv,d,m,n", [
    (40, 32, 8, 64, 8, 600), (16, 16, 8, 64, 8, 20 * 128),                                # a tile a CTA, 320 and 128 slabs; 32 and 16 rows
    (16, 32, 8, 64, 8, 50000), (16, 32, 8, 64, 8, 8 * SPAN - 50),                         # maxima in registers; groups that gather, owners
    (8, 16, 8, 64, 16, 4 * SPAN - 50), (8, 32, 8, 128, 8, 9 * SPAN - 50), (8, 8, 4, 128, 8, 12 * SPAN - 50)])   # in tensor memory
def test_repeated_passes_bring_the_same_bits(L, Hq, Hkv, d, m, n):
    """Every stage of tensor memory is filled, summed, folded and filled again many times a pass; sums are taken in a fixed order and
    maxima are exact, so a load that saw another round's logits shows as a difference."""
    import paper_2603_02631_b200 as spf
    q, k = make(L, Hq, Hkv, d, m, n)
    first, again = out(L, Hq, m, n), out(L, Hq, m, n)
    p, r = spf.PromptBuffers(q, k, *first), spf.PromptBuffers(q, k, *again)
    ws, status = scratch(spf.spf_score_workspace_bytes([p])), torch.zeros(1, dtype=torch.int32, device="cuda")
    spf.spf_score([p], ws, dev_status=status)
    for _ in range(20):
        spf.spf_score([r], ws, dev_status=status)
        assert torch.equal(first[0], again[0]) and torch.equal(first[1], again[1])
    spf.spf_score_shard_lse_ex(r, ws, status)
    spf.spf_score_shard_apply_ex(r, again[1], ws, status)            # the log-sum-exps went through base e: half a unit each way
    torch.testing.assert_close(again[0], first[0], rtol=1e-5, atol=0)
    assert int(status) == 0


LENS = [1, 5000, 130, 700, 2048, 12000, 257]


@pytest.mark.parametrize("geom", [(3, 8, 2, 64, 16), (3, 16, 2, 128, 8), (2, 6, 2, 64, 8)])     # 64, 64 and 32 rows
@pytest.mark.parametrize("form", ["flat", "strided", "paged", "fp8"])
def test_batches_of_every_form_equal_their_prompts(geom, form):
    import paper_2603_02631_b200 as spf
    L, Hq, Hkv, d, m = geom
    size, score = {"paged": (spf.spf_score_paged_workspace_bytes, spf.spf_score_paged),
                   "fp8": (spf.spf_score_fp8_workspace_bytes, spf.spf_score_fp8)}.get(form, (spf.spf_score_workspace_bytes, spf.spf_score))
    bufs = []
    for i, n in enumerate(LENS):
        q, k = make(L, Hq, Hkv, d, m, n, seed=i)
        if form == "fp8":
            k = [x.float().to(torch.float8_e4m3fn).view(torch.uint8) for x in k]
            bufs.append(spf.Fp8PromptBuffers(q, k, torch.rand(L, Hkv, device="cuda") + 0.5, *out(L, Hq, m, n)))
        elif form == "paged":
            blocks = -(-n // 128)
            table = torch.randperm(blocks + 2, device="cuda")[:blocks]
            pools = []
            for x in k:
                pool = torch.zeros(blocks + 2, Hkv, 128, d, dtype=torch.bfloat16, device="cuda")
                pool[table] = torch.nn.functional.pad(x, (0, 0, 0, blocks * 128 - n)).view(Hkv, blocks, 128, d).transpose(0, 1)
                pools.append(pool)
            bufs.append(spf.PagedPromptBuffers(q, pools, table.int(), n, *out(L, Hq, m, n)))
        else:
            if form == "strided":                          # token-major, rows apart
                k = [torch.empty(n, Hkv + 1, d + 8, dtype=torch.bfloat16, device="cuda")[:, :Hkv, :d].transpose(0, 1).copy_(x) for x in k]
            bufs.append(spf.PromptBuffers(q, k, *out(L, Hq, m, n)))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    score(bufs, scratch(size(bufs)), dev_status=status)
    got = [(b.importance.clone(), b.lse.clone()) for b in bufs]
    for path, rtol, atol in ((2, 1e-5, 1e-5), (1, 2e-4, 1e-4)):
        before = spf.spf_set_score_path(path)
        try:
            for b, (importance, lse) in zip(bufs, got):
                score([b], scratch(size([b])), dev_status=status)
                torch.testing.assert_close(importance, b.importance, rtol=rtol, atol=0)
                torch.testing.assert_close(lse, b.lse, rtol=0, atol=atol)
        finally:
            spf.spf_set_score_path(before)
    assert int(status) == 0


@pytest.mark.parametrize("L,Hq,Hkv,d,m,tiles", [
    (4, 8, 2, 64, 8, 3), (4, 4, 2, 64, 8, 9), (2, 2, 1, 128, 8, 12), (2, 4, 1, 128, 8, 14),
    # either side of the edges between the forms (test_split_cpu.py)
    *[(2, 4, 1, 64, 8, t) for t in (5, 6)], *[(2, 2, 1, 64, 16, t) for t in (3, 4)], *[(2, 4, 1, 128, 8, t) for t in (9, 10)],
    *[(2, 2, 1, 64, 8, t) for t in (19, 20)], *[(2, 2, 1, 128, 8, t) for t in (19, 20)], *[(2, 1, 1, 64, 16, t) for t in (10, 11)]])
def test_eight_bit_keys_of_many_tiles(L, Hq, Hkv, d, m, tiles):
    """Maxima in registers and in tensor memory, logits kept and computed twice."""
    import paper_2603_02631_b200 as spf
    n = tiles * SPAN - 77
    q, k = make(L, Hq, Hkv, d, m, n)
    k = [x.float().to(torch.float8_e4m3fn).view(torch.uint8) for x in k]
    scale = torch.rand(L, Hkv, device="cuda") + 0.5
    a, b = (spf.Fp8PromptBuffers(q, k, scale, *out(L, Hq, m, n)) for _ in range(2))
    ws, status = scratch(spf.spf_score_fp8_workspace_bytes([a])), torch.zeros(1, dtype=torch.int32, device="cuda")
    for path, buf in ((2, a), (1, b)):
        before = spf.spf_set_score_path(path)
        try:
            spf.spf_score_fp8([buf], ws, dev_status=status)
        finally:
            spf.spf_set_score_path(before)
    assert int(status) == 0
    torch.testing.assert_close(a.importance, b.importance, rtol=2e-4, atol=0)
    torch.testing.assert_close(a.lse, b.lse, rtol=0, atol=1e-4)


@pytest.mark.parametrize("n,k", [(20000, 7000), (20000, 19990), (4096, 5), (32768, 16000)])
def test_selection_of_more_distinct_scores_than_a_bin_is_ranked(n, k):
    """A tight cluster between a zero and a large outlier falls into a bin or two of 2048, and is cut again."""
    import paper_2603_02631_b200 as spf
    scores = 1 + torch.randperm(n, device="cuda").float() * 2.0 ** -22
    scores[17], scores[n // 2] = 0.0, 1e30
    i32 = lambda *s: torch.empty(*s, dtype=torch.int32, device="cuda")
    kept, ids = i32(k), torch.arange(n, dtype=torch.int32, device="cuda")
    spf.spf_select_compact(scores, n, k, 1, n, ids, ids, ids, kept, i32(n), None, i32(k, 2), i32(k, 2), torch.zeros(2, dtype=torch.int64, device="cuda"))
    assert torch.equal(kept, torch.argsort(scores, descending=True, stable=True)[:k].sort().values.int())


def test_prompts_on_two_streams():
    """Selectors of their own: every call's CTAs are resident together (a cooperative launch), whichever stream comes first."""
    import paper_2603_02631_b200 as spf
    geom, n = (8, 16, 4, 64, 8), 20000
    text = [torch.arange(n, dtype=torch.int32, device="cuda")] * 3
    streams, prompts = [torch.cuda.Stream() for _ in range(2)], [make(*geom, n, seed=s) for s in range(2)]
    want = [spf.Selector(*geom, n).run(q, k, *text, 0.2) for q, k in prompts]
    sels = [spf.Selector(*geom, n) for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(20):
        for s, sel, (q, k) in zip(streams, sels, prompts):
            got = sel.run(q, k, *text, 0.2, stream=s)
            del got
    torch.cuda.synchronize()
    for sel, w in zip(sels, want):
        assert int(sel.dev_status) == 0 and torch.equal(sel.importance, w.importance) and torch.equal(sel.counts, w.counts)


def test_a_captured_call_replays():
    import paper_2603_02631_b200 as spf
    geom, n = (4, 8, 2, 64, 8), 5000
    text, (q, k) = [torch.arange(n, dtype=torch.int32, device="cuda")] * 3, make(*geom, n)
    sel = spf.Selector(*geom, n)
    want = sel.run(q, k, *text, 0.2).importance.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sel.run(q, k, *text, 0.2)
    for _ in range(2):
        sel.importance.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(sel.importance, want) and int(sel.dev_status) == 0
