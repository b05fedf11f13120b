"""The scoring and selection kernels at the sizes where their tiles, rings and dispatch change."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu
SPAN = 148 * 128                       # tokens that give each SM of a B200 one tile of keys


def reference(q, k_layers):
    """Importance and log-sum-exps in double precision: mean over the lookahead of the max over (layer, head) of the softmax."""
    best, lses = None, []
    for ql, kl in zip(q, k_layers):
        heads = kl.shape[0]
        rows = ql.double().reshape(heads, -1, ql.shape[-1])                       # [Hkv, group * m, d]
        for h in range(heads):
            logits = rows[h] @ kl[h].double().T / ql.shape[-1] ** 0.5
            lse = torch.logsumexp(logits, dim=-1)
            p = (logits - lse[:, None]).view(-1, ql.shape[1], kl.shape[1]).amax(0)
            best = p if best is None else torch.maximum(best, p)
            lses.append(lse.reshape(-1))
    return best.exp().mean(0), torch.cat(lses)


def make(L, Hq, Hkv, d, m, n, seed=0):
    gen = torch.Generator(device="cuda").manual_seed(seed + 131 * n + m)
    q = torch.randn(L, Hq, m, d, generator=gen, device="cuda").to(torch.bfloat16)
    return q, [torch.randn(Hkv, n, d, generator=gen, device="cuda").to(torch.bfloat16) for _ in range(L)]


def text(n):
    ids = torch.arange(n, dtype=torch.int32, device="cuda") * 7 % 32000
    return ids, torch.arange(n, dtype=torch.int32, device="cuda") * 3, torch.arange(n, dtype=torch.int32, device="cuda") * 3 + 2


EDGES = [
    # one and two tiles, ragged; few CTAs per group, several groups that meet
    *[(3, 8, 2, 64, 8, n) for n in (1, 127, 128, 129, 255, 700, 5000)],
    # a tile to each CTA of groups of 40 and more
    *[(1, 2, 1, 128, 8, n) for n in (40 * 128, 40 * 128 + 1, SPAN)],
    # groups that are padded to a power of two
    *[(2, 2 * g, 2, 64, 8, 3001) for g in (3, 5, 6, 7)],
    # maxima in registers up to 8 tiles a CTA, in tensor memory beyond
    *[(2, 2, 1, 128, 8, t * SPAN + more) for t in (7, 8) for more in (-1, 1)],
    # 32 rows, 64 dimensions: logits computed twice
    *[(2, 4, 1, 64, 8, t * SPAN - 50) for t in (9, 10, 11, 12)],
    # from logits kept (maxima in registers, in tensor memory) to logits computed twice: test_split_cpu.py has the edges
    (2, 4, 1, 64, 8, 8 * SPAN - 50), *[(2, 4, 1, 128, 8, t * SPAN - 50) for t in (8, 9, 10, 11)],
    *[(2, 2, 1, 64, 16, t * SPAN - 50) for t in (4, 6, 7)], *[(2, 1, 1, 64, 16, t * SPAN - 50) for t in (10, 11)],
    *[(2, 2, 1, 64, 8, t * SPAN - 50) for t in (12, 13)], *[(1, 4, 1, 64, 4, t * SPAN - 50) for t in (23, 24)],
    # 64 rows: odd and even numbers of tiles, the two-pass form's rings from most to fewest stages
    *[(3, 4, 1, 64, 16, t * SPAN - 50) for t in (1, 2, 3, 6, 7, 11, 12, 15, 16)],
    (2, 8, 1, 128, 8, 3 * SPAN + 5), (2, 8, 2, 64, 5, 9001),
]


@pytest.mark.parametrize("L,Hq,Hkv,d,m,n", EDGES)
def test_scores_at_the_edges_of_tiles_and_rings(L, Hq, Hkv, d, m, n):
    """Tolerance: a logit is a dot product of d products in fp32, wrong by at most d * 2^-24 * sum |q_i k_i| * scale, which is
    below 128 * 2^-24 * 0.8 * 128 / 11.3 = 7e-5 for these inputs; a log-sum-exp is off by no more than its logits.  A
    probability's relative error is the two together."""
    import paper_2603_02631_b200 as spf
    q, k = make(L, Hq, Hkv, d, m, n)
    sel = spf.Selector(L, Hq, Hkv, d, m, n)
    s = sel.run(q, k, *text(n), keep=0.2)
    want, lse = reference(q, k)
    assert int(sel.dev_status) == 0
    assert ((s.importance.double() - want).abs() / want).max() < 2e-4
    assert (s.lse.double().reshape(-1) - lse).abs().max() < 1e-4


ROWS_AND_GROUPS = [
    # row sums added up in every CTA up to 56 CTAs to a group (64 rows: 12), by owners beyond
    *[(1, 4, 1, 64, 8, n) for n in (56 * 128, 56 * 128 + 1)], *[(1, 4, 1, 64, 16, n) for n in (12 * 128, 12 * 128 + 1, 28 * 128 + 1)],
    *[(1, 2, 1, 128, 8, n) for n in (56 * 128, 56 * 128 + 1)],
    # rows dealt to the columns: each padded group with the fewest and the most lookahead queries of 16, 32 and 64 rows
    *[(2, 2 * g, 2, 64, m, 2500) for g, ms in ((1, (1, 16, 17, 32)), (2, (1, 8, 9, 16, 17, 32)), (4, (1, 4, 5, 8, 9, 16)), (8, (1, 2, 3, 4, 5, 8)))
      for m in ms],
    # 8 heads in 16 columns, with the maxima in registers and (9 tiles a CTA) in tensor memory
    (1, 8, 1, 64, 2, 5 * SPAN - 50), (1, 6, 1, 64, 2, 9 * SPAN - 50),
    # more slabs than CTAs, and groups of CTAs that meet
    (40, 8, 4, 64, 8, 600), (40, 8, 4, 64, 8, 3000),
]


@pytest.mark.parametrize("L,Hq,Hkv,d,m,n", ROWS_AND_GROUPS)
def test_rows_are_dealt_to_columns_and_sums_to_warps(L, Hq, Hkv, d, m, n):
    """Tolerance as above."""
    import paper_2603_02631_b200 as spf
    q, k = make(L, Hq, Hkv, d, m, n)
    sel = spf.Selector(L, Hq, Hkv, d, m, n)
    s = sel.run(q, k, *text(n), keep=0.2)
    want, lse = reference(q, k)
    assert int(sel.dev_status) == 0
    assert ((s.importance.double() - want).abs() / want).max() < 2e-4
    assert (s.lse.double().reshape(-1) - lse).abs().max() < 1e-4


@pytest.mark.parametrize("L,Hq,Hkv,d,m,tiles", [
    *[(2, 1, 1, 64, 8, t) for t in (14, 15, 16, 27, 28)], (1, 2, 1, 64, 8, 20), (1, 2, 1, 64, 8, 56), (3, 1, 1, 128, 16, 28), (1, 8, 1, 64, 2, 57)])
def test_sixteen_rows_on_the_fused_path_up_to_its_longest_prompts(L, Hq, Hkv, d, m, tiles):
    """Running maxima of 28 tiles a CTA at 16 slots a key, or of 56 at 8, leave room for four accumulators of 16 columns.
    Tolerance as above."""
    import paper_2603_02631_b200 as spf
    n = tiles * SPAN - 50
    q, k = make(L, Hq, Hkv, d, m, n)
    sel = spf.Selector(L, Hq, Hkv, d, m, n)
    before = spf.spf_set_score_path(2)
    try:
        s = sel.run(q, k, *text(n), keep=0.2)
    finally:
        spf.spf_set_score_path(before)
    want, lse = reference(q, k)
    assert int(sel.dev_status) == 0
    assert ((s.importance.double() - want).abs() / want).max() < 2e-4
    assert (s.lse.double().reshape(-1) - lse).abs().max() < 1e-4


def test_batch_of_more_prompts_than_one_launch_takes():
    """Lengths from one token to several tiles per SM, together and one by one: only the order of sums differs (a row sum of
    n terms in fp32, at most n * 2^-24 apart, far less in practice)."""
    import paper_2603_02631_b200 as spf
    L, Hq, Hkv, d, m = 2, 8, 2, 64, 8
    lens = [1, 128, 129, 4000, 900, 31, 12000, 257, 640, 5, 2048, 777, 60000, 333, 1500, 90, 2500, 64, 1023]

    class Prompt:
        pass

    prompts = []
    for i, n in enumerate(lens):
        p = Prompt()
        p.n_tokens, (p.q, p.k) = n, make(L, Hq, Hkv, d, m, n, seed=i)
        p.token_ids, p.char_start, p.char_end = text(n)
        prompts.append(p)
    batch = spf.BatchSelector(L, Hq, Hkv, d, m, lens)
    got = batch.run(prompts, 0.3)
    assert int(batch.dev_status) == 0
    for p, s in zip(prompts, got):
        one = spf.Selector(L, Hq, Hkv, d, m, p.n_tokens)
        w = one.run(p.q, p.k, p.token_ids, p.char_start, p.char_end, 0.3)
        torch.testing.assert_close(s.importance, w.importance, rtol=1e-5, atol=0)
        torch.testing.assert_close(s.lse, w.lse, rtol=1e-5, atol=1e-5)


class Item(ctypes.Structure):
    _fields_ = [(name, ctypes.c_int64 if name in ("n_tokens", "k") else ctypes.c_void_p) for name in
                ("importance", "n_tokens", "chunk_scores", "k", "token_ids", "char_start", "char_end", "kept_chunks", "out_ids", "out_pos",
                 "out_tok_spans", "out_char_spans", "out_counts")]


@pytest.mark.parametrize("lens,chunk,pool,edge,force,levels", [
    ([1, 2, 31, 32, 33, 64], 32, 13, 0, (0, 0), 0),                    # fewer chunks than a batch of eight
    ([255, 256, 257, 2048, 2049, 4097, 8193, 8200], 32, 13, 1, (1, 1), 0),   # clusters of 1, 2, 4 and 8 CTAs
    ([1000, 3], 1, 1, 0, (0, 1), 0), ([20000], 7, 255, 1, (1, 0), 0),  # windows longer than chunks
    ([32768, 32769, 40000], 1, 3, 0, (0, 0), 0),                       # 32768 chunks in shared memory, more in three launches
    ([131071], 32, 13, 0, (0, 0), 3), ([30000], 1, 1, 0, (1, 1), 1),   # hundreds and thousands of equal scores
    ([64] * 30, 16, 5, 0, (0, 0), 0),                                  # more prompts than one launch takes
    ([100001, 70000], 33, 13, 0, (0, 0), 0), ([100001], 1000, 13, 0, (0, 1), 0),   # chunks of more than one row of a warp
    ([100001], 16384, 13, 0, (0, 1), 0), ([100001], 100001, 13, 0, (0, 0), 0), ([9000], 20000, 13, 0, (0, 0), 0),
])
@pytest.mark.parametrize("keep", [0.001, 0.3, 1.0])
def test_pool_select_compact_equals_the_separate_calls(lens, chunk, pool, edge, force, levels, keep):
    import paper_2603_02631_b200 as spf
    lib = spf.lib
    lib.spf_pool_select_compact.argtypes = [ctypes.POINTER(Item)] + [ctypes.c_int32] * 6 + [ctypes.c_void_p]
    items, got, want, alive = (Item * len(lens))(), [], [], []
    for i, n in enumerate(lens):
        gen = torch.Generator(device="cuda").manual_seed(n + i)
        imp = torch.rand(n, generator=gen, device="cuda") ** 4 - 0.1
        if levels:
            imp = (torch.rand(n, generator=gen, device="cuda") * levels).floor()
        chunks = -(-n // chunk)
        k = max(spf.spf_keep_count(chunks, keep), min(chunks, sum(force)))
        ids, start, end = text(n)
        both = []
        for _ in range(2):
            i32 = lambda *size: torch.full(size, -1, dtype=torch.int32, device="cuda")
            both.append(dict(scores=torch.empty(chunks, device="cuda"), kept=i32(k), ids=i32(n), pos=i32(n), tok=i32(k, 2), ch=i32(k, 2),
                             counts=torch.zeros(2, dtype=torch.int64, device="cuda")))
        a, b = both
        items[i] = Item(imp.data_ptr(), n, a["scores"].data_ptr(), k, ids.data_ptr(), start.data_ptr(), end.data_ptr(), a["kept"].data_ptr(),
                        a["ids"].data_ptr(), a["pos"].data_ptr(), a["tok"].data_ptr(), a["ch"].data_ptr(), a["counts"].data_ptr())
        spf.spf_chunk_pool_edge(imp, pool, chunk, edge, b["scores"])
        spf.spf_select_topk_forced(b["scores"], chunks, k, bool(force[0]), bool(force[1]), b["kept"])
        spf.spf_compact_spans(b["kept"], k, chunk, n, ids, start, end, b["ids"], b["pos"], b["tok"], b["ch"], b["counts"])
        got.append(a)
        want.append(b)
        alive.append((imp, ids, start, end))
    stream = torch.cuda.current_stream().cuda_stream
    assert lib.spf_pool_select_compact(items, len(lens), pool, chunk, edge, *force, stream) == 0
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        for name in a:
            assert torch.equal(a[name], b[name]), name


@pytest.mark.parametrize("n", [1, 31, 1023, 1024, 1025, 8191, 8192, 8193, 40001])
@pytest.mark.parametrize("levels", [0, 3])
def test_separate_selection_where_its_steps_and_block_sizes_change(n, levels):
    """Keys in registers up to 8192 chunks, 1024 kept chunks and more; all distinct, and thousands of equal ones.  Against a
    stable sort and a walk over the kept chunks: whole numbers, nothing to tolerate."""
    import paper_2603_02631_b200 as spf
    gen = torch.Generator(device="cuda").manual_seed(n)
    scores = torch.rand(n, generator=gen, device="cuda")
    if levels:
        scores = (scores * levels).floor()
    order = torch.argsort(scores, descending=True, stable=True)
    ids, start, end = text(n)
    for k in sorted({1, min(n, 1024), min(n, 1025), -(-n // 3), n}):
        i32 = lambda *size: torch.full(size, -1, dtype=torch.int32, device="cuda")
        kept, out, pos, tok, ch = i32(k), i32(n), i32(n), i32(k, 2), i32(k, 2)
        counts = torch.zeros(2, dtype=torch.int64, device="cuda")
        spf.spf_select_topk(scores, n, k, kept)
        want = order[:k].sort().values.int()
        assert torch.equal(kept, want)
        spf.spf_compact_spans(kept, k, 1, n, ids, start, end, out, pos, tok, ch, counts)
        first = torch.cat([torch.ones(1, dtype=torch.bool, device="cuda"), want[1:] != want[:-1] + 1])
        a = want[first]
        b = torch.cat([want[:-1][first[1:]], want[-1:]]) + 1
        spans = len(a)
        assert counts.tolist() == [k, spans]
        assert torch.equal(tok[:spans], torch.stack([a, b], 1)) and torch.equal(pos[:k], want) and torch.equal(out[:k], ids[want.long()])
        assert torch.equal(ch[:spans], torch.stack([start[a.long()], end[b.long() - 1]], 1)) and bool((tok[spans:] == -1).all())


@pytest.mark.parametrize("chunk,pool,edge", [(32, 13, 0), (32, 13, 1), (64, 255, 0), (7, 5, 0), (1000, 13, 1)])
def test_pooling_of_values_near_the_end_of_the_range(chunk, pool, edge):
    """Scores that are representable come out, whatever the sums on the way to them; infinities and NaN reach the chunks whose
    windows hold them and no other.  Tolerance: sums of up to chunk + pool terms of one sign in fp32, 2^-24 per addition."""
    import paper_2603_02631_b200 as spf
    n, lib = 9001, spf.lib
    gen = torch.Generator(device="cuda").manual_seed(chunk)
    imp = (1 + torch.rand(n, generator=gen, device="cuda")) * (1.6e38 / max(chunk, pool))
    imp[700], imp[4000], imp[4010], imp[8000] = float("inf"), float("inf"), float("-inf"), float("nan")
    half, chunks = pool // 2, -(-n // chunk)
    padded = torch.nn.functional.pad(imp.double(), (half, half))
    windows = padded.unfold(0, pool, 1).sum(1)
    reach = torch.nn.functional.pad(torch.ones(n, dtype=torch.float64, device="cuda"), (half, half)).unfold(0, pool, 1).sum(1)
    smooth = windows / (reach if edge else pool)
    want = torch.stack([x.mean() for x in smooth.split(chunk)])
    scores = torch.empty(chunks, device="cuda")
    spf.spf_chunk_pool_edge(imp, pool, chunk, edge, scores)
    torch.testing.assert_close(scores.double(), want, rtol=(chunk + pool) * 2.0 ** -24, atol=0, equal_nan=True)
    assert bool(scores.isfinite().any())
    both, i32 = torch.empty(chunks, device="cuda"), lambda *size: torch.empty(size, dtype=torch.int32, device="cuda")
    ids, out = text(n), (i32(1), i32(n), i32(n), i32(2), i32(2), torch.empty(2, dtype=torch.int64, device="cuda"))
    lib.spf_pool_select_compact.argtypes = [ctypes.POINTER(Item)] + [ctypes.c_int32] * 6 + [ctypes.c_void_p]
    item = (Item * 1)(Item(imp.data_ptr(), n, both.data_ptr(), 1, *[t.data_ptr() for t in (*ids, *out)]))
    assert lib.spf_pool_select_compact(item, 1, pool, chunk, edge, 0, 0, torch.cuda.current_stream().cuda_stream) == 0
    torch.testing.assert_close(both, scores, rtol=0, atol=0, equal_nan=True)


def test_selector_refuses_what_does_not_fit():
    import paper_2603_02631_b200 as spf
    q, k = make(2, 4, 2, 64, 8, 300)
    sel, ids = spf.Selector(2, 4, 2, 64, 8, 300), text(300)
    for bad, error in [((q.float(), k), TypeError), ((q.cpu(), k), TypeError), ((q[0], k), ValueError), ((q, k[:1]), ValueError),
                       ((q, [k[0], k[1][:, :299]]), ValueError), ((q, [k[0].float(), k[1]]), TypeError), ((q, []), ValueError)]:
        with pytest.raises(error):
            sel.run(*bad, *ids, keep=0.2)
    with pytest.raises(ValueError):
        spf.Selector(2, 4, 2, 64, 8, 299).run(q, k, *ids, keep=0.2)
    with pytest.raises(ValueError):
        sel.run(q, k, ids[0][:299], *ids[1:], keep=0.2)
