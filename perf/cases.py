"""What a user of this library has it do, as cases that can be prepared, run and timed.

A pass is the whole path for one prompt (or one batch of prompts) through the package's public classes: token
importance from the draft model's lookahead queries and prompt keys, chunk pooling, top-k chunks, compacted token
ids and character spans.  What a serving program keeps between prompts -- the selector with its buffers -- is made
in ``prepare``; everything else happens in ``run``.

The fields of a case: ``entry`` (which public call: ``run``, ``paged``, ``fp8``, ``batch`` or ``host``), the draft
model's geometry ``L`` layers, ``Hq`` query heads, ``Hkv`` key heads, ``d`` head dimension, ``m`` lookahead queries,
``n`` prompt tokens, ``chunk`` tokens per chunk, ``keep`` rate, ``block`` tokens per block of a paged key cache,
``batch`` prompts with lengths spread over [``n_lo``, ``n``] by ``len_seed``.
"""
import math
import random

import torch

import paper_2603_02631_b200 as spf

POOL_KERNEL = 13          # the paper's smoothing window
VOCAB = 32000
RANK = 16                 # rank of the component that all layers and heads share
MAX_DRAWN_KEY_BYTES = 12e9   # below the largest listed case (about 36 GB of keys)


def _case(name, entry, L, Hq, Hkv, d, m, n, chunk, keep, **more):
    return dict(name=name, entry=entry, L=L, Hq=Hq, Hkv=Hkv, d=d, m=m, n=n, chunk=chunk, keep=keep, **more)


def listed():
    return [
        # the smallest call: a two-layer draft and a short prompt; launches and host work count
        _case("tiny2k", "run", 2, 4, 2, 64, 8, 2048, 32, 0.25),
        # an ordinary chat-length prompt, odd length, on a small draft (16 layers, 32/8 heads of 64)
        _case("short4k", "run", 16, 32, 8, 64, 8, 4001, 32, 0.25),
        # the same draft at 32k tokens
        _case("small32k", "run", 16, 32, 8, 64, 8, 32768, 32, 0.10),
        # a deeper draft with heads of 128 at 64k tokens, chunks of 64
        _case("wide64k", "run", 28, 16, 8, 128, 8, 65536, 64, 0.10),
        # long context with 16 lookahead queries: the workload of the repository's benchmark
        _case("long128k", "run", 16, 32, 8, 64, 16, 131072, 32, 0.10),
        # the length of book-sized question answering, chunks of 128, low keep rate, odd length
        _case("long250k", "run", 28, 16, 8, 128, 8, 250003, 128, 0.06),
        # three query heads per key head: a group that is no power of two
        _case("group3_20k", "run", 28, 24, 8, 128, 8, 20011, 32, 0.15),
        # a serving engine's paged cache with its smallest blocks
        _case("paged50k", "paged", 16, 32, 8, 64, 8, 50000, 32, 0.10, block=128),
        # an 8-bit key cache at long context
        _case("fp8_128k", "fp8", 16, 32, 8, 64, 16, 131072, 32, 0.10),
        # a batch of short prompts of different lengths
        _case("batch_short", "batch", 16, 32, 8, 64, 8, 8192, 32, 0.20, batch=8, n_lo=700, len_seed=1),
        # a ragged batch of long prompts
        _case("batch_long", "batch", 28, 16, 8, 128, 8, 131072, 32, 0.10, batch=8, n_lo=16384, len_seed=4),
        # a prompt whose tensors are in pinned host memory, results back on the host
        _case("host8k", "host", 16, 32, 8, 64, 8, 8192, 32, 0.20),
    ]


def draw(rng):
    entry = rng.choice(["run", "run", "run", "paged", "fp8", "batch", "host"])
    d = rng.choice([64, 128])
    m = rng.choice([1, 4, 5, 8, 8, 8, 12, 16])
    groups = [g for g in (1, 2, 3, 4, 8) if g * (-(-m // 8) * 8) <= 64]
    group, hkv = rng.choice(groups), rng.choice([2, 4, 8, 8])
    layers = rng.choice([2, 4, 12, 16, 16, 24, 28, 28, 32, 36])
    top = {"host": 16384, "batch": 65536}.get(entry, 262144)
    n = int(math.exp(rng.uniform(math.log(1024), math.log(top))))
    case = _case("", entry, layers, hkv * group, hkv, d, m, n, rng.choice([32, 32, 64, 128]),
                 rng.choice([0.03, 0.06, 0.10, 0.10, 0.15, 0.25, 0.50]))
    del case["name"]
    if entry == "paged":
        case["block"] = rng.choice([128, 256, 1024, 4096])
    if entry == "batch":
        case.update(batch=rng.randint(2, 8), n_lo=max(256, n // 8), len_seed=rng.randrange(1 << 20))
    while _key_bytes(case) > MAX_DRAWN_KEY_BYTES:
        case["n"] = case["n"] // 2 + 1
        if entry == "batch":
            case["n_lo"] = max(256, case["n"] // 8)
    return case


# ---------------------------------------------------------------------------------------------- inputs
def _lengths(case):
    """Prompt lengths of the case: one, or a batch's lengths (the longest is always ``n``)."""
    if case["entry"] != "batch":
        return [case["n"]]
    rng = random.Random(case["len_seed"])
    lens = [rng.randint(case["n_lo"], case["n"]) for _ in range(case["batch"] - 1)] + [case["n"]]
    rng.shuffle(lens)
    return lens


def _element_bytes(case):
    return 1 if case["entry"] == "fp8" else 2


def _key_bytes(case):
    return sum(_lengths(case)) * case["L"] * case["Hkv"] * case["d"] * _element_bytes(case)


class _Prompt:
    """One prompt's tensors, named as ``BatchSelector.run`` reads them."""


def _make_prompt(case, n, seed):
    """Queries and keys of N(0, 1) with what attention maps of long prompts have: a low-rank part that all layers and
    heads share, and spans of keys that a quarter of the (layer, kv-head) pairs attend to strongly (one span in four)
    or weakly."""
    L, Hq, Hkv, d, m = (case[x] for x in ("L", "Hq", "Hkv", "d", "m"))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def randn(*shape):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32)

    def randint(lo, hi, shape):
        return torch.randint(lo, hi, shape, generator=gen, device="cuda")

    def rand(*shape):
        return torch.rand(*shape, generator=gen, device="cuda")

    # spans: one per segment of the prompt, 16 to 128 tokens long; span_of[t] is the span of token t, `spans` if none
    spans = max(1, min(64, n // 256))
    seg = n // spans
    length = randint(16, max(17, min(129, seg)), (spans,))
    first = (rand(spans) * (seg - length).clamp_min(0)).long()
    pos = torch.arange(n, device="cuda")
    which = (pos // seg).clamp_max(spans - 1)
    inside = (pos - which * seg >= first[which]) & (pos - which * seg < first[which] + length[which])
    span_of = torch.where(inside, which, spans)
    alpha = math.sqrt(8.0 * math.sqrt(d))                  # a strong span's keys gain about 8 nats
    strength = torch.where(torch.arange(spans, device="cuda") % 4 == 0, alpha, alpha / 4)

    tok, qry = randn(n, RANK), randn(m, RANK)
    p = _Prompt()
    p.n_tokens, p.k, q = n, [], []
    for _ in range(L):
        basis = randn(Hkv, RANK, d) * (2.0 / math.sqrt(d))
        kl, ql = randn(Hkv, n, d), randn(Hkv, Hq // Hkv, m, d)
        kl.baddbmm_(tok.expand(Hkv, n, RANK), basis)
        ql += torch.matmul(qry, basis)[:, None]
        u = torch.nn.functional.normalize(randn(Hkv, d), dim=-1)
        gain = torch.zeros(Hkv, spans + 1, device="cuda")
        gain[:, :spans] = strength * (rand(Hkv, spans) < 0.25)
        kl.addcmul_(gain[:, span_of][:, :, None], u[:, None, :])
        ql += alpha * u[:, None, None, :]
        p.k.append(kl.to(torch.bfloat16))
        q.append(ql.reshape(Hq, m, d).to(torch.bfloat16))
        del kl
    p.q = torch.stack(q)
    p.token_ids = randint(0, VOCAB, (n,)).to(torch.int32)
    chars = randint(1, 9, (n,))
    ends = torch.cumsum(chars, 0)
    p.char_start, p.char_end = (ends - chars).to(torch.int32), ends.to(torch.int32)
    return p


def _to_e4m3(k_layers):
    """The keys as E4M3 bytes with one scale per (layer, kv-head)."""
    rows, scales = [], []
    while k_layers:
        kl = k_layers.pop(0).float()
        scale = kl.abs().amax(dim=(1, 2)) / 448.0
        rows.append((kl / scale[:, None, None]).to(torch.float8_e4m3fn).view(torch.uint8))
        scales.append(scale)
    return rows, torch.stack(scales)


def _to_blocks(k_layers, block, seed):
    """The keys scattered over a pool of blocks in a random order, three blocks of the pool unused."""
    Hkv, n, d = k_layers[0].shape
    count = -(-n // block)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    table = torch.randperm(count + 3, generator=gen, device="cuda")[:count]
    pools = []
    while k_layers:
        kl = torch.nn.functional.pad(k_layers.pop(0), (0, 0, 0, count * block - n))
        pool = torch.zeros(count + 3, Hkv, block, d, dtype=torch.bfloat16, device="cuda")
        pool[table] = kl.view(Hkv, count, block, d).transpose(0, 1)
        pools.append(pool)
    return pools, table.to(torch.int32)


def _clear(selector):
    """Results shorter than their buffers leave the rest as it was: zeros, so that whole buffers can be compared."""
    for t in (selector.kept, selector.out_ids, selector.out_pos, selector.tok_spans, selector.char_spans):
        t.zero_()


def prepare(case, seed):
    geom = [case[x] for x in ("L", "Hq", "Hkv", "d", "m")]
    lens = _lengths(case)
    options = dict(chunk=case["chunk"], pool_kernel=POOL_KERNEL)
    prompts = [_make_prompt(case, n, 1009 * seed + 7 * i) for i, n in enumerate(lens)]
    state = {"entry": case["entry"], "chunk": case["chunk"], "keep": case["keep"], "prompts": prompts}
    p = prompts[0]
    if case["entry"] == "batch":
        state["selector"] = spf.BatchSelector(*geom, lens, **options)
        for slot in state["selector"].slots:
            _clear(slot)
        return state
    if case["entry"] != "host":
        state["selector"] = spf.Selector(*geom, case["n"], **options)
        _clear(state["selector"])
    if case["entry"] == "paged":
        p.pools, p.table = _to_blocks(p.k, case["block"], seed)
    elif case["entry"] == "fp8":
        p.k, p.scale = _to_e4m3(p.k)
    elif case["entry"] == "host":
        p.q, p.k = p.q.cpu().pin_memory(), [k.cpu().pin_memory() for k in p.k]
        p.token_ids, p.char_start, p.char_end = (t.cpu().pin_memory() for t in (p.token_ids, p.char_start, p.char_end))
        state["arena"] = torch.empty(spf.spf_compress_host_arena_bytes(*geom, p.n_tokens, case["chunk"], POOL_KERNEL, case["keep"]),
                                     dtype=torch.uint8, device="cuda")
        k = spf.spf_keep_count(-(-p.n_tokens // case["chunk"]), case["keep"])
        rows = min(k * case["chunk"], p.n_tokens)
        sizes = [("out_ids", (rows,)), ("out_pos", (rows,)), ("tok_spans", (k, 2)), ("char_spans", (k, 2))]
        state["host_out"] = {name: torch.zeros(size, dtype=torch.int32).pin_memory() for name, size in sizes}
        state["host_out"]["counts"] = torch.zeros(2, dtype=torch.int64).pin_memory()
    return state


# ---------------------------------------------------------------------------------------------- one pass
def _outputs(s):
    return {"importance": s.importance, "lse": s.lse, "chunk_scores": s.chunk_scores, "out_ids": s.out_ids,
            "out_pos": s.out_pos, "tok_spans": s.tok_spans, "char_spans": s.char_spans, "counts": s.counts}


def run(state):
    entry, keep, p = state["entry"], state["keep"], state["prompts"][0]
    if entry == "host":
        out = state["host_out"]
        spf.spf_compress_host(p.q, p.k, p.token_ids, p.char_start, p.char_end, state["chunk"], POOL_KERNEL, keep, state["arena"],
                              out["out_ids"], out["out_pos"], out["tok_spans"], out["char_spans"], out["counts"])
        return out
    sel = state["selector"]
    if entry == "batch":
        return [_outputs(s) for s in sel.run(state["prompts"], keep)]
    if entry == "paged":
        s = sel.run_paged(p.q, p.pools, p.table, p.n_tokens, p.token_ids, p.char_start, p.char_end, keep)
    elif entry == "fp8":
        s = sel.run_fp8(p.q, p.k, p.scale, p.token_ids, p.char_start, p.char_end, keep)
    else:
        s = sel.run(p.q, p.k, p.token_ids, p.char_start, p.char_end, keep)
    return dict(_outputs(s), kept_chunks=s.kept_chunks, status=sel.dev_status)


# ---------------------------------------------------------------------------------------------- yardsticks
def work(case):
    """Bytes: keys, queries, the kept tokens' ids and each result once.  Operations: one product of every query row
    with every key (the softmax over them comes on top and is not counted)."""
    L, Hq, d, m = case["L"], case["Hq"], case["d"], case["m"]
    total = _key_bytes(case)
    for n in _lengths(case):
        chunks = -(-n // case["chunk"])
        kept = min(n, spf.spf_keep_count(chunks, case["keep"]) * case["chunk"])
        total += L * Hq * m * d * 2 + L * Hq * m * 4       # queries in, log-sum-exps out
        total += 4 * n + 4 * chunks + 12 * kept            # importance and chunk scores out; kept ids in, ids and positions out
    return {"bytes": total, "flops": 2 * sum(_lengths(case)) * L * Hq * m * d}


def tolerance(case):
    """32-bit results: a base-2 logit of up to about 60 carries 60 * 2^-24 of rounding, and a probability's relative
    error is that of its logit and its row's log-sum-exp together.  Whole values are the same except where two chunks'
    scores tie to within that error."""
    return {"rel": 1e-5, "differ": 0.01}
