"""spf_compress_host: the whole path for host buffers through one C call, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from workloads import CONFIGS, bf16_bits, make_prompt, small_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pinned", [True, False])
def test_compress_host_matches_the_oracle(pinned):
    import paper_2603_02631_b200 as spf
    cfg = small_config("hostpath", n_layers=3, n_q_heads=8, n_kv_heads=2, head_dim=64, n_lookahead=8, lengths=(5003,),
                       chunk=32, keep=(0.2,), rank=4, n_needles=3, n_strong=2, seed=77)
    prompt = make_prompt(cfg)                             # host tensors
    keep = 0.2
    ref = oracle.compress(bf16_bits(prompt.q), [bf16_bits(x) for x in prompt.k], prompt.token_ids.numpy(),
                          prompt.char_start.numpy(), prompt.char_end.numpy(), chunk=cfg.chunk, keep=keep,
                          pool_kernel=cfg.pool_kernel)
    pin = (lambda t: t.contiguous().pin_memory()) if pinned else (lambda t: t.contiguous())
    sel = spf.Selector(cfg.n_layers, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.n_lookahead, prompt.n_tokens,
                       chunk=cfg.chunk, pool_kernel=cfg.pool_kernel)
    for _ in range(2):                                    # the second call reuses the arena and the result buffers
        got = sel.run_host(pin(prompt.q), [pin(x) for x in prompt.k], pin(prompt.token_ids), pin(prompt.char_start),
                           pin(prompt.char_end), keep)
        assert got["ids"].tolist() == ref["ids"].tolist()
        assert got["pos"].tolist() == ref["pos"].tolist()
        assert got["tok_spans"].tolist() == ref["tok_spans"].tolist()
        assert got["char_spans"].tolist() == ref["char_spans"].tolist()


def test_compress_host_reports_a_small_arena():
    import paper_2603_02631_b200 as spf
    prompt = make_prompt(CONFIGS["tiny"])
    cfg = prompt.cfg
    k = spf.spf_keep_count(prompt.n_tokens // cfg.chunk, 0.25)
    arena = torch.empty(1024, dtype=torch.uint8, device="cuda")
    out = [torch.empty(k * cfg.chunk, dtype=torch.int32), torch.empty(k * cfg.chunk, dtype=torch.int32),
           torch.empty((k, 2), dtype=torch.int32), torch.empty((k, 2), dtype=torch.int32), torch.empty(2, dtype=torch.int64)]
    with pytest.raises(spf.SpfError) as err:
        spf.spf_compress_host(prompt.q, prompt.k, prompt.token_ids, prompt.char_start, prompt.char_end, cfg.chunk,
                              cfg.pool_kernel, 0.25, arena, *out)
    assert err.value.status == -3


def test_compress_host_writes_nothing_of_an_attempt_it_gives_up():
    """A head that overflows the fused path's row sums: the prompt is scored again with the general kernels, and the buffers hold
    that result and, beyond its rows, what they held before."""
    import paper_2603_02631_b200 as spf
    L, Hq, Hkv, m, d, n, chunk, keep = 1, 4, 1, 8, 64, 3000, 32, 0.3
    gen = torch.Generator().manual_seed(3)
    q, k = torch.randn(L, Hq, m, d, generator=gen), torch.randn(Hkv, n, d, generator=gen)
    q[0, 3] *= 60                                         # logits of several hundred nats against other heads' single digits
    q, k = q.to(torch.bfloat16), k.to(torch.bfloat16)
    ids = torch.arange(n, dtype=torch.int32)
    sel = spf.Selector(L, Hq, Hkv, d, m, n)
    dev = [t.cuda() for t in (q, k, ids)]
    sel.run(dev[0], [dev[1]], dev[2], dev[2], dev[2], keep)
    assert int(sel.dev_status) == -6                      # what the first attempt reports
    before = spf.spf_set_score_path(1)
    try:
        want = sel.run(dev[0], [dev[1]], dev[2], dev[2], dev[2], keep).host()
    finally:
        spf.spf_set_score_path(before)
    out = [torch.full((n,), -7, dtype=torch.int32).pin_memory(), torch.full((n,), -7, dtype=torch.int32).pin_memory(),
           torch.full((n, 2), -7, dtype=torch.int32).pin_memory(), torch.full((n, 2), -7, dtype=torch.int32).pin_memory(),
           torch.zeros(2, dtype=torch.int64).pin_memory()]
    arena = torch.empty(spf.spf_compress_host_arena_bytes(L, Hq, Hkv, d, m, n, chunk, 13, keep), dtype=torch.uint8, device="cuda")
    spf.spf_compress_host(q, [k], ids, ids, ids, chunk, 13, keep, arena, *out)
    kept, spans = out[4].tolist()
    assert out[0][:kept].tolist() == want["ids"].tolist() and out[2][:spans].tolist() == want["tok_spans"].tolist()
    for t, rows in zip(out, (kept, kept, spans, spans)):
        assert bool((t[rows:] == -7).all())
