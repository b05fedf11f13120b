"""What callers may rely on beyond the numbers: which tensors a call holds, which buffers it takes, what it leaves alone."""
import os
import subprocess
import sys

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu
GEOM = (2, 4, 2, 64, 8)                # L, Hq, Hkv, d, m


def make(n, seed=0, geom=GEOM):
    L, Hq, Hkv, d, m = geom
    gen = torch.Generator(device="cuda").manual_seed(seed + 131 * n)
    q = torch.randn(L, Hq, m, d, generator=gen, device="cuda").to(torch.bfloat16)
    return q, [torch.randn(Hkv, n, d, generator=gen, device="cuda").to(torch.bfloat16) for _ in range(L)]


def text(n):
    ids = torch.arange(n, dtype=torch.int32, device="cuda")
    return ids * 7 % 32000, ids * 3, ids * 3 + 2


class Fresh:
    """A prompt that keeps its tensors in another form and makes those of the call when it is asked for them."""

    def __init__(self, n, seed):
        q, k = make(n, seed)
        self.n_tokens, self._q, self._k, self._text = n, q.cpu(), [x.cpu() for x in k], [t.cpu() for t in text(n)]

    q = property(lambda self: self._q.cuda())
    k = property(lambda self: [x.cuda() for x in self._k])
    token_ids = property(lambda self: self._text[0].cuda())
    char_start = property(lambda self: self._text[1].cuda())
    char_end = property(lambda self: self._text[2].cuda())


def test_tensors_made_for_the_call_live_until_it_is_enqueued():
    """Each prompt's tensors are dropped by their maker at once; the next prompt's, or the workspace, would get their memory."""
    import paper_2603_02631_b200 as spf
    prompts = [Fresh(3000, seed) for seed in range(4)]
    batch = spf.BatchSelector(*GEOM, [3000] * 4)
    got = batch.run(prompts, 0.3)
    torch.cuda.synchronize()
    for p, s in zip(prompts, got):
        one = spf.Selector(*GEOM, 3000).run(p.q, p.k, p.token_ids, p.char_start, p.char_end, 0.3)
        torch.testing.assert_close(s.importance, one.importance, rtol=1e-5, atol=0)
        assert torch.equal(s.out_ids[:int(s.counts[0])], one.out_ids[:int(one.counts[0])])
    # a sequence that makes its items, and a workspace that has to be allocated after them
    class Lazy:
        def __init__(self, host):
            self.host = host

        def __len__(self):
            return len(self.host)

        def __getitem__(self, i):
            return self.host[i].cuda()

    p = prompts[0]
    s = spf.Selector(*GEOM, 3000).run(p.q, Lazy(p._k), p.token_ids, p.char_start, p.char_end, 0.3)
    torch.testing.assert_close(s.importance, got[0].importance, rtol=1e-5, atol=0)
    with pytest.raises(TypeError):                         # one pass over an iterator is all there is: refused
        spf.Selector(*GEOM, 3000).run(p.q, iter(p.k), p.token_ids, p.char_start, p.char_end, 0.3)


def test_positions_and_status_are_optional():
    """spf_compact_spans takes no positions and spf_score no status; a selector whose buffer is None asks for neither."""
    import paper_2603_02631_b200 as spf
    q, k = make(700)
    full, bare = spf.Selector(*GEOM, 700), spf.Selector(*GEOM, 700)
    bare.out_pos = bare.dev_status = None
    want, got = full.run(q, k, *text(700), 0.3), bare.run(q, k, *text(700), 0.3)
    kept = int(want.counts[0])
    assert torch.equal(want.out_ids[:kept], got.out_ids[:kept]) and got.out_pos is None
    batch, p = spf.BatchSelector(*GEOM, [700]), Fresh(700, 0)
    batch.slots[0].out_pos = batch.dev_status = None
    got = batch.run([p], 0.3)[0]
    assert torch.equal(want.out_ids[:kept], got.out_ids[:kept])


@pytest.mark.parametrize("chunk", [0, -3, 1 << 32, (1 << 32) + 32])
def test_selector_refuses_chunks_that_make_no_sense(chunk):
    """Read on every call: the attribute can be set after construction.  2^32 is zero in 32 bits, 2^32 + 32 is 32."""
    import paper_2603_02631_b200 as spf
    q, k = make(300)
    sel, batch = spf.Selector(*GEOM, 300), spf.BatchSelector(*GEOM, [300])
    sel.chunk = batch.chunk = chunk
    with pytest.raises(ValueError):
        sel.run(q, k, *text(300), 0.3)
    with pytest.raises(ValueError):
        batch.run([Fresh(300, 0)], 0.3)


def test_a_batch_is_scored_with_a_workspace_for_its_longest_prompt():
    """Fewer prompts share a launch, at every size of the workspace between that and the whole batch's."""
    import paper_2603_02631_b200 as spf
    lens = [300, 5000, 17, 2500, 5000, 128, 1, 900, 64, 3000, 700, 31, 4000, 222, 1500, 90, 2047, 640]
    bufs = []
    for i, n in enumerate(lens):
        q, k = make(n, i)
        bufs.append(spf.PromptBuffers(q, k, torch.empty(n, device="cuda"), torch.empty(2 * 4 * 8, device="cuda")))
    want = []
    for b in bufs:
        spf.spf_score([b], torch.empty(spf.spf_score_workspace_bytes([b]), dtype=torch.uint8, device="cuda"))
        want.append((b.importance.clone(), b.lse.clone()))
    least, most = max(spf.spf_score_workspace_bytes([b]) for b in bufs), spf.spf_score_workspace_bytes(bufs)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for size in (least, least + 256, (least + most) // 2, most):
        for b in bufs:
            b.importance.fill_(-1)
            b.lse.fill_(-1)
        ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        ws[size:] = 77
        spf.spf_score(bufs, ws[:size], dev_status=status)
        assert int(status) == 0 and bool((ws[size:] == 77).all())
        for b, (importance, lse) in zip(bufs, want):
            torch.testing.assert_close(b.importance, importance, rtol=1e-5, atol=0)
            torch.testing.assert_close(b.lse, lse, rtol=1e-5, atol=1e-5)


TWO_CONTEXTS = """
import ctypes, numpy as np, torch
import paper_2603_02631_b200 as spf
from paper_2603_02631_b200 import binding as b
L, Hq, Hkv, m, d, n, chunk, keep = 2, 4, 2, 8, 64, 300000, 32, 0.3
gen = torch.Generator().manual_seed(1)
q = torch.randn(L, Hq, m, d, generator=gen).to(torch.bfloat16)
k = [torch.randn(Hkv, n, d, generator=gen).to(torch.bfloat16) for _ in range(L)]
ids = torch.arange(n, dtype=torch.int32)
shape, prm = b._Shape(L, Hq, Hkv, d, m, 0.0), b._SelectParams(chunk, 13, keep)
layers = (ctypes.c_void_p * L)(*[x.data_ptr() for x in k])
lp = ctypes.cast(layers, ctypes.POINTER(ctypes.c_void_p))
size = spf.lib.spf_compress_host_arena_bytes(ctypes.byref(shape), n, ctypes.byref(prm))

def compress(arena):
    out = [torch.full((n,), -1, dtype=torch.int32), torch.full((n,), -1, dtype=torch.int32), torch.full((n, 2), -1, dtype=torch.int32),
           torch.full((n, 2), -1, dtype=torch.int32), torch.zeros(2, dtype=torch.int64)]
    rc = spf.lib.spf_compress_host(ctypes.byref(shape), n, lp, q.data_ptr(), ids.data_ptr(), ids.data_ptr(), ids.data_ptr(), ctypes.byref(prm),
                                   arena, size, *[t.data_ptr() for t in out], None)
    return rc, out

first = compress(torch.empty(size, dtype=torch.uint8, device="cuda").data_ptr())
assert first[0] == 0, spf.spf_last_error()
cu = ctypes.CDLL("libcuda.so.1")
ctx, ptr, dev = ctypes.c_void_p(), ctypes.c_uint64(), ctypes.c_int()
assert cu.cuDeviceGet(ctypes.byref(dev), 0) == 0 and cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, dev) == 0
assert cu.cuMemAlloc_v2(ctypes.byref(ptr), ctypes.c_size_t(size)) == 0
second = compress(ptr.value)
assert second[0] == 0, spf.spf_last_error()
assert all(torch.equal(x, y) for x, y in zip(first[1], second[1]))
"""


def test_a_second_context_on_the_device():
    """What a kernel is allowed in one context says nothing about another's.  All device memory of the second call is its own
    context's; the call either runs or is refused by the host."""
    proc = subprocess.run([sys.executable, "-c", TWO_CONTEXTS], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert proc.returncode == 0, proc.stderr[-2000:]
