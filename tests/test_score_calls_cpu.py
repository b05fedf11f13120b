"""Host side of the scoring calls: what a batch needs and is refused for, without a device."""
import ctypes
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HUGE = """
import ctypes, paper_2603_02631_b200 as spf
from paper_2603_02631_b200 import binding as b
forms = {"": b._Prompt(0, None, 0, 0, None, None, None), "_paged": b._PagedPrompt(0, None, 1, 128, 4096, None, None, None),
         "_fp8": b._Fp8Prompt(0, None, 0, 0, 4096, None, None, None)}
shape = b._Shape(2, 4, 2, 64, 8, 0.0)
for form, prompt in forms.items():
    arr = (type(prompt) * 1)(prompt)
    score, size = getattr(spf.lib, "spf_score" + form), getattr(spf.lib, "spf_score" + form + "_workspace_bytes")
    assert score(ctypes.byref(shape), arr, 2**31 - 1, None, 0, None, None) == -1, form
    assert size(ctypes.byref(shape), arr, 2**31 - 1) == 0, form
    assert "n_tokens" in spf.spf_last_error()
"""


def test_a_batch_of_any_size_is_refused_with_a_status():
    """Nothing is allocated by the number of prompts: the first one is looked at, and found empty.  (In a process of its own:
    an exception that left the C entry would end it.)"""
    proc = subprocess.run([sys.executable, "-c", HUGE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert proc.returncode == 0, proc.stderr[-2000:]


WORKSPACE = """
import ctypes, paper_2603_02631_b200 as spf
from paper_2603_02631_b200 import binding as b
L = 4
shape = b._Shape(L, 16, 4, 64, 8, 0.0)
layers = (ctypes.c_void_p * L)(*([1 << 20] * L))
lp = ctypes.cast(layers, ctypes.POINTER(ctypes.c_void_p))
p = 1 << 20
make = {"": lambda n: b._Prompt(n, lp, n * 64, 64, p, p, None), "_paged": lambda n: b._PagedPrompt(n, lp, 4096, 128, p, p, p, None),
        "_fp8": lambda n: b._Fp8Prompt(n, lp, n * 64, 64, p, p, p, None)}
lens = [300, 40000, 17, 25000, 40000, 128] * 5
for form, one in make.items():
    score, size = getattr(spf.lib, "spf_score" + form), getattr(spf.lib, "spf_score" + form + "_workspace_bytes")
    batch = (type(one(1)) * len(lens))(*[one(n) for n in lens])
    alone = max(size(ctypes.byref(shape), (type(one(1)) * 1)(one(n)), 1) for n in set(lens))
    together = size(ctypes.byref(shape), batch, len(lens))
    assert 0 < alone < together
    # without a device a call that gets past the checks ends with SPF_ERR_CUDA
    assert score(ctypes.byref(shape), batch, len(lens), 256, together, None, None) == -4
    assert score(ctypes.byref(shape), batch, len(lens), 256, alone, None, None) == -4, form
    assert score(ctypes.byref(shape), batch, len(lens), 256, alone - 1, None, None) == -3
"""


def test_a_workspace_for_the_longest_prompt_is_enough_for_a_batch():
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")       # the pointers are made up: no device may be reached
    proc = subprocess.run([sys.executable, "-c", WORKSPACE], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert proc.returncode == 0, proc.stderr[-2000:]
