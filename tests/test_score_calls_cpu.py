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
