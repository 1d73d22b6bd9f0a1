"""The extension module belongs to the Python and the torch in its name; without one of their own, other interpreters use the library all the same."""
import os
import subprocess
import sys

import torch

import paper_2502_08141_b200 as lw

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_another_torch_takes_the_interpreted_way():
    from paper_2502_08141_b200 import build
    build.build()
    assert torch.__version__ in lw.PY_CALLS_PATH and os.path.exists(lw.PY_CALLS_PATH)
    code = """
import warnings
import numpy as np
import torch
torch.__version__ = "0.0.0+another"
import paper_2502_08141_b200 as lw
with warnings.catch_warnings(record=True) as seen:
    warnings.simplefilter("always")
    plan = lw.lowra_plan(np.array([1, 2, 4, 1], np.uint8), 128)
    lw.lib()
assert plan["packed_bytes"] == 128
assert [w.category for w in seen] == [RuntimeWarning] and "interpreted" in str(seen[0].message), seen
assert lw._py_calls is None and not lw._fits(0)
"""
    subprocess.run([sys.executable, "-c", code], cwd=ROOT, check=True, timeout=300)


def test_own_module_is_loaded():
    from paper_2502_08141_b200 import build
    build.build()
    lw.lib()
    assert lw._py_calls is not None and lw._fits is lw._py_calls.fits
