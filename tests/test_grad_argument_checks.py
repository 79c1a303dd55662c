"""psr_grad refuses empty batches and empty sequences at every precision, before
it looks at the context or the arrays (no GPU needed: the context handle is a
placeholder).  A child process, because a crash must not end the run."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
@pytest.mark.parametrize("n,L", [(1, 0), (0, 4), (1, -1), (-1, 4)])
def test_empty_sizes_are_refused(precision, n, L):
    code = (
        "import sys, numpy as np\n"
        "from paper_2605_13807_gb300 import binding as B, inputs\n"
        "t = inputs.glorot_params(3, 128, seed=0)\n"
        "p = B.make_params(t, 3, 128, False, sys.argv[1], ctx=1)\n"
        "s, g = np.zeros(4, np.uint8), np.zeros_like(t)\n"
        "import ctypes as C\n"
        "print(B.lib().psr_grad(C.byref(p), B._ptr(s), int(sys.argv[2]), int(sys.argv[3]), None, B._ptr(g)))\n")
    r = subprocess.run([sys.executable, "-c", code, precision, str(n), str(L)], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr[-500:])
    assert int(r.stdout) == 1  # PSR_EINVAL
