"""The no-allocation preconditioner call as a program's first preconditioner call, in a process of
its own: every kernel it launches was loaded when the handle was factored, whichever right-hand-side
tile the batch takes (3-D: 1, 4, 8, 16 wide in complex64, 1 and 2 in complex128; 2-D: 1 and 4), so the
device's free memory does not change across the call."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys
import numpy as np, torch
from paper_1208_3956_gb300 import helm, media
n, prec, B = eval(sys.argv[1]), sys.argv[2], int(sys.argv[3])
c = media.smooth_medium(n, 2.0, 1.0, 2.0, 7)
g = helm.HelmDD(c, 1.0 / 24, media.omega_for(c, 1.0 / 24, 8.0), 2, 3, 2, prec).factor()
f = torch.as_tensor(media.random_rhs((B,) + g.shape, 31), device="cuda")
out = torch.empty_like(f)
torch.cuda.synchronize()
free0 = torch.cuda.mem_get_info()[0]
g.apply_precond_noalloc(f, out=out)
torch.cuda.synchronize()
free1 = torch.cuda.mem_get_info()[0]
print("CHANGE", free0 - free1)
"""


@pytest.mark.parametrize("n,prec,B", [((13, 9, 11), "mixed", 5), ((13, 9, 11), "mixed", 9), ((13, 9, 11), "fp64", 2),
                                      ((31, 29), "mixed", 2)])
def test_first_call_of_a_process_allocates_nothing(n, prec, B):
    r = subprocess.run([sys.executable, "-c", CODE, repr(n), prec, str(B)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["CHANGE", "0"], r.stdout
