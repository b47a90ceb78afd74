"""Low-order gradient without the tensor cores (IQP_LO_TC=0): the pair sums H are
added up in FP64 over the ranges of 2048 samples, as they were, so a pair whose
range sums are exact in FP32 is exact. One gate on qubit 0 with 2 theta = pi / 2, one
on {0, 1} with theta = 0, the observable {0}, z_1 = 0: every s_0 W is alpha, and
both gradients are 2 s alpha. alpha = 1 + 2^-19: 16 of them add up exactly in 24
bits, 39 ranges do not."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
S = 2048 * 39  # whole ranges: any other count's sum would round in FP32 itself

CODE = """
import sys, numpy as np, torch
sys.path.insert(0, %r)
from paper_2501_04776_gb300 import api
from paper_2501_04776_gb300 import inputs as I
n, s = 2, %d
Z = I.uniform_bits(I.Rng(1), s, 1, 2)
Z[:, 0] &= np.uint64(1)
G, A = I.pack_bits(np.array([[1, 0], [1, 1]])), I.pack_bits(np.array([[1, 0]]))
th = torch.tensor([np.pi / 4, 0.0], dtype=torch.float32, device="cuda")
al = torch.tensor([1 + 2.0 ** -19], dtype=torch.float64, device="cuda")
g = api.expval_grad(n, th, *(api.to_device_bits(x) for x in (G, A, Z)), al, None, "loworder_fp32")
assert api.read_status() == 0
print(*(float(x).hex() for x in g.cpu()))
"""


def test_ranges_add_up_in_fp64():
    out = subprocess.run([sys.executable, "-c", CODE % (ROOT, S)], check=True, timeout=300, capture_output=True, text=True,
                         env=dict(os.environ, IQP_LO_TC="0"), cwd=ROOT).stdout.split()
    want = 2 * S * (1 + 2.0 ** -19)
    assert [float.fromhex(x) for x in out] == [want, want]
