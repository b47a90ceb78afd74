"""The finaliser's quotients (a reciprocal from the host and one correction by the
exact remainder) are FP64 division's, bit for bit. Gates on one qubit each with theta = pi / 4
and observables of two qubits: every phase is 0 or +-pi, every cosine 1 or -1, so the sum is
an integer and the estimate has to be that integer divided by the number of samples."""
import numpy as np
import pytest

from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SIZES = [3, 7, 49, 63, 65, 129, 777, 1023, 2501, 10_007, 16_385]


@pytest.mark.parametrize("form", ["fp32", "split_bf16", "sparse_fp32", "loworder_fp32"])
def test_quotients_are_exact(form):
    import torch
    from paper_2501_04776_gb300 import api
    n = 120
    G = api.to_device_bits(I.pack_index_lists([[q] for q in range(n)], n))
    A = api.to_device_bits(I.pack_index_lists([[q, q + 1] for q in range(0, n, 2)], n))
    th = torch.full((n,), np.pi / 4, dtype=torch.float32, device="cuda")
    differ = 0
    for s in SIZES:
        Z = I.uniform_bits(I.Rng(s), s, n, 1)
        bits = I.unpack_bits(Z, n)
        total = (1 - 2 * (bits[:, 0::2] == bits[:, 1::2])).sum(0).astype(np.float64)
        ev = api.expval_raw(n, th, G, A, api.to_device_bits(Z), form)[0].cpu().numpy()
        assert np.array_equal(ev, total / s)
        differ += int((total * (1.0 / s) != total / s).sum())
    assert differ > 50  # the reciprocal alone would show
