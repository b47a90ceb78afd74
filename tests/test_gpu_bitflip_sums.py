"""The bitflip model's integer sums (from 2^25 parity bits on) against the FP64
oracle, and where they hand over to the FP64 kernels: negative cosines, words
that do not fill a table block, logarithms that sum past the limit, a parameter
that is not a number. The values' tolerance is the model's (1e-12 absolute), the
gradient's 1e-10 relative; both sides are FP64 to the last bits."""
import numpy as np
import pytest

import oracle
from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,l,kind", [(60, 9001, 4000, "small"), (50, 2049, 16400, "negative"), (200, 33600, 1025, "small"),
                                        (40, 6000, 6000, "large"), (60, 9001, 4000, "zero")])
def test_values_and_gradient(n, m, l, kind):
    import torch
    from paper_2501_04776_gb300 import api
    rng = I.Rng(m)
    G = I.random_k_body(rng, m, n, [1, 2, 3], 1)
    th = 0.05 * (2 * rng.uniform(m, 2) - 1)
    if kind == "negative":
        th[::97] = 1.2
    elif kind == "large":
        th *= 60
    elif kind == "zero":
        th[:] = 0
    th = th.astype(np.float32)
    A = I.bernoulli_bits(rng, l, n, 0.05, 3)
    w = rng.normal(l, 4)
    args = (n, torch.from_numpy(th).cuda(), api.to_device_bits(G), api.to_device_bits(A))
    ev = api.bitflip_expval_raw(*args).cpu().numpy()
    g = api.bitflip_grad(*args, torch.from_numpy(w).cuda()).cpu().numpy()
    want = oracle.bitflip_expval(n, G, A, th.astype(np.float64))
    want_g = oracle.bitflip_grad(n, G, A, th.astype(np.float64), w)
    assert np.max(np.abs(ev - want)) <= 1e-12
    big = np.abs(want) > 1e-290
    assert np.max(np.abs(ev[big] / want[big] - 1)) <= 1e-11  # sign and digits of small values too
    assert np.linalg.norm(g - want_g) <= 1e-10 * np.linalg.norm(want_g) if want_g.any() else not g.any()


def test_not_a_number_stays_in_its_rows():
    import torch
    from paper_2501_04776_gb300 import api
    n, m, l = 60, 9001, 4000
    rng = I.Rng(3)
    G, A = I.random_k_body(rng, m, n, [1, 2], 1), I.bernoulli_bits(rng, l, n, 0.05, 3)
    th = (0.05 * rng.normal(m, 2)).astype(np.float32)
    th[17] = 0
    odd = oracle.parity(n, A, G[17:18])[:, 0].astype(bool)
    want = oracle.bitflip_expval(n, G, A, th.astype(np.float64))
    th[17] = np.nan
    ev = api.bitflip_expval_raw(n, torch.from_numpy(th).cuda(), api.to_device_bits(G), api.to_device_bits(A)).cpu().numpy()
    assert np.isnan(ev[odd]).all() and np.max(np.abs(ev[~odd] - want[~odd])) <= 1e-12
