"""Last rounds of phase tiles cut into equal ranges over the chip, against the FP64
oracle on sampled observables: tile counts that leave few, about three quarters
and nearly all of the CTA pairs' number over, so that a tile lies in one to
many ranges. Tolerances: the forms' own (1e-4 split BF16, 1e-5 FP32; gradients
1e-4 relative)."""
import numpy as np
import pytest

import oracle
from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# tiles of 256 observables x 512 (split BF16, a round and more) or 256 samples, on 76 CTA pairs
@pytest.mark.parametrize("form,m,l,s", [("split_bf16", 2100, 4096, 16_384), ("split_bf16", 2100, 2560, 7600),
                                        ("split_bf16", 1030, 256, 19_000), ("split_bf16", 5000, 500, 14_000),
                                        ("fp32", 9000, 2560, 3300), ("fp32", 2100, 256, 34_000), ("fp32", 2100, 300, 700)])
def test_ragged_rounds_match_oracle(form, m, l, s):
    import torch
    from paper_2501_04776_gb300 import api
    n, rows = 300, 16
    rng = I.Rng(m + l)
    G, A, Z = I.random_k_body(rng, m, n, [1, 2, 3], 1), I.bernoulli_bits(rng, l, n, 0.1, 3), I.uniform_bits(rng, s, n, 4)
    th = (0.6 * rng.normal(m, 2) / np.sqrt(m)).astype(np.float32)
    pick = np.sort(rng.integers(rows, l, 5))
    pick = np.unique(np.r_[0, pick, l - 1])
    al = np.zeros(l)
    al[pick] = rng.normal(len(pick), 6) / s
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd, ald = torch.from_numpy(th).cuda(), torch.from_numpy(al).cuda()
    one = api.expval_value_and_grad(n, thd, Gd, Ad, Zd, ald, None, form)
    ev, _ = api.expval_raw(n, thd, Gd, Ad, Zd, form)
    g = api.expval_grad(n, thd, Gd, Ad, Zd, ald, None, form)
    assert api.read_status() == 0
    t64, tol = th.astype(np.float64), 1e-4 if form == "split_bf16" else 1e-5
    want, want_se, _, _ = oracle.expval(n, G, A[pick], Z, t64)
    want_g = oracle.expval_grad(n, G, A[pick], Z, t64, al[pick], None)
    for e in (one[0], ev):
        assert np.max(np.abs(e.cpu().numpy()[pick] - want)) <= tol
        assert bool(torch.isfinite(e).all())
    assert np.max(np.abs(one[1].cpu().numpy()[pick] - want_se)) <= tol
    for x in (one[2], g):
        assert np.linalg.norm(x.cpu().numpy() - want_g) <= 1e-4 * np.linalg.norm(want_g)
    # every observable, not the sampled ones alone: the same estimates from the two calls and from the row-sparse form
    ref, _ = api.expval_raw(n, thd, Gd, Ad, Zd, "sparse_fp32")
    for e in (one[0], ev):
        assert float((e - ref).abs().max()) <= tol + 1e-5
