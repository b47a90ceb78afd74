"""Row-sparse form at the edges of its gate lists and sample ranges, against
the FP64 oracle: rows with more odd gates than one list holds (4096), rows of
more words than one listing step (2048), runs of set bits (whole-warp words)
beside lone ones, batches that do not fill (five gates, 32 gates), ranges of
1024 samples with one sample more or less. Tolerances are the form's own
(1e-5 on estimates, 1e-4 relative on gradients)."""
import numpy as np
import pytest

import oracle
from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# n, gates, l, s, observable bit probability
CASES = [(20, 9000, 5, 1025, 0.5), (520, "local", 6, 1024, 0.02), (64, 64, 1, 31, 0.3), (3, 4, 3, 33, 0.5),
         (90, 161, 7, 2047, 0.1), (40, "local", 33, 3000, 0.1)]


def problem(n, gates, l, s, p, indep=False):
    rng = I.Rng(7 * n + l)
    G = I.local_gates_packed(n) if gates == "local" else I.random_k_body(rng, gates, n, [1, 2, 3], 1)
    th = (0.5 * rng.normal(G.shape[0], 2) / np.sqrt(G.shape[0])).astype(np.float32)
    A = I.bernoulli_bits(rng, l, n, p, 5)
    A[0] = 0  # no odd gate at all
    return G, th, A, I.uniform_bits(rng, l * s if indep else s, n, 6), rng.normal(l, 7) / s, rng.normal(l, 8) / s


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("case", CASES, ids=["n%d-%s-l%d-s%d" % c[:4] for c in CASES])
def test_shared_batches_match_oracle(case):
    import torch
    from paper_2501_04776_gb300 import api
    n, (G, th, A, Z, al, be) = case[0], problem(*case)
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd, ald, bed = (torch.from_numpy(x).cuda() for x in (th, al, be))
    t64 = th.astype(np.float64)
    want, want_se, _, _ = oracle.expval(n, G, A, Z, t64)
    want_g = oracle.expval_grad(n, G, A, Z, t64, al, be)
    ev, se = api.expval_raw(n, thd, Gd, Ad, Zd, "sparse_fp32")
    g = api.expval_grad(n, thd, Gd, Ad, Zd, ald, bed, "sparse_fp32")
    one = api.expval_value_and_grad(n, thd, Gd, Ad, Zd, ald, bed, "sparse_fp32")
    for e, d, x in ((ev, se, g), one):
        assert np.max(np.abs(e.cpu().numpy() - want)) <= 1e-5
        assert np.max(np.abs(d.cpu().numpy() - want_se)) <= 1e-5
        assert rel(x.cpu().numpy(), want_g) <= 1e-4 or not want_g.any()
    assert torch.equal(ev, one[0]) and torch.equal(g, one[2])


@pytest.mark.parametrize("case", [c for c in CASES if c[1] != "local" or c[0] < 100],
                         ids=["n%d-%s-l%d-s%d" % c[:4] for c in CASES if c[1] != "local" or c[0] < 100])
def test_independent_batches_match_oracle(case):
    import torch
    from paper_2501_04776_gb300 import api
    n, (G, th, A, Z, al, be) = case[0], problem(*case, indep=True)
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd, ald, bed = (torch.from_numpy(x).cuda() for x in (th, al, be))
    t64 = th.astype(np.float64)
    want, want_se, _, _ = oracle.expval_indep(n, G, A, Z, t64)
    ev, se = api.expval_indep_raw(n, thd, Gd, Ad, Zd)
    assert np.max(np.abs(ev.cpu().numpy() - want)) <= 1e-5 and np.max(np.abs(se.cpu().numpy() - want_se)) <= 1e-5
    want_g = oracle.expval_indep_grad(n, G, A, Z, t64, al, be)
    g = api.expval_indep_grad(n, thd, Gd, Ad, Zd, ald, bed).cpu().numpy()
    assert rel(g, want_g) <= 1e-4 or not want_g.any()
