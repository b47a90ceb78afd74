"""Low-order form at the limits of its observable lists, 128 qubits (64 where
the observables and samples are few) and 256 pairs, against the FP64 oracle:
observables one below, at and one above each, alone over the limit and beside
listed ones, with sample counts that end inside a lane's four.
Tolerances are the form's own (1e-5 on estimates, 1e-4 relative on gradients)."""
import numpy as np
import pytest

import oracle
from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu

N = 300


def by_qubits():
    """400 pairs over 300 qubits (an observable of 128 has about 70 of them), 127 to 129 qubits."""
    rng = I.Rng(4)
    gates = [[q] for q in range(N)] + [sorted(int(q) for q in np.argsort(rng.uniform(N, 100 + k))[:2]) for k in range(400)]
    rows = []
    for r, w in enumerate((127, 128, 129, 128, 129, 1, 127)):
        rows.append(np.argsort(rng.uniform(N, 50 + r))[:w])
    return gates, rows


def by_pairs():
    """All 253 pairs of 23 qubits and a chain from the last: 253 + j pairs on 23 + j qubits."""
    gates = [[q] for q in range(N)] + [[q, r] for q in range(23) for r in range(q + 1, 23)]
    gates += [[q, q + 1] for q in range(22, 60)]
    return gates, [np.arange(23 + j) for j in (2, 3, 4, 0, 3, 4)] + [np.arange(200, 240)]


@pytest.mark.parametrize("repeat,s", [(1, 1021), (1, 2050), (100, 1021)])
@pytest.mark.parametrize("build,edges", [(by_qubits, [127, 128, 129]), (by_pairs, [255, 256, 257])], ids=["qubits", "pairs"])
def test_limits_match_oracle(build, edges, repeat, s):
    import torch
    from paper_2501_04776_gb300 import api
    gates, rows = build()
    pairs = {tuple(g) for g in gates if len(g) == 2}
    inside = [sum(a in r and b in r for a, b in pairs) for r in (set(r.tolist()) for r in rows)]
    sizes = [len(r) for r in rows]
    assert set(edges) <= set(sizes if build is by_qubits else inside)  # the edges are there ...
    assert max(inside if build is by_qubits else sizes) <= 100          # ... and the other limit is far
    rows = rows * repeat
    bits = np.zeros((len(rows), N), dtype=np.uint8)
    for k, r in enumerate(rows):
        bits[k, r] = 1
    rng = I.Rng(s)
    G, A, Z = I.pack_index_lists(gates, N), I.pack_bits(bits), I.uniform_bits(rng, s, N, 6)
    th = (0.5 * rng.normal(len(gates), 2) / np.sqrt(len(gates))).astype(np.float32)
    al, be = rng.normal(len(rows), 7) / s, rng.normal(len(rows), 8) / s
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd, ald, bed = (torch.from_numpy(x).cuda() for x in (th, al, be))
    ev, se, phi = api.expval_keep_phi_raw(N, thd, Gd, Ad, Zd, "loworder_fp32")
    g = api.expval_grad(N, thd, Gd, Ad, Zd, ald, bed, "loworder_fp32")
    kept = api.expval_grad_from_phi(N, thd, Gd, Ad, Zd, phi, ald, bed, "loworder_fp32")
    one = api.expval_value_and_grad(N, thd, Gd, Ad, Zd, ald, bed, "loworder_fp32")
    assert api.read_status() == 0
    t64 = th.astype(np.float64)
    want, want_se, _, _ = oracle.expval(N, G, A, Z, t64)
    want_g = oracle.expval_grad(N, G, A, Z, t64, al, be)
    for e, d in ((ev, se), one[:2]):
        assert np.max(np.abs(e.cpu().numpy() - want)) <= 1e-5 and np.max(np.abs(d.cpu().numpy() - want_se)) <= 1e-5
    for x in (g, kept, one[2]):
        assert np.linalg.norm(x.cpu().numpy() - want_g) <= 1e-4 * np.linalg.norm(want_g)


def test_more_heavy_observables_than_blocks():
    """1000 observables of 130 to 140 qubits and 5000 samples: 2000 work items for at most five blocks per SM."""
    import torch
    from paper_2501_04776_gb300 import api
    n, l, s = 140, 1000, 5000
    rng = I.Rng(9)
    G = I.random_k_body(rng, 300, n, [1, 2], 1)
    bits = np.ones((l, n), dtype=np.uint8)
    for a in range(l):
        bits[a, np.argsort(rng.uniform(n, 100 + a))[:a % 11]] = 0
    A, Z = I.pack_bits(bits), I.uniform_bits(rng, s, n, 3)
    th = (0.5 * rng.normal(300, 2) / np.sqrt(300)).astype(np.float32)
    al, be = rng.normal(l, 7) / s, rng.normal(l, 8) / s
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd, ald, bed = (torch.from_numpy(x).cuda() for x in (th, al, be))
    ev, se = api.expval_raw(n, thd, Gd, Ad, Zd, "loworder_fp32")
    g = api.expval_grad(n, thd, Gd, Ad, Zd, ald, bed, "loworder_fp32")
    assert api.read_status() == 0
    t64 = th.astype(np.float64)
    want, want_se, _, _ = oracle.expval(n, G, A, Z, t64)
    want_g = oracle.expval_grad(n, G, A, Z, t64, al, be)
    assert np.max(np.abs(ev.cpu().numpy() - want)) <= 1e-5 and np.max(np.abs(se.cpu().numpy() - want_se)) <= 1e-5
    assert np.linalg.norm(g.cpu().numpy() - want_g) <= 1e-4 * np.linalg.norm(want_g)
