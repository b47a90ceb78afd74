"""Low-order form at the edges of its observable lists and sample blocks, against
the FP64 oracle: observables of 63 to 66 qubits (64 are listed), of few and of
more than 256 pairs, empty ones, all in one call; samples one short of and one
past 1024; H in one K piece and in several; a workspace without the lists.
Tolerances are the form's own (1e-5 on estimates, 1e-4 relative on gradients)."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def problem(n, s, gates):
    """Observables of 0, 1, 2, 23, 24, 63, 64, 65, 66 qubits and all of them, in a shuffled order."""
    rng = I.Rng(n + s)
    G = I.local_gates_packed(n) if gates == "all" else I.random_k_body(rng, gates, n, [1, 2], 1)
    th = (0.5 * rng.normal(G.shape[0], 2) / np.sqrt(G.shape[0])).astype(np.float32)
    weights = [w for w in (64, 0, 23, 66, 1, 63, 24, 2, 65, n, 5, 64) if w <= n]
    bits = np.zeros((len(weights), n), dtype=np.uint8)
    for r, w in enumerate(weights):
        bits[r, np.argsort(rng.uniform(n, 50 + r))[:w]] = 1
    l = len(weights)
    return G, th, I.pack_bits(bits), I.uniform_bits(rng, s, n, 6), rng.normal(l, 7) / s, rng.normal(l, 8) / s


def check(n, G, th, A, Z, al, be, ev, se, g):
    t64 = th.astype(np.float64)
    want, want_se, _, _ = oracle.expval(n, G, A, Z, t64)
    want_g = oracle.expval_grad(n, G, A, Z, t64, al, be)
    assert np.max(np.abs(ev.cpu().numpy() - want)) <= 1e-5 and np.max(np.abs(se.cpu().numpy() - want_se)) <= 1e-5
    assert np.linalg.norm(g.cpu().numpy() - want_g) <= 1e-4 * np.linalg.norm(want_g)


@pytest.mark.parametrize("n,s,gates", [(67, 1023, "all"), (130, 1025, 900), (70, 3000, "all"), (300, 257, 5000), (20, 5, 60)])
def test_lists_match_oracle(n, s, gates):
    import torch
    from paper_2501_04776_gb300 import api
    G, th, A, Z, al, be = problem(n, s, gates)
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd, ald, bed = (torch.from_numpy(x).cuda() for x in (th, al, be))
    ev, se, phi = api.expval_keep_phi_raw(n, thd, Gd, Ad, Zd, "loworder_fp32")
    g = api.expval_grad(n, thd, Gd, Ad, Zd, ald, bed, "loworder_fp32")
    kept = api.expval_grad_from_phi(n, thd, Gd, Ad, Zd, phi, ald, bed, "loworder_fp32")
    one = api.expval_value_and_grad(n, thd, Gd, Ad, Zd, ald, bed, "loworder_fp32")
    check(n, G, th, A, Z, al, be, ev, se, g)
    assert torch.equal(g, kept) and torch.equal(ev, one[0]) and torch.equal(se, one[1]) and torch.equal(g, one[2])
    assert api.read_status() == 0


def test_small_workspace_takes_the_block_form():
    import torch
    from paper_2501_04776_gb300 import _lib, api
    n, s = 70, 1500
    G, th, A, Z, al, be = problem(n, s, "all")
    m, l = G.shape[0], A.shape[0]
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd, ald, bed = (torch.from_numpy(x).cuda() for x in (th, al, be))
    lib = _lib.load()
    full = api.workspace_bytes(_lib.OP_EXPVAL_GRAD, n, m, l, s, 0, "loworder_fp32")
    ws = torch.zeros(full, dtype=torch.uint8, device="cuda")
    ev, se = (torch.empty(l, dtype=torch.float64, device="cuda") for _ in range(2))
    g = torch.empty(m, dtype=torch.float64, device="cuda")

    def p(t):
        return ctypes.c_void_p(t.data_ptr())

    for nbytes in (full, full - 256):
        rc = lib.iqp_expval_value_and_grad(n, p(Gd), m, Gd.shape[1], p(Ad), l, Ad.shape[1], p(Zd), s, Zd.shape[1], p(thd),
                                           p(ald), p(bed), _lib.LOWORDER_FP32, p(ev), p(se), p(g), p(ws), nbytes,
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        check(n, G, th, A, Z, al, be, ev, se, g)
