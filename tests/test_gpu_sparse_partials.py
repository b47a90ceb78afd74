"""Row-sparse statistics where the workspace has room for a partial per 2048 samples
only, as before partials of 1024: what such a workspace took, it still takes, and the
results are those of the full one to FP64 rounding (the two ranges' sums are
merged in FP64; 1e-14 of values of order one, standard errors 1e-12 relative)."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def problem(n, m, l, s):
    rng = I.Rng(n + s)
    G = I.random_k_body(rng, m, n, [1, 2, 3], 1) if m else I.local_gates_packed(n)
    th = (0.5 * rng.normal(G.shape[0], 2) / np.sqrt(G.shape[0])).astype(np.float32)
    return G, th, I.bernoulli_bits(rng, l, n, 0.2, 3), I.uniform_bits(rng, s, n, 4), rng.normal(l, 5) / s


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("l,s", [(3, 1025), (700, 2047), (700, 2048), (5, 2049), (900, 5000), (2, 7169)])
def test_pairs_of_ranges(l, s):
    import torch
    from paper_2501_04776_gb300 import _lib, api
    n = 40
    G, th, A, Z, al = problem(n, 500, l, s)
    m, lib = G.shape[0], _lib.load()
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd, ald = torch.from_numpy(th).cuda(), torch.from_numpy(al).cuda()
    full = api.workspace_bytes(_lib.OP_EXPVAL_GRAD, n, m, l, s, 0, "sparse_fp32")
    ws = torch.zeros(full, dtype=torch.uint8, device="cuda")

    def run(nbytes):
        ev, se = (torch.empty(l, dtype=torch.float64, device="cuda") for _ in range(2))
        g = torch.empty(m, dtype=torch.float64, device="cuda")
        st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert lib.iqp_expval_value_and_grad(n, ptr(Gd), m, Gd.shape[1], ptr(Ad), l, Ad.shape[1], ptr(Zd), s, Zd.shape[1],
                                             ptr(thd), ptr(ald), None, _lib.SPARSE_FP32, ptr(ev), ptr(se), ptr(g), ptr(ws),
                                             nbytes, st) == 0
        return ev.cpu().numpy(), se.cpu().numpy(), g.cpu().numpy()

    a, b = run(full), run(full - 256)
    assert np.max(np.abs(a[0] - b[0])) <= 1e-14 and np.array_equal(a[2], b[2])
    assert np.max(np.abs(a[1] - b[1])) <= 1e-12 * np.max(a[1]) + 1e-16
    want, want_se, _, _ = oracle.expval(n, G, A, Z, th.astype(np.float64))
    assert np.max(np.abs(b[0] - want)) <= 1e-5 and np.max(np.abs(b[1] - want_se)) <= 1e-5


def test_no_alloc_call_takes_what_it_took():
    """64 MiB hold these observables' parities and 16 bytes per 2048 samples, not 32."""
    import torch
    from paper_2501_04776_gb300 import _lib, api
    n, l, s, rows = 8, 1_100_000, 2048, 300
    G, th, A, Z, _ = problem(n, 0, l, s)
    lib = _lib.load()
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd = torch.from_numpy(th).cuda()
    ev, se = (torch.empty(l, dtype=torch.float64, device="cuda") for _ in range(2))
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.iqp_expval_noalloc(n, ptr(Gd), G.shape[0], Gd.shape[1], ptr(Ad), l, Ad.shape[1], ptr(Zd), s, Zd.shape[1],
                                  ptr(thd), _lib.SPARSE_FP32, ptr(ev), ptr(se), st) == 0
    assert lib.iqp_noalloc_read_status(st) == 0
    pick = np.r_[0:rows, l - rows:l]
    want, want_se, _, _ = oracle.expval(n, G, A[pick], Z, th.astype(np.float64))
    assert np.max(np.abs(ev.cpu().numpy()[pick] - want)) <= 1e-5 and np.max(np.abs(se.cpu().numpy()[pick] - want_se)) <= 1e-5
