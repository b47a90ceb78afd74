"""The FP32 form on the tensor cores (three BF16 planes of 2 theta and of W,
the first on an integer grid): estimates, standard errors and gradients against
the FP64 oracle, beside the SIMT kernels (IQP_FP32_TC=0) on the same inputs,
at the edges of tiles, planes and accumulation chunks.

Tolerances. A plane triple keeps 2 theta_j to 2^-26 of the largest |2 theta|
(at most pi after reduction) and the phase is rounded to FP32 a few times, so
|dPhi| <= nnz 2^-26 cmax + 2^-22 |Phi|, with nnz <= m gates per observable; an
estimate moves by at most that. The gradient's tolerance is the library's
1e-4; its error may not exceed the SIMT kernels' by more than 1e-6."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# n, m, l, s, theta: sizes at and one past tiles of 128 / 256, one observable
# (its estimate by the SIMT kernels, its gradient on the tensor cores), more
# gates than one accumulation chunk (65536)
CASES = [(8, 36, 1, 2000, "normal"), (70, 513, 128, 129, "normal"), (130, 1027, 257, 1025, "wide"), (64, 500, 129, 640, "zero"),
         (40, 300, 300, 257, "turns"), (200, 70_001, 5, 300, "normal"), (100, 9001, 140, 2000, "spread")]


def problem(n, m, l, s, kind):
    rng = I.Rng(100 + m)
    G = I.random_k_body(rng, m, n, [1, 2, 3], 1)
    th = rng.normal(m, 2) * 0.6 / np.sqrt(m)
    if kind == "wide":      # a few parameters far above the rest
        th[::200] *= 200
    elif kind == "zero":
        th[:] = 0
    elif kind == "turns":   # beyond a full turn: only 2 theta mod 2 pi matters
        th += np.pi * np.round(3 * rng.normal(m, 3))
    elif kind == "spread":  # magnitudes over eight decades
        th *= 10.0 ** (-8 * rng.uniform(m, 4))
    A = I.bernoulli_bits(rng, l, n, 0.1, 5)
    Z = I.uniform_bits(rng, s, n, 6)
    return G, th.astype(np.float32), A, Z, rng.normal(l, 7) / s, rng.normal(l, 8) / s


def results(case):
    """(expval, std_err, gradient, and the same from the one-call form) with the library this process loaded."""
    import torch
    from paper_2501_04776_gb300 import api
    n = case[0]
    G, th, A, Z, al, be = problem(*case)
    G, A, Z = (api.to_device_bits(x) for x in (G, A, Z))
    th, al, be = (torch.from_numpy(x).cuda() for x in (th, al, be))
    ev, se = api.expval_raw(n, th, G, A, Z, "fp32")
    g = api.expval_grad(n, th, G, A, Z, al, be, "fp32")
    one = api.expval_value_and_grad(n, th, G, A, Z, al, be, "fp32")
    assert api.read_status() == 0
    return [x.cpu().numpy() for x in (ev, se, g, *one)]


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.fixture(scope="module")
def simt(tmp_path_factory):
    """The SIMT kernels' results of every case, from one child process."""
    out = str(tmp_path_factory.mktemp("simt") / "r.npz")
    code = ("import sys, numpy as np; sys.path[:0] = [%r, %r]\n"
            "import test_gpu_fp32_planes as t\n"
            "np.savez(%r, **{'%%d_%%d' %% (i, k): x for i, c in enumerate(t.CASES) for k, x in enumerate(t.results(c))})"
            % (ROOT, os.path.dirname(os.path.abspath(__file__)), out))
    subprocess.run([sys.executable, "-c", code], check=True, timeout=300, env=dict(os.environ, IQP_FP32_TC="0"), cwd=ROOT)
    return np.load(out)


@pytest.mark.parametrize("k", range(len(CASES)), ids=["%s-m%d-l%d-s%d" % (c[4], *c[1:4]) for c in CASES])
def test_planes_match_oracle_and_simt(simt, k):
    n, m, l, s, kind = CASES[k]
    G, th, A, Z, al, be = problem(*CASES[k])
    got = results(CASES[k])
    t64 = th.astype(np.float64)
    ev, se, _, _ = oracle.expval(n, G, A, Z, t64)
    grad = oracle.expval_grad(n, G, A, Z, t64, al, be)
    nnz = int(oracle.parity(n, A, G).sum(1).max())
    c = np.abs(np.remainder(2 * t64 + np.pi, 2 * np.pi) - np.pi)
    phi = np.sqrt(nnz) * c.std() * 6 + c.max()
    tol = nnz * 2.0 ** -26 * c.max() + 2.0 ** -22 * phi + 2.0 ** -23  # the last: cosf itself
    for e, d, g in (got[:3], got[3:]):
        assert np.max(np.abs(e - ev)) <= tol
        assert np.max(np.abs(d - se)) <= tol
        assert rel(g, grad) <= 1e-4 if np.linalg.norm(grad) else not g.any()
    if s > 1 and kind != "zero":
        err = [rel(got[2], grad), rel(simt["%d_2" % k], grad)]
        assert err[0] <= 1e-6 + err[1], err


def test_small_workspace_runs_the_simt_kernels():
    """A workspace that ends before the planes' regions is accepted, as it was,
    and gives the SIMT kernels' results."""
    import ctypes

    import torch
    from paper_2501_04776_gb300 import _lib, api
    n, m, l, s, _ = CASES[1]
    G, th, A, Z, _, _ = problem(*CASES[1])
    want, _, _, _ = oracle.expval(n, G, A, Z, th.astype(np.float64))
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd = torch.from_numpy(th).cuda()
    lib, ev = _lib.load(), torch.empty(l, dtype=torch.float64, device="cuda")
    full = api.workspace_bytes(_lib.OP_EXPVAL, n, m, l, s, 0, "fp32")
    ws = torch.zeros(full, dtype=torch.uint8, device="cuda")

    def p(t):
        return ctypes.c_void_p(t.data_ptr())

    def call(nbytes):
        return lib.iqp_expval(n, p(Gd), m, Gd.shape[1], p(Ad), l, Ad.shape[1], p(Zd), s, Zd.shape[1], p(thd), _lib.FP32,
                              p(ev), None, p(ws), nbytes, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))

    for nbytes in (full, full - 256, full - 20 * 2 ** 20):
        assert call(nbytes) == 0
        assert np.max(np.abs(ev.cpu().numpy() - want)) <= 1e-5
    assert call(4096) != 0
