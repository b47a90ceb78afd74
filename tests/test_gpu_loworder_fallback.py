"""Low-order form where the samples cannot be described to the tensor cores: one
row with a row stride of 2^40 bytes, which no tensor map takes and no kernel steps over. The
contraction is summed without them then, and the results are those of the same row
at its own stride (the tolerances of the form: 1e-5, 1e-4 relative)."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [20, 130, 300])
def test_row_stride_beyond_tensor_maps(n):
    import torch
    from paper_2501_04776_gb300 import _lib, api
    rng = I.Rng(n)
    G = I.local_gates_packed(n)
    th = (rng.normal(G.shape[0], 2) / n).astype(np.float32)
    A, Z = I.bernoulli_bits(rng, 40, n, 0.1, 3), I.uniform_bits(rng, 1, n, 4)
    al = rng.normal(40, 5)
    m, l = G.shape[0], A.shape[0]
    Gd, Ad, Zd = (api.to_device_bits(x) for x in (G, A, Z))
    thd, ald = torch.from_numpy(th).cuda(), torch.from_numpy(al).cuda()
    lib = _lib.load()
    ws = torch.zeros(api.workspace_bytes(_lib.OP_EXPVAL_GRAD, n, m, l, 1, 0, "loworder_fp32"), dtype=torch.uint8,
                     device="cuda")
    ev = torch.empty(l, dtype=torch.float64, device="cuda")
    g = torch.empty(m, dtype=torch.float64, device="cuda")

    def p(t):
        return ctypes.c_void_p(t.data_ptr())

    rc = lib.iqp_expval_value_and_grad(n, p(Gd), m, Gd.shape[1], p(Ad), l, Ad.shape[1], p(Zd), 1, 1 << 37, p(thd), p(ald),
                                       None, _lib.LOWORDER_FP32, p(ev), None, p(g), p(ws), ws.numel(),
                                       ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0 and lib.iqp_read_status(p(ws), ws.numel(), None) == 0
    t64 = th.astype(np.float64)
    want, _, _, _ = oracle.expval(n, G, A, Z, t64)
    want_g = oracle.expval_grad(n, G, A, Z, t64, al, None)
    assert np.max(np.abs(ev.cpu().numpy() - want)) <= 1e-5
    assert np.linalg.norm(g.cpu().numpy() - want_g) <= 1e-4 * np.linalg.norm(want_g)
