"""The MMD loss and gradient where the data parities change route: observable
blocks of low weight (gathered rows of the transposed data), heavy ones (the
dense fold), both in one call, and a workspace that ends before the gather's
scratch; against the FP64 oracle, every flag. Tolerances are the library's
(1e-4 split BF16, 1e-5 FP32 forms, gradients 1e-4 relative); the parity sums
behind them are exact, so a wrong route shows at order one."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {"split_bf16": 1e-4, "fp32": 1e-5, "sparse_fp32": 1e-5, "loworder_fp32": 1e-5}


def problem(n, l, s, N, kind):
    rng = I.Rng(31 * n + l)
    G = I.local_gates_packed(n)[: 40 * n]
    th = (0.4 * rng.normal(G.shape[0], 1) / np.sqrt(n)).astype(np.float32)
    light = I.bernoulli_bits(rng, l, n, 0.03, 2)
    dense = I.bernoulli_bits(rng, l, n, 0.5, 3)
    A = {"light": light, "dense": dense}.get(kind)
    if A is None:  # blocks of 32: all light, all dense, a dense row at the end
        A = light.copy()
        A[32:64] = dense[32:64]
        A[l - 1] = dense[l - 1]
    X = I.prototype_data(rng, N, n, 8, 0.1, 5)
    return G, th, A, I.uniform_bits(rng, s, n, 4), X


@pytest.mark.parametrize("n,l,s,N", [(150, 70, 300, 65), (150, 97, 257, 1000), (200, 33, 129, 9000)])
@pytest.mark.parametrize("kind", ["light", "dense", "mixed"])
@pytest.mark.parametrize("prec", ["split_bf16", "sparse_fp32", "loworder_fp32"])
def test_loss_and_gradient(n, l, s, N, kind, prec):
    import torch
    from paper_2501_04776_gb300 import api
    G, th, A, Z, X = problem(n, l, s, N, kind)
    args = [torch.from_numpy(th).cuda()] + [api.to_device_bits(x) for x in (G, A, Z, X)]
    for unbiased in (True, False):
        for sq in (False, True):
            loss, grad = api.mmd_loss_raw(n, *args, prec, unbiased, with_grad=True, sqrt_loss=sq)
            want, _, want_g = oracle.mmd_loss_ex(n, G, A, Z, X, th.astype(np.float64), unbiased, sq, False, grad=True)
            assert abs(float(loss) - want) <= TOL[prec]
            assert np.linalg.norm(grad.cpu().numpy() - want_g) <= 1e-4 * np.linalg.norm(want_g)
            again, _ = api.mmd_loss_raw(n, *args, prec, unbiased, sqrt_loss=sq)
            assert float(again) == float(loss)
    assert api.read_status() == 0


def test_small_workspace_folds_densely():
    import torch
    from paper_2501_04776_gb300 import _lib, api
    n, l, s, N = 150, 97, 257, 1000
    G, th, A, Z, X = problem(n, l, s, N, "mixed")
    thd = torch.from_numpy(th).cuda()
    Gd, Ad, Zd, Xd = (api.to_device_bits(x) for x in (G, A, Z, X))
    want, _, _ = oracle.mmd_loss_ex(n, G, A, Z, X, th.astype(np.float64), True, False, False, grad=True)
    lib, loss = _lib.load(), torch.empty(1, dtype=torch.float64, device="cuda")
    full = api.workspace_bytes(_lib.OP_MMD_LOSS, n, G.shape[0], l, s, N, "sparse_fp32")
    ws = torch.zeros(full, dtype=torch.uint8, device="cuda")

    def p(t):
        return ctypes.c_void_p(t.data_ptr())

    def call(nbytes):
        return lib.iqp_mmd_loss(n, p(Gd), G.shape[0], Gd.shape[1], p(Ad), l, Ad.shape[1], p(Zd), s, Zd.shape[1], p(Xd), N,
                                Xd.shape[1], p(thd), _lib.SPARSE_FP32, _lib.MMD_UNBIASED, p(loss), p(ws), nbytes,
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))

    for nbytes in (full, full - 256):
        assert call(nbytes) == 0
        assert abs(float(loss) - want) <= 1e-5
