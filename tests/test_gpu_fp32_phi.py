"""FP32 on the tensor cores with Phi kept from the statistics pass: autograd's
gradient with and without keep_phi, the MMD gradient, and the refusals.

W comes from the same FP32 Phi by the same formula, the maxima and integer grids
are those of the same W, and every sum that follows is taken in a fixed order, so
estimates and gradients are equal bit for bit. The MMD gradient against the
row-sparse form (another order of FP32 sums): the library's 1e-4."""
import numpy as np
import pytest

from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# one row and column past the tiles; rows of exactly 2048 samples and one past; a split last round with many parts; more gates
# than an accumulation chunk
CASES = [(60, 300, 257, 257), (80, 2050, 3, 2048), (80, 2050, 3, 2049), (40, 9001, 130, 100), (200, 70_001, 5, 300)]


def problem(n, m, l, s):
    rng = I.Rng(7 + m + s)
    th = (rng.normal(m, 2) / np.sqrt(m)).astype(np.float32)
    return (I.random_k_body(rng, m, n, [1, 2, 3], 1), th, I.bernoulli_bits(rng, l, n, 0.1, 5), I.uniform_bits(rng, s, n, 6),
            rng.normal(l, 7), I.bernoulli_bits(rng, 130, n, 0.4, 8))


@pytest.mark.parametrize("n,m,l,s", CASES)
def test_kept_phase_gives_the_same_gradient(n, m, l, s):
    import torch
    from paper_2501_04776_gb300 import _lib, api
    G, th, A, Z, w, X = problem(n, m, l, s)
    assert _lib.load().iqp_planes_used(n, m, l, s) == 1
    G, A, Z, X = (api.to_device_bits(x) for x in (G, A, Z, X))
    w = torch.from_numpy(w).cuda()
    got = []
    for keep in (True, False):
        theta = torch.from_numpy(th).cuda().requires_grad_()
        ev, se = api.expval(theta, G, A, Z, n, "fp32", keep_phi=keep)
        (ev * w).sum().backward()
        got.append([x.detach().cpu().numpy() for x in (ev, se, theta.grad)])
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    theta = torch.from_numpy(th).cuda()
    loss, grad = api.mmd_loss_raw(n, theta, G, A, Z, X, "fp32", with_grad=True)
    want_loss, want = api.mmd_loss_raw(n, theta, G, A, Z, X, "sparse_fp32", with_grad=True)
    assert abs(float(loss) - float(want_loss)) <= 1e-4
    assert float((grad - want).norm()) <= 1e-4 * float(want.norm())
    assert api.read_status() == 0


def test_refusals():
    from paper_2501_04776_gb300 import _lib, api
    lib = _lib.load()
    n, m, l, s = 60, 300, 257, 257
    assert lib.iqp_planes_used(n, 36, 64, 1024) == 0 and lib.iqp_planes_used(n, 0, l, s) == 0
    G, th, A, Z, w, X = problem(n, m, l, s)
    import torch
    G, A, Z = (api.to_device_bits(x) for x in (G, A, Z))
    theta = torch.from_numpy(th).cuda()
    ev = torch.empty(l, dtype=torch.float64, device="cuda")
    phi = torch.empty((l, 320), dtype=torch.float32, device="cuda")
    need = lib.iqp_workspace_bytes(_lib.OP_EXPVAL, n, m, l, s, 0, _lib.FP32)
    ws = torch.zeros(need, dtype=torch.uint8, device="cuda")

    def call(ldphi=320, size=need, rows=s, p=phi.data_ptr()):
        return lib.iqp_planes_keep_phi(n, G.data_ptr(), m, G.shape[1], A.data_ptr(), l, A.shape[1], Z.data_ptr(), rows,
                                       Z.shape[1], theta.data_ptr(), ev.data_ptr(), ev.data_ptr(), p, ldphi, ws.data_ptr(),
                                       size, torch.cuda.current_stream().cuda_stream)

    assert call() == 0
    assert call(ldphi=256) == _lib.ERR_ARG and call(p=None) == _lib.ERR_ARG
    assert call(p=phi.data_ptr() + 4) == _lib.ERR_ALIGN
    assert call(size=need - 4096) == _lib.ERR_UNSUPPORTED  # the planes' regions end past it
    assert call(rows=3) == _lib.ERR_UNSUPPORTED            # too few terms: the SIMT kernels' range
    torch.cuda.synchronize()
