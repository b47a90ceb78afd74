"""FP32 gradient of more W than the planes hold at a time (2 GiB): the scratch is
bounded, and the gradient is that of its observables in two calls of one block each,
from the same Phi. Both sum the same partial rows (whole tiles of 128 observables) in FP64,
157 tiles of two rows, in another order: 314 2^-53 of the sum of magnitudes, here 1e-12 of the largest
entry times the square root of the observables' number."""
import pytest


def test_planes_are_bounded():
    """FP32 takes 2 GiB and its partials (a double2 per 64 samples) beside what split BF16 takes, whose W has the same size."""
    from paper_2501_04776_gb300 import _lib, build
    build.build()
    lib, (n, m, l, s) = _lib.load(), (300, 45_150, 100_000, 100_000)
    by = [lib.iqp_workspace_bytes(_lib.OP_EXPVAL_GRAD, n, m, l, s, 0, p) for p in (_lib.FP32, _lib.SPLIT_BF16)]
    assert by[0] - by[1] <= 2 ** 31 + l * (s // 64 + 1) * 16 + 2 ** 26


@pytest.mark.gpu
def test_blocks_of_observables():
    import torch
    from paper_2501_04776_gb300 import _lib, api
    from paper_2501_04776_gb300 import inputs as I
    n, m, l, s, half = 60, 700, 20_001, 20_000, 78 * 128
    rng = I.Rng(5)
    G = api.to_device_bits(I.random_k_body(rng, m, n, [1, 2, 3], 1))
    A, Z = api.to_device_bits(I.bernoulli_bits(rng, l, n, 0.1, 3)), api.to_device_bits(I.uniform_bits(rng, s, n, 4))
    th = torch.from_numpy(rng.normal(m, 2)).float().cuda() * 0.02
    al = torch.from_numpy(rng.normal(l, 5)).cuda() / s
    assert 6 * l * s > 2 ** 31 and 6 * (l - half) * s < 2 ** 31
    _, _, phi = api._planes_keep_phi(n, th, G, A, Z)
    whole = api._planes_grad_from_phi(n, th, G, A, Z, phi, al)
    parts = sum(api._planes_grad_from_phi(n, th, G, A[a:b], Z, phi[a:b], al[a:b]) for a, b in ((0, half), (half, l)))
    assert api.read_status() == 0
    assert float((whole - parts).abs().max()) <= 1e-12 * l ** 0.5 * float(whole.abs().max())
    again = api.expval_grad(n, th, G, A, Z, al, None, "fp32")  # Phi recomputed
    assert float((again - whole).norm()) <= 1e-5 * float(whole.norm())
    api._WS._bufs.clear()
    del phi
    torch.cuda.empty_cache()
