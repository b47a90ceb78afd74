"""The bitflip gradient gate by gate against its formula in FP64, where the integer
sums take it (from 2^25 parity bits on): gates whose observables' values are many
decades below the others', weights of one sign so that no sum cancels, weights
whose squares leave the range of doubles, gates that no observable meets, and values of
one size.

Tolerance, per gate: a value is a product of at most 9000 factors, each within
2^-52, here, and the exponential of a sum of logarithms there; the terms are positive, and their sum
is within 2^-52 times its length, at most 16400: 25400 2^-52 = 6e-12 relative."""
import numpy as np
import pytest

from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -900, 2.0 ** 900])
@pytest.mark.parametrize("m,l,decay", [(8200, 4100, 30.0), (8200, 4100, 0.0), (16_400, 2049, 12.0), (2049, 16_400, 30.0)])
def test_every_gate_keeps_its_digits(m, l, decay, scale):
    import torch
    from paper_2501_04776_gb300 import api
    n, h = 80, 40
    rng = I.Rng(m + l)
    G, A = I.random_k_body(rng, m, h, [1, 2, 3], 1), I.bernoulli_bits(rng, l, h, 0.1, 2)
    # the second half of the gates and of the observables: on qubits 40 .. 79, values about e^-decay
    mh, lh = m // 2, l // 2
    A[lh:] = I.bernoulli_bits(rng, l - lh, h, 0.5, 6)  # half of its gates each
    for M, r in ((G, mh), (A, lh)):
        M[r:, 1] = M[r:, 0] >> np.uint64(64 - h)
        M[r:, 0] <<= np.uint64(h)
    P = (I.unpack_bits(A, n).astype(np.float32) @ I.unpack_bits(G, n).astype(np.float32).T) % 2  # l x m
    P[:, 7] = G[7] = 0  # no observable meets gate 7
    odd = P[lh:].sum(1).mean()
    th = 0.02 * (2 * rng.uniform(m, 3) - 1)
    if decay:  # 2 theta^2 per odd gate
        th[mh:] = np.sqrt(decay / (2 * odd)) * (1 + 0.1 * rng.uniform(m - mh, 4))
    th[5] = 0.0
    th = th.astype(np.float32)
    w = scale * (0.5 + rng.uniform(l, 5))
    g = api.bitflip_grad(n, torch.from_numpy(th).cuda(), api.to_device_bits(G), api.to_device_bits(A),
                         torch.from_numpy(w).cuda()).cpu().numpy()
    x, P = 2 * th.astype(np.float64), P.astype(np.float64)
    ev = np.exp(P @ np.log(np.cos(x)))
    want = -2 * np.tan(x) * ((w / scale * ev) @ P) * scale
    assert g[5] == 0 and g[7] == 0
    live = want != 0
    assert live.sum() > 0.9 * m and not g[~live].any()
    assert np.max(np.abs(g[live] / want[live] - 1)) <= 6e-12
