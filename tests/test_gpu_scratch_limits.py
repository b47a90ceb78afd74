"""Calls on a device that has no room for the full workspace: they run with the
smallest one, as they did before the optional regions, and give the same
results to the forms' tolerances (1e-5 on estimates and the loss, 1e-4 relative on gradients,
1e-12 on bitflip values). The allocator is replaced by one that refuses; no memory is exhausted."""
import pytest

pytestmark = pytest.mark.gpu

FORMS = ["fp32", "split_bf16", "sparse_fp32", "loworder_fp32"]


@pytest.fixture
def tight(monkeypatch):
    """allow(op, ...): a fresh workspace pool that refuses more than the smallest workspaces of the operations named."""
    import torch
    from paper_2501_04776_gb300 import _lib, api
    pool = api._Workspace()
    most, refused = [0], []
    get = pool.get

    def limited(nbytes, device, stream=None):
        if nbytes > most[0]:
            refused.append(nbytes)
            raise torch.OutOfMemoryError("refused")
        return get(nbytes, device, stream)

    monkeypatch.setattr(pool, "get", limited)

    def allow(*ops):
        pool._bufs.clear()
        pool.refused.clear()
        refused.clear()
        most[0] = max(_lib.load().iqp_workspace_min_bytes(*op) for op in ops)
        monkeypatch.setattr(api, "_WS", pool)
        return refused

    return allow


def problem(n=40, l=300, s=1500):
    import torch
    from paper_2501_04776_gb300 import api
    from paper_2501_04776_gb300 import inputs as I
    rng = I.Rng(11)
    G = I.local_gates_packed(n)
    th = torch.from_numpy(rng.normal(G.shape[0], 2)).float().cuda() * 0.02
    return n, th, [api.to_device_bits(x) for x in (G, I.bernoulli_bits(rng, l, n, 0.1, 3), I.uniform_bits(rng, s, n, 4),
                                                   I.uniform_bits(rng, 400, n, 5))], torch.from_numpy(rng.normal(l, 6)).cuda()


def near(a, b, tol):
    return float((a - b).norm()) <= tol * float(b.norm())


@pytest.mark.parametrize("form", FORMS)
def test_estimates_and_loss(tight, form):
    import torch
    from paper_2501_04776_gb300 import _lib, api
    n, th, (G, A, Z, X), w = problem()
    m, l, s, N = G.shape[0], A.shape[0], Z.shape[0], X.shape[0]

    def run():
        t = th.clone().requires_grad_(True)
        ev, se = api.expval(t, G, A, Z, n, form)
        (g,) = torch.autograd.grad((w * ev).sum(), t)
        loss = api.mmd_loss(t, G, A, Z, X, n, form)
        (h,) = torch.autograd.grad(loss, t)
        one = api.expval_value_and_grad(n, th, G, A, Z, -w / s, None, form)
        return ev.detach(), se, g, loss.detach(), h, one[0], one[2]

    a = run()
    code = api.precision_code(form)
    refused = tight(*((op, n, m, l, s, N, code) for op in (_lib.OP_EXPVAL, _lib.OP_EXPVAL_GRAD, _lib.OP_MMD_LOSS,
                                                           _lib.OP_MMD_LOSS_GRAD)))
    b = run()
    assert refused and api.read_status() == 0
    for x, y, grad in zip(b, a, (0, 0, 1, 0, 1, 0, 1)):
        assert near(x, y, 1e-4) if grad else float((x - y).abs().max()) <= (1e-4 if form == "split_bf16" else 1e-5)


def test_bitflip_and_independent_batches(tight):
    import torch
    from paper_2501_04776_gb300 import _lib, api
    n, th, (G, A, Z, _), w = problem(200, 2000, 500)  # 20100 gates x 2000: the integer sums' sizes
    m, l, s = G.shape[0], A.shape[0], 1100
    Zi = api.uniform_bits(3, 4, 30 * s, n)

    def run():
        t = th.clone().requires_grad_(True)
        ev = api.bitflip_expval(t, G, A, n)
        (g,) = torch.autograd.grad((w * ev).sum(), t)
        iv, _ = api.expval_indep(t[:900], G[:900], A[:30], Zi, n)
        (h,) = torch.autograd.grad((w[:30] * iv).sum(), t)
        return ev.detach(), g, iv.detach(), h

    a = run()
    refused = tight((_lib.OP_BITFLIP, n, m, l, 1, 0, _lib.FP32), (_lib.OP_EXPVAL_INDEP_GRAD, n, 900, 30, s, 0, 0))
    b = run()
    assert refused
    assert float((a[0] - b[0]).abs().max()) <= 1e-12 and near(b[1], a[1], 1e-6)  # the gradient comes back in FP32
    assert float((a[2] - b[2]).abs().max()) <= 1e-5 and near(b[3], a[3], 1e-4)


def test_a_refused_size_is_not_asked_for_again(tight):
    from paper_2501_04776_gb300 import _lib, api
    n, th, (G, A, Z, _), _ = problem()
    refused = tight((_lib.OP_EXPVAL, n, G.shape[0], A.shape[0], Z.shape[0], 0, _lib.FP32))
    for _ in range(3):
        api.expval_raw(n, th, G, A, Z, "fp32")
        ev, _ = api.expval(th.clone().requires_grad_(True), G, A, Z, n, "fp32")  # would keep Phi, with the planes
    assert len(refused) == 1
