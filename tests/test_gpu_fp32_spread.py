"""FP32 with parameters of very different sizes and many gates: estimates,
standard errors and gradients against the FP64 oracle over observables that the
dominating parameters do not touch, beside the SIMT kernels (IQP_FP32_TC=0) on the
same inputs. 256 x 19456 fills a round of the chip with whole tiles, so that every gate of a
tile is summed in one go up to the chunk (8192 gates); the small sizes are split.

Tolerances: the library's own, 1e-5 absolute on estimates and standard errors and 1e-4
relative on the gradient, whatever the parameters; and the error is no larger
than the SIMT kernels', whose FP32 sums round at every term, plus two roundings of
a cosine or a sum (2^-23; the gradient: the planes' other test's 1e-6)."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2501_04776_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# n, m, l, s, kind: one parameter near pi / 2 and the rest of 0.003 ("one"), or
# every other one 500 times the rest ("half")
CASES = [(2000, 45_000, 256, 19_456, "one"), (2000, 65_536, 256, 19_456, "one"), (2000, 65_537, 256, 19_456, "half"),
         (2000, 8192, 24, 1100, "one"), (2000, 8193, 24, 1100, "half"), (60, 700, 8, 16_385, "one")]
ROWS = 24  # observables that the oracle takes (the first; the gradient weighs no others)


def problem(n, m, l, s, kind):
    """The dominating gates act on the last n / 2 qubits, the observables on the others."""
    rng = I.Rng(7 + m)
    h = n // 2
    G = np.zeros((m, I.words_per_row(n)), dtype=np.uint64)
    small = I.random_k_body(rng, m, h, [3], 1)
    G[:, :small.shape[1]] = small
    th = 0.003 * (2 * rng.uniform(m, 2) - 1)
    big = np.arange(m) % 2 == 1 if kind == "half" else np.arange(m) == m // 3
    G[big] = 0
    q = h + rng.integers(m, h, 3)
    G[big, q[big] // 64] = np.uint64(1) << (q[big] % 64).astype(np.uint64)
    th[big] = 0.499 * np.pi if kind == "one" else 500 * th[big]
    A = np.zeros((l, I.words_per_row(n)), dtype=np.uint64)
    bits = I.bernoulli_bits(rng, l, h, 0.5, 5)
    A[:, :bits.shape[1]] = bits
    al = rng.normal(l, 7) / s
    al[ROWS:] = 0
    return G, th.astype(np.float32), A, I.uniform_bits(rng, s, n, 6), al


def results(case):
    import torch
    from paper_2501_04776_gb300 import api
    n = case[0]
    G, th, A, Z, al = problem(*case)
    G, A, Z = (api.to_device_bits(x) for x in (G, A, Z))
    th, al = torch.from_numpy(th).cuda(), torch.from_numpy(al).cuda()
    one = api.expval_value_and_grad(n, th, G, A, Z, al, None, "fp32")
    two = (*api.expval_raw(n, th, G, A, Z, "fp32"), api.expval_grad(n, th, G, A, Z, al, None, "fp32"))
    assert api.read_status() == 0
    return [x.cpu().numpy() for x in (*one, *two)]


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.fixture(scope="module")
def simt(tmp_path_factory):
    """The SIMT kernels' results of every case, from one child process."""
    out = str(tmp_path_factory.mktemp("simt") / "r.npz")
    code = ("import sys, numpy as np; sys.path[:0] = [%r, %r]\n"
            "import test_gpu_fp32_spread as t\n"
            "np.savez(%r, **{'%%d_%%d' %% (i, k): x for i, c in enumerate(t.CASES) for k, x in enumerate(t.results(c))})"
            % (ROOT, os.path.dirname(os.path.abspath(__file__)), out))
    subprocess.run([sys.executable, "-c", code], check=True, timeout=300, env=dict(os.environ, IQP_FP32_TC="0"), cwd=ROOT)
    return np.load(out)


@pytest.mark.parametrize("k", range(len(CASES)), ids=["%s-m%d-s%d" % (c[4], c[1], c[3]) for c in CASES])
def test_spread_parameters_keep_fp32(simt, k):
    n, m, l, s, _ = CASES[k]
    G, th, A, Z, al = problem(*CASES[k])
    t64, A, al = th.astype(np.float64), A[:ROWS], al[:ROWS]
    ev, se, _, _ = oracle.expval(n, G, A, Z, t64)
    grad = oracle.expval_grad(n, G, A, Z, t64, al, None)

    def errors(e, d, g):
        return np.max(np.abs(e[:ROWS] - ev)), np.max(np.abs(d[:ROWS] - se)), rel(g, grad)

    got = results(CASES[k])
    plain = errors(*(simt["%d_%d" % (k, i)] for i in range(3)))
    for e in (errors(*got[:3]), errors(*got[3:])):
        assert e[0] <= min(1e-5, plain[0] + 2.0 ** -23), (e, plain)
        assert e[1] <= min(1e-5, plain[1] + 2.0 ** -23), (e, plain)
        assert e[2] <= min(1e-4, plain[2] + 1e-6), (e, plain)
