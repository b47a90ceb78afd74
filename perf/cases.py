"""Performance cases of the IQP estimator: what a program that uses this
library has it do, through the calls of `paper_2501_04776_gb300.api`.

The paths (`case["path"]`):
  expval     estimates and standard errors of a circuit, no gradient
  step       a training step on a loss linear in the estimates: autograd
             forward and backward
  vgrad      the same step in one call, for weights known beforehand
  mmd        the MMD^2 loss and its gradient on given samples
  train      the MMD^2 step of the training loop with its on-device draws of
             observables and samples
  bitflip    the stochastic bitflip model: exact values and their gradient
  indep      one sample batch per observable: estimates and gradient

Circuits, observables, samples and parameters follow the recipes of
`paper_2501_04776_gb300.inputs` (one- and two-body circuits, random k-body
generators, bits of observables Bernoulli, samples uniform, data from noisy
prototypes), drawn here with torch on the GPU from the case's seed.

theta is float32, as in training; the Monte-Carlo estimates, losses and
gradients carry FP32 accuracy by the library's own statement (1e-5 in its FP32
forms, 1e-4 in split BF16) and the program keeps them in theta's type. The
bitflip values are exact FP64 products and stay float64.
"""
import math

import numpy as np
import torch

from paper_2501_04776_gb300 import api

DEV = "cuda"


# ---------------------------------------------------------------- the cases

def _case(path, n, gates, m, l, s, p, scale, precision="split_bf16", N=0, dist="normal"):
    if gates == "local":  # all one- and two-body generators
        m = n * (n + 1) // 2
    return {"path": path, "precision": precision, "gates": gates, "n": int(n), "m": int(m), "l": int(l),
            "s": int(s), "N": int(N), "p": float(p), "theta": float(scale), "dist": dist}


def _p_sigma(n):
    """Bit probability of MMD observables for the bandwidth sigma = sqrt(n)/4."""
    return 0.5 * (1.0 - math.exp(-8.0 / n))


def listed():
    cases = []

    def add(name, c):
        cases.append(dict(c, name=name))

    # Exploring an 8-qubit circuit interactively: every call is launches and host time.
    add("expval-n8", _case("expval", 8, "local", 0, 64, 1024, 0.5, 0.3))
    # The same circuit trained in the plain FP32 form.
    add("step-n8-fp32", _case("step", 8, "local", 0, 64, 1024, 0.5, 0.3, "fp32"))
    # A mid-size circuit with odd sizes, default precision, one optimiser step per call.
    add("vgrad-n100-ragged", _case("vgrad", 100, "random3", 3001, 777, 2501, 0.05, 0.05, dist="uniform"))
    # The 300-qubit one- and two-body circuit of the paper's accuracy study: autograd step ...
    add("step-n300", _case("step", 300, "local", 0, 1000, 10000, 0.1, 0.01))
    # ... and the same step in FP32, where a user wants the FP32 tolerance.
    add("step-n300-fp32", _case("step", 300, "local", 0, 1000, 10000, 0.1, 0.01, "fp32"))
    # The paper's benchmark size: 10^4 observables x 10^4 samples x 10^5 gates.
    add("vgrad-n1000", _case("vgrad", 1000, "random3", 100_000, 10_000, 10_000, 0.05, 0.05, dist="uniform"))
    # Generative training on 1000 qubits, all one- and two-body gates: the loss step in its low-order form ...
    add("mmd-n1000-loworder", _case("mmd", 1000, "local", 0, 2000, 5000, _p_sigma(1000), 0.01, "loworder_fp32", 10_000))
    # ... and in the general row-sparse form, which takes generators of any weight.
    add("mmd-n1000-sparse", _case("mmd", 1000, "local", 0, 2000, 5000, _p_sigma(1000), 0.01, "sparse_fp32", 10_000))
    # A million gates on 5000 qubits.
    add("vgrad-n5000-loworder", _case("vgrad", 5000, "random2", 1_000_000, 4096, 16384, 0.01, 0.005, "loworder_fp32"))
    # A small generative model, trained with draws on the device.
    add("train-n200", _case("train", 200, "local", 0, 500, 2000, _p_sigma(200), 0.02, "loworder_fp32", 3000))
    # The classical counterpart of the benchmark circuit (stochastic bit flips), trained exactly.
    add("bitflip-n1000", _case("bitflip", 1000, "random3", 100_000, 10_000, 1, 0.05, 0.05, "fp64", dist="uniform"))
    # Uncorrelated estimates: each observable with its own samples.
    add("indep-n200", _case("indep", 200, "random3", 5000, 256, 2000, 0.05, 0.05, "sparse_fp32", dist="uniform"))
    return cases


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["expval", "step", "step", "vgrad", "vgrad", "mmd", "mmd", "train", "bitflip", "indep"])
    if path in ("expval", "step", "vgrad"):
        kind = rng.choice(["local", "local-fp32", "random3", "random2-loworder", "random2-sparse"])
        if kind.startswith("local"):
            n = _log(rng, 8, 300)
            l, s = _log(rng, 32, 1000), _log(rng, 500, 10_000)
            # |Phi| of order one at every width, as in training
            return _case(path, n, "local", 0, l, s, min(0.5, max(0.1, 4 / n)), 0.3 * 8 / max(n, 8),
                         "fp32" if kind == "local-fp32" else "split_bf16")
        if kind == "random3":
            return _case(path, _log(rng, 50, 5000), "random3", _log(rng, 300, 30_000), _log(rng, 50, 5000),
                         _log(rng, 500, 10_000), 0.05, 0.05, dist="uniform")
        n = _log(rng, 200, 5000)
        low = kind == "random2-loworder"
        return _case(path, n, "random2", _log(rng, 2000, 500_000 if low else 200_000), _log(rng, 50, 4000 if low else 1000),
                     _log(rng, 500, 16_000 if low else 8000), 0.01, 0.005, "loworder_fp32" if low else "sparse_fp32")
    if path == "mmd":
        n = _log(rng, 30, 1000)
        return _case("mmd", n, "local", 0, _log(rng, 100, 2000), _log(rng, 500, 5000), _p_sigma(n), 0.3 / math.sqrt(n),
                     rng.choice(["loworder_fp32", "loworder_fp32", "sparse_fp32", "split_bf16"]), _log(rng, 500, 10_000))
    if path == "train":
        n = _log(rng, 20, 1000)
        return _case("train", n, "local", 0, _log(rng, 100, 2000), _log(rng, 500, 5000), _p_sigma(n),
                     0.3 / math.sqrt(n), "loworder_fp32", _log(rng, 500, 10_000))
    if path == "bitflip":
        return _case("bitflip", _log(rng, 50, 2000), "random3", _log(rng, 500, 100_000), _log(rng, 50, 10_000), 1, 0.05,
                     0.05, "fp64", dist="uniform")
    return _case("indep", _log(rng, 20, 1000), "random3", _log(rng, 300, 10_000), _log(rng, 20, 400),
                 _log(rng, 200, 4000), 0.05, 0.05, "sparse_fp32", dist="uniform")


# ------------------------------------------------------------------ inputs

def _words(n):
    w = (n + 63) // 64
    return w + (w & 1)


def _bit(q):
    return torch.bitwise_left_shift(torch.ones_like(q), q & 63)


def _pack(bits):
    """(rows, n) bool -> (rows, words) int64, least significant bit first."""
    rows, n = bits.shape
    out = torch.zeros(rows, _words(n) * 64, dtype=torch.bool, device=bits.device)
    out[:, :n] = bits
    weight = _bit(torch.arange(64, device=bits.device))
    return (out.view(rows, -1, 64) * weight).sum(-1)


def _random_bits(gen, rows, n, p):
    """Packed rows of Bernoulli(p) bits."""
    step = max(1, 2**26 // n)
    return torch.cat([_pack(torch.rand(min(step, rows - r), n, device=DEV, generator=gen) < p)
                      for r in range(0, rows, step)])


def _from_qubits(qubits, n):
    """Packed generators from lists of (rows, qubits), each pair once."""
    m = max(int(r.max()) for r, _ in qubits) + 1
    G = torch.zeros(m * _words(n), dtype=torch.int64, device=DEV)
    for r, q in qubits:
        G.scatter_add_(0, r * _words(n) + (q >> 6), _bit(q))
    return G.view(m, _words(n))


def _generators(gen, case):
    n, m = case["n"], case["m"]
    if case["gates"] == "local":
        a, b = torch.triu_indices(n, n, 1, device=DEV)
        one, two = torch.arange(n, device=DEV), n + torch.arange(a.numel(), device=DEV)
        return _from_qubits([(one, one)] + ([(two, a), (two, b)] if n > 1 else []), n)
    most = {"random2": 2, "random3": 3}[case["gates"]]

    def below(k):
        return torch.randint(0, k, (m,), device=DEV, generator=gen)

    k, rows = 1 + below(most), torch.arange(m, device=DEV)
    q0, q1, q2 = below(n), below(n - 1), below(n - 2)
    q1 = q1 + (q1 >= q0)
    lo, hi = torch.minimum(q0, q1), torch.maximum(q0, q1)
    q2 = q2 + (q2 >= lo)
    q2 = q2 + (q2 >= hi)
    return _from_qubits([(rows, q0), (rows[k >= 2], q1[k >= 2])] + ([(rows[k >= 3], q2[k >= 3])] if most == 3 else []), n)


def _inputs(case, seed):
    gen = torch.Generator(DEV).manual_seed(seed)
    n, m, l, s, path = case["n"], case["m"], case["l"], case["s"], case["path"]
    i = {"G": _generators(gen, case), "seed": seed}
    if case["dist"] == "uniform":
        i["theta"] = case["theta"] * (2 * torch.rand(m, device=DEV, generator=gen) - 1)
    else:
        i["theta"] = case["theta"] * torch.randn(m, device=DEV, generator=gen)
    if path != "train":
        i["A"] = _random_bits(gen, l, n, case["p"])
    if path not in ("train", "bitflip"):
        i["Z"] = _random_bits(gen, l * s if path == "indep" else s, n, 0.5)
    if case["N"]:
        proto = _random_bits(gen, 8, n, 0.5)
        i["X"] = proto[torch.randint(0, 8, (case["N"],), device=DEV, generator=gen)] ^ _random_bits(gen, case["N"], n, 0.05)
    else:
        i["w"] = torch.randn(l, device=DEV, generator=gen)  # the loss is sum_a w_a <Z_a>
    return i


def prepare(case, seed):
    state = dict(_inputs(case, seed), case=case)
    if case["path"] != "expval" and case["path"] != "vgrad":
        state["theta"].requires_grad_(True)
    if case["path"] == "vgrad":  # gradient coefficients of the linear loss
        state["alpha"] = -state["w"].double() / case["s"]
    return state


# --------------------------------------------------------------------- run

def run(state):
    c, G, theta = state["case"], state["G"], state["theta"]
    path, n, precision = c["path"], c["n"], c["precision"]
    if path == "expval":
        ev, se = api.expval(theta, G, state["A"], state["Z"], n, precision)
        return [ev.to(theta.dtype), se.to(theta.dtype)]
    if path == "vgrad":
        ev, se, grad = api.expval_value_and_grad(n, theta, G, state["A"], state["Z"], state["alpha"], None, precision)
        return [ev.to(theta.dtype), se.to(theta.dtype), grad.to(theta.dtype)]
    if path in ("step", "indep"):
        if path == "step":
            ev, se = api.expval(theta, G, state["A"], state["Z"], n, precision)
        else:
            ev, se = api.expval_indep(theta, G, state["A"], state["Z"], n)
        ev = ev.to(theta.dtype)
        (grad,) = torch.autograd.grad(torch.dot(state["w"], ev), theta)
        return [ev.detach(), se.to(theta.dtype), grad]
    if path == "bitflip":
        ev = api.bitflip_expval(theta, G, state["A"], n)
        (grad,) = torch.autograd.grad(torch.dot(state["w"].double(), ev), theta)
        return [ev.detach(), grad]
    if path == "train":
        A = api.bernoulli_bits(state["seed"], 1001, c["l"], n, c["p"])
        Z = api.uniform_bits(state["seed"], 1000, c["s"], n)
    else:
        A, Z = state["A"], state["Z"]
    loss = api.mmd_loss(theta, G, A, Z, state["X"], n, precision)
    (grad,) = torch.autograd.grad(loss, theta)
    out = [loss.detach().to(theta.dtype), grad]
    return out + [A, Z] if path == "train" else out


# -------------------------------------------------------------------- work

def _pairs(case):
    """Qubit pairs that carry a two-body generator (expected)."""
    n = case["n"]
    total = n * (n - 1) / 2
    if case["gates"] == "local":
        return total
    return total * -math.expm1(-(case["m"] / 2) / total)


def _odd(case):
    """Share of the (observable, generator) pairs of odd overlap (expected)."""
    e = 1 - 2 * case["p"]
    n, m = case["n"], case["m"]
    if case["gates"] == "local":
        return (n * (1 - e) / 2 + (m - n) * (1 - e * e) / 2) / m
    k = 3 if case["gates"] == "random3" else 2
    return sum((1 - e**j) / 2 for j in range(1, k + 1)) / k


def work(case):
    """Inputs read once and outputs written once; the multiply-adds of the
    phases (and of the gradient) in the form that the case asks for."""
    n, m, l, s, path = case["n"], case["m"], case["l"], case["s"], case["path"]
    row = _words(n) * 8
    grad = path != "expval"
    data = m * row + 4 * m + l * row + case["N"] * row + 8 * l + (4 * m if grad else 0)
    if path != "bitflip":
        data += (l * s if path == "indep" else s) * row
    if path == "bitflip":
        flops = 2.0 * _odd(case) * l * m  # a product for the value, a sum for the gradient
    elif case["precision"] == "loworder_fp32":
        weight = n * case["p"]  # per observable: its qubits, and the pairs among them that carry a gate
        share = _pairs(case) / max(1.0, n * (n - 1) / 2)
        per = 2.0 * _pairs(case) * s * 2 + 2.0 * l * s * (weight + share * weight * weight / 2)
        flops = per * (2 if grad else 1)
    elif case["precision"] == "sparse_fp32":
        flops = 2.0 * _odd(case) * l * m * s * (2 if grad else 1)
    else:
        flops = 2.0 * l * m * s * (2 if grad else 1)
    if case["N"]:  # data parities: an AND and an XOR per 32-bit word
        flops += 2.0 * l * case["N"] * ((n + 31) // 32)
    return {"bytes": float(data), "flops": flops}


# ------------------------------------------------------------------- exact

def _unpack(words, n, dtype=torch.float64):
    """(rows, words) -> (rows, n) of 0 and 1."""
    bits = torch.bitwise_right_shift(words.unsqueeze(-1), torch.arange(64, device=words.device)) & 1
    return bits.view(words.shape[0], -1)[:, :n].to(dtype)


def _signs(G, R, n):
    """(-1)^(g_j . r) as float64, rows of R by rows of G."""
    return 1.0 - 2.0 * torch.remainder(_unpack(R, n, torch.float32) @ _unpack(G, n, torch.float32).T, 2.0).double()


def _statistics(phi):
    c = torch.cos(phi)
    mean = c.mean(1)
    return c, mean, torch.sqrt((c * c).mean(1).sub(mean * mean).clamp_min(0) / phi.shape[1])


def _mmd_parts(i, case, c):
    """MMD^2 (unbiased) and W = sin Phi (alpha + beta cos Phi) without its sine, from the cosines."""
    l, s, N, n = case["l"], case["s"], case["N"], case["n"]
    T = torch.cat([(1.0 - 2.0 * torch.remainder(_unpack(a, n, torch.float32) @ _unpack(i["X"], n, torch.float32).T, 2.0))
                   .double().sum(1) for a in i["A"].split(512)])
    S1, S2 = c.sum(1), (c * c).sum(1)
    p, q = T / N, S1 / s
    loss = ((T * T - N) / (N * (N - 1.0)) - 2 * p * q + (S1 * S1 - S2) / (s * (s - 1.0))).mean()
    alpha = (2 * p / s - 2 * S1 / (s * (s - 1.0))) / l
    return loss, alpha, torch.full_like(alpha, 2.0 / (s * (s - 1.0)) / l)


def _exact_dense(i, case):
    """Phi = (2 theta . P_A) S_Z^T over all gates, block by block."""
    n, m = case["n"], case["m"]
    th = i["theta"].double()
    blocks = [slice(j, min(m, j + 20_000)) for j in range(0, m, 20_000)]

    def operands(b):
        P = (1.0 - _signs(i["G"][b], i["A"], n)) / 2
        return P, _signs(i["G"][b], i["Z"], n)

    phi = torch.zeros(i["A"].shape[0], i["Z"].shape[0], dtype=torch.float64, device=DEV)
    for b in blocks:
        P, S = operands(b)
        phi += (P * (2 * th[b])) @ S.T

    def gradient(W):
        out = []
        for b in blocks:
            P, S = operands(b)
            out.append(2 * (P * (W @ S)).sum(0))
        return torch.cat(out)
    return phi, gradient


def _exact_pairs(i, case):
    """The same for generators on one or two qubits, through the pair matrix."""
    n, m = case["n"], case["m"]
    first, last = [], []
    for g in i["G"].split(max(1, 2**28 // n)):
        bits = _unpack(g, n, torch.uint8)
        first.append(torch.argmax(bits, 1))
        last.append(n - 1 - torch.argmax(bits.flip(1), 1))
    first, last = torch.cat(first), torch.cat(last)
    th = 2 * i["theta"].double()
    single = first == last
    d = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, first[single], th[single])
    C = torch.zeros(n * n, dtype=torch.float64, device=DEV).index_add_(0, (first * n + last)[~single], th[~single]).view(n, n)
    C = C + C.T
    S = (1.0 - 2.0 * _unpack(i["Z"], n)).T.contiguous()  # n x s
    base = d[:, None] + C @ S
    supports = [torch.nonzero(a).view(-1) for a in _unpack(i["A"], n, torch.bool)]
    phi = torch.zeros(len(supports), S.shape[1], dtype=torch.float64, device=DEV)
    for a, Q in enumerate(supports):
        SQ = S[Q]
        phi[a] = (SQ * (base[Q] - C[Q][:, Q] @ SQ)).sum(0)

    def gradient(W):
        V, K = torch.zeros_like(S), torch.zeros(n, n, dtype=torch.float64, device=DEV)
        for a, Q in enumerate(supports):
            SQ = S[Q]
            V[Q] += W[a]
            K[Q[:, None], Q[None, :]] += (SQ * W[a]) @ SQ.T
        U = S * V
        H = U @ S.T
        one = 2 * U.sum(1)
        two = 2 * (H + H.T) - 4 * K
        return torch.where(single, one[first], two[first, last])
    return phi, gradient


def _exact_indep(i, case):
    n, l, s = case["n"], case["l"], case["s"]
    th = i["theta"].double()
    P = (1.0 - _signs(i["G"], i["A"], n)) / 2
    phi = torch.stack([_signs(i["G"], i["Z"][a * s:(a + 1) * s], n) @ (2 * th * P[a]) for a in range(l)])

    def gradient(W):
        out = torch.zeros_like(th)
        for a in range(l):
            out += 2 * P[a] * (W[a] @ _signs(i["G"], i["Z"][a * s:(a + 1) * s], n))
        return out
    return phi, gradient


def _exact_bitflip(i, case):
    n, th, w = case["n"], i["theta"].double(), i["w"].double()
    c, t = torch.cos(2 * th), -2 * torch.tan(2 * th)
    ev, total = [], torch.zeros_like(th)
    for r in range(0, case["l"], 256):
        P = _signs(i["G"], i["A"][r:r + 256], n) < 0
        e = torch.where(P, c, torch.ones_like(c)).prod(1)
        ev.append(e)
        total += (w[r:r + 256] * e) @ P.double()
    return [torch.cat(ev), t * total]


def exact(case, seed):
    path, two_body = case["path"], case["gates"] in ("local", "random2")
    if path == "bitflip":
        return _exact_bitflip(_inputs(case, seed), case)
    # pairs: cheap at every size; otherwise two dense FP64 products of 2 l m s each
    if not two_body and 4.0 * case["l"] * case["m"] * case["s"] > 6e12:
        return None
    i = _inputs(case, seed)
    if path == "train":
        i["A"] = _bernoulli_draw(seed, 1001, case["l"], case["n"], case["p"])
        i["Z"] = _uniform_draw(seed, 1000, case["s"], case["n"])
    phi, gradient = (_exact_indep if path == "indep" else _exact_pairs if two_body else _exact_dense)(i, case)
    c, mean, err = _statistics(phi)
    if path == "expval":
        return [mean, err]
    if case["N"]:
        loss, alpha, beta = _mmd_parts(i, case, c)
        out = [loss, gradient(torch.sin(phi) * (alpha[:, None] + beta[:, None] * c))]
        return out + [None, None] if path == "train" else out
    alpha = -i["w"].double() / case["s"]
    return [mean, err, gradient(torch.sin(phi) * alpha[:, None])]


# The counter-based random bits of the training loop (splitmix64), in numpy.

def _splitmix(seed, stream, count):
    with np.errstate(over="ignore"):
        z = (np.uint64(seed) * np.uint64(0xD1B54A32D192ED03) + np.uint64(stream) * np.uint64(0xAEF17502108EF2D9)
             + np.arange(1, count + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15))
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _uniform_draw(seed, stream, rows, n):
    words = _splitmix(seed, stream, rows * _words(n)).reshape(rows, _words(n))
    keep = np.zeros(_words(n), dtype=np.uint64)
    keep[:n // 64] = np.uint64(2**64 - 1)
    if n % 64:
        keep[n // 64] = np.uint64(2**(n % 64) - 1)
    return torch.from_numpy((words & keep).view(np.int64)).to(DEV)


def _bernoulli_draw(seed, stream, rows, n, p):
    u = (_splitmix(seed, stream, rows * n) >> np.uint64(11)).astype(np.float64) * 2.0**-53
    return _pack(torch.from_numpy((u < p).reshape(rows, n)).to(DEV))
