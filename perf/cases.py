"""What a user of the library has it compute, as measurable cases.

Each case is one call of a public entry point on inputs of the sizes the
paper and this repository's configurations use: exact enumeration (Algorithm
1) from a few qubits up to N = 18, many small states in one batch, the two
Monte Carlo estimators up to N = 30, the exact x-marginal, the gate kernels
that prepare and precondition states, and the mixed-state entropy.

States are "haar" (i.i.d. complex Gaussian amplitudes, the paper's main Monte
Carlo input) or "doped": T-doped Clifford states in phase-polynomial form, an
H layer, random CZ and S gates, n_t T gates on random parities and H on a
random half of the qubits. A doped state with few T gates has the non-trivial
stabilizer group that the nullity recount works on.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2601_00761_gb300 as sre

EXACT_OUT = ("M", "S", "parseval", "r2", "stab_count", "nullity")
MC_OUT = ("M", "S", "err_M", "M_rb", "err_rb")


def listed():
    return [
        # The smallest exact sweep of the paper's figures: one T-doped state, latency and launches count.
        {"name": "exact_n10", "kind": "exact", "N": 10, "state": "doped", "n_t": 20, "precision": "fp32"},
        # Nullity of a weakly doped state: the largest N of one tile per family, many families recounted in FP64.
        {"name": "nullity_n15", "kind": "nullity", "N": 15, "state": "doped", "n_t": 4},
        # Exact enumeration of a T-doped state at the size of the exact-enumeration workload (two passes).
        {"name": "exact_n18", "kind": "exact", "N": 18, "state": "doped", "n_t": 32, "precision": "fp32"},
        # The split-BF16 tensor-core option at the paper's largest exact size.
        {"name": "exact_n16_bf16x3", "kind": "exact", "N": 16, "state": "haar", "n_t": 0, "precision": "bf16x3"},
        # An ensemble average over T-doped circuits: many states of uneven N in one call.
        {"name": "batched_n8_16", "kind": "batched", "N": 8, "N_max": 16, "count": 128, "state": "doped", "n_t": 12},
        # The headline: N = 24 Haar state, 4096 families from the exact marginal, 256 strings drawn from each.
        {"name": "mc_marginal_n24", "kind": "mc_marginal", "N": 24, "n_x": 4096, "z_per_x": 256, "state": "haar", "n_t": 0},
        # The paper's own estimator past the exact range: uniform x on a doped state, an odd N and a ragged count.
        {"name": "mc_uniform_n21", "kind": "mc_uniform", "N": 21, "n_x": 5001, "z_per_x": 1, "state": "doped", "n_t": 40},
        # The largest state: 8 GB, three passes per family.
        {"name": "mc_marginal_n30", "kind": "mc_marginal", "N": 30, "n_x": 128, "z_per_x": 64, "state": "haar", "n_t": 0},
        # The exact x-marginal as a result of its own.
        {"name": "marginal_n27", "kind": "marginal", "N": 27, "state": "haar", "n_t": 0},
        # Clifford preconditioning by a random {H, S, CNOT} list with T gates among them.
        {"name": "circuit_n26", "kind": "circuit", "N": 26, "gates": 1000, "state": "haar", "n_t": 0},
        # Brick-wall preconditioning: depth 2N of general two-qubit gates.
        {"name": "brickwall_n24", "kind": "brickwall", "N": 24, "layers": 48, "state": "haar", "n_t": 0},
        # Entropy of half of the qubits of a pure state.
        {"name": "mixed_n24", "kind": "mixed", "N": 24, "N_A": 12, "state": "haar", "n_t": 0},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["exact", "exact", "nullity", "batched", "mc_marginal", "mc_marginal", "mc_uniform", "marginal",
                       "circuit", "brickwall", "mixed"])
    state = rng.choice(["haar", "doped"])
    if kind == "exact":
        prec = rng.choice(["fp32", "fp32", "bf16x3"])
        N = rng.randint(6, 18 if prec == "fp32" else 16)
        return {"kind": kind, "N": N, "state": state, "n_t": rng.randint(N, 3 * N), "precision": prec}
    if kind == "nullity":
        N = rng.randint(6, 16)
        return {"kind": kind, "N": N, "state": "doped", "n_t": rng.randint(1, N - 4)}
    if kind == "batched":
        lo = rng.randint(6, 12)
        return {"kind": kind, "N": lo, "N_max": rng.randint(lo, 16), "count": log_int(3, 128), "state": "doped",
                "n_t": rng.randint(1, 24)}
    if kind in ("mc_marginal", "mc_uniform"):
        N = rng.randint(12, 30)
        n_x = log_int(16, min(20000, 1 << (36 - N))) if N <= 29 else rng.randint(16, 128)
        z = log_int(8, 512) if kind == "mc_marginal" else 1
        return {"kind": kind, "N": N, "n_x": n_x, "z_per_x": z, "state": state if N <= 22 else "haar", "n_t": rng.randint(N, 2 * N)}
    if kind == "marginal":
        return {"kind": kind, "N": rng.randint(10, 28), "state": "haar", "n_t": 0}
    if kind == "circuit":
        return {"kind": kind, "N": rng.randint(8, 26), "gates": log_int(20, 1000), "state": "haar", "n_t": 0}
    if kind == "brickwall":
        N = rng.randint(6, 25)
        return {"kind": kind, "N": N, "layers": rng.randint(2, 2 * N), "state": "haar", "n_t": 0}
    N = rng.randint(14, 26)
    return {"kind": kind, "N": N, "N_A": rng.randint(5, min(12, N // 2)), "state": "haar", "n_t": 0}


# ------------------------------------------------------------------ inputs
def _state(kind, N, n_t, seed):
    """complex64 state on the GPU, from the seed alone."""
    d = 1 << N
    if kind == "haar":
        g = torch.Generator(device="cuda").manual_seed(seed)
        psi = torch.view_as_complex(torch.randn(d, 2, generator=g, device="cuda", dtype=torch.float32))
        return psi.mul_(1.0 / math.sqrt(2.0 * d))
    r = np.random.Generator(np.random.PCG64(seed))
    b = torch.arange(d, device="cuda", dtype=torch.int32)
    octant = torch.zeros(d, device="cuda", dtype=torch.int32)     # phase in units of pi / 4
    def masks(rows):
        return [int(v) for v in (rows * (1 << np.arange(N))).sum(1)]
    cz = np.triu(r.integers(0, 2, (N, N)), 1)
    for i, m in enumerate(masks(cz)):
        if m:
            octant += 4 * (((b >> i) & 1) * _parity(b & m))
    for i in np.nonzero(r.integers(0, 2, N))[0]:
        octant += 2 * ((b >> int(i)) & 1)
    for m in masks(r.integers(0, 2, (n_t, N))):
        octant += _parity(b & m)
    psi = torch.polar(torch.full((d,), d ** -0.5, device="cuda", dtype=torch.float64),
                      (octant & 7).double() * (math.pi / 4))
    for q in np.nonzero(r.integers(0, 2, N))[0]:
        psi = _h(psi, int(q))
    return psi.to(torch.complex64)


def _parity(v):
    for s in (16, 8, 4, 2, 1):
        v = v ^ (v >> s)
    return v & 1


def _h(psi, q):
    v = psi.view(-1, 2, 1 << q)
    a, b = v[:, 0], v[:, 1]
    return (torch.stack([a + b, a - b], 1) * math.sqrt(0.5)).reshape(-1)


def _sizes(case):
    """The Ns of a batch: every size of the range in turn."""
    span = case["N_max"] - case["N"] + 1
    return [case["N"] + (7 * i + i // span) % span for i in range(case["count"])]


def _gates(case, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    n, N = case["gates"], case["N"]
    op = r.choice(np.array([0, 1, 3]), n)                           # H, S, CNOT
    op[15::16] = 4                                                 # a T after every 15 Cliffords
    q0 = r.integers(0, N, n)
    q1 = (q0 + r.integers(1, N, n)) % N
    return np.stack([op, q0, np.where(op == 3, q1, 0)], 1).astype(np.uint8)


def _brickwall(case, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    N = case["N"]
    pairs = np.array([(q, q + 1) for layer in range(case["layers"]) for q in range(layer % 2, N - 1, 2)], np.int32)
    a = r.standard_normal((len(pairs), 4, 4)) + 1j * r.standard_normal((len(pairs), 4, 4))
    u, t = np.linalg.qr(a)
    diag = np.einsum("kii->ki", t)
    return (u * (diag / np.abs(diag))[:, None, :]).astype(np.complex64), pairs


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": seed}
    if kind == "batched":
        st["psis"] = [_state(case["state"], N, 1 + (case["n_t"] * (i + 1)) % (2 * N), seed * 1009 + i)
                      for i, N in enumerate(_sizes(case))]
        return st
    # an ensemble for the nullity has circuits of more and of fewer T gates
    n_t = case["n_t"] + seed % 4 if kind == "nullity" else case["n_t"]
    st["psi"] = _state(case["state"], case["N"], n_t, seed)
    if kind == "circuit":
        st["gates"] = _gates(case, seed)
    if kind == "brickwall":
        st["mats"], st["pairs"] = _brickwall(case, seed)
    if kind in ("circuit", "brickwall"):
        st["out"] = torch.empty_like(st["psi"])
    return st


# --------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "exact":
        prec = sre.SRE_BF16X3_TC if case["precision"] == "bf16x3" else sre.SRE_FP32_SIMT
        r = sre.sre_exact(state["psi"], precision=prec)
        return {k: r[k] for k in EXACT_OUT}
    if kind == "nullity":
        nu, count = sre.stabilizer_nullity(state["psi"])
        return {"nullity": nu, "stab_count": count}
    if kind == "batched":
        rs = sre.sre_exact_batched(state["psis"])
        return {k: torch.tensor([r[k] for r in rs]) for k in EXACT_OUT}
    if kind == "mc_marginal":
        r = sre.sre_mc(state["psi"], sre.SRE_MC_MARGINAL, case["n_x"], case["z_per_x"], seed=state["seed"],
                       return_samples=True)
        return {k: r[k] for k in MC_OUT + ("xs", "zs", "c")}
    if kind == "mc_uniform":
        r = sre.sre_mc(state["psi"], sre.SRE_MC_UNIFORM, case["n_x"], seed=state["seed"])
        return {k: r[k] for k in MC_OUT + ("r2",)}
    if kind == "marginal":
        return sre.pauli_x_marginal(state["psi"])
    if kind in ("circuit", "brickwall"):
        # the state is kept and a preconditioned copy of it is made
        out = state["out"].copy_(state["psi"])
        if kind == "circuit":
            sre.apply_clifford_tdoped_circuit(out, state["gates"])
        else:
            sre.apply_two_qubit_gates(out, state["mats"], state["pairs"])
        return out
    r = sre.sre_mixed(state["psi"], case["N_A"])
    return {k: r[k] for k in ("M", "S2", "W")}


# -------------------------------------------------------------------- work
def _family_flops(N):
    """One X-mask family: the half-length complex product and transform (one
    real add per string and bit), and the four moments (ten per string)."""
    d = 2.0 ** N
    return 4.0 * d + (N - 1) * d + 10.0 * d


def work(case):
    kind, N = case["kind"], case["N"]
    d = 2.0 ** N
    if kind in ("exact", "nullity"):
        return {"bytes": 8 * d, "flops": d * _family_flops(N)}
    if kind == "batched":
        Ns = _sizes(case)
        return {"bytes": sum(8 * 2.0 ** n for n in Ns), "flops": sum(2.0 ** n * _family_flops(n) for n in Ns)}
    if kind == "mc_marginal":
        draws = case["n_x"] * case["z_per_x"]
        return {"bytes": 8 * d + 8 * case["n_x"] + 12 * draws, "flops": case["n_x"] * _family_flops(N) + 2 * N * d}
    if kind == "mc_uniform":
        return {"bytes": 8 * d, "flops": case["n_x"] * _family_flops(N)}
    if kind == "marginal":
        return {"bytes": 16 * d, "flops": (2 * N + 5) * d}
    if kind == "circuit":
        return {"bytes": 32 * d, "flops": 2 * d * case["gates"]}
    if kind == "brickwall":
        n = sum(len(range(layer % 2, N - 1, 2)) for layer in range(case["layers"]))
        return {"bytes": 32 * d, "flops": 32 * d * n}
    dA = 2.0 ** case["N_A"]
    # the Hermitian Gram matrix (half of it) and the subsystem's families
    return {"bytes": 8 * d, "flops": 4 * d * dA + dA * _family_flops(case["N_A"])}


# --------------------------------------------------- the same in 64 bits
def _wht(x):
    """Walsh-Hadamard transform of the last dimension, float64."""
    n = x.shape[-1]
    shape, bits = x.shape, n.bit_length() - 1
    low = min(4, bits)
    h = torch.ones(1, 1, dtype=torch.float64, device=x.device)
    for _ in range(low):
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    x = torch.matmul(x.reshape(-1, 1 << low), h)
    y = torch.empty_like(x)
    for s in range(low, bits):
        v, w = x.view(-1, 2, 1 << s), y.view(-1, 2, 1 << s)
        torch.add(v[:, 0], v[:, 1], out=w[:, 0])
        torch.sub(v[:, 0], v[:, 1], out=w[:, 1])
        x, y = y, x
    return x.reshape(shape)


def _family_sums(psi, xs, N):
    """For each x the sums over z of q, q^2, q^3, q log2 q (q = c_{x,z}^2), and the number of |c| = 1."""
    d = 1 << N
    psi = psi.to(torch.complex128)
    psi = psi / torch.linalg.vector_norm(psi)
    b = torch.arange(d, device=psi.device)
    out = torch.empty(len(xs), 5, dtype=torch.float64, device=psi.device)
    step = max(1, (1 << 27) >> N)
    for i in range(0, len(xs), step):
        x = xs[i:i + step]
        f = psi[b[None, :] ^ x[:, None]].conj_physical_().mul_(psi)
        # Re f and Im f feed the strings of even and of odd |x & z|, and never the same
        q = _wht(f.real + f.imag).square_()
        del f
        o = out[i:i + step]
        o[:, 0] = q.sum(1)
        o[:, 3] = torch.special.xlogy(q, q).sum(1) / math.log(2.0)
        o[:, 4] = ((q - 1.0).abs() < 2e-6).sum(1)
        q2 = q * q
        o[:, 1] = q2.sum(1)
        o[:, 2] = q2.mul_(q).sum(1)
    return out


def _r2(m, d):
    nz = m[1:]
    return float(nz.std(correction=0) / (m.sum() / d))


def _exact_state(psi, N):
    d = 2.0 ** N
    t = _family_sums(psi, torch.arange(1 << N, device=psi.device), N)
    T = [float(v) for v in t.sum(0)]
    P = T[0] / d
    H = N + math.log2(P) - T[3] / (d * P)
    S = [H, T[1] / (d * d * P * P), T[2] / (d * P) ** 3]
    count = int(T[4])
    return {"M": [H - N, -math.log2(S[1]) - N, -0.5 * math.log2(S[2]) - N], "S": S, "parseval": P, "r2": _r2(t[:, 1], d),
            "stab_count": count, "nullity": N - (count.bit_length() - 1)}


def _uniforms(n, seed):
    """Word 0 of Philox4x64-10 with key (seed, 0) and counter (i, 0, 0, 0), i < n, as a number in [0, 1)."""
    u = np.empty(n)
    for i in range(n):
        word = np.random.Philox(counter=np.array([(i - 1) % 2 ** 64, *([2 ** 64 - 1 if i == 0 else 0] * 3)], np.uint64),
                                key=np.array([seed, 0], np.uint64)).random_raw(1)[0]
        u[i] = (int(word) >> 11) * 2.0 ** -53
    return u


def _marginal(psi, N):
    q = psi.abs().double().square() if N > 27 else (psi.real.double().square() + psi.imag.double().square())
    return _wht(_wht(q / q.sum()).square_()) / 2.0 ** N


def _exact_mc(case, psi, seed):
    N, n_x = case["N"], case["n_x"]
    d = 2.0 ** N
    u = _uniforms(n_x, seed)
    uniform = case["kind"] == "mc_uniform"
    if uniform:
        xs = np.minimum(1 + (u * (d - 1)).astype(np.int64), (1 << N) - 1)
        xs = torch.from_numpy(xs).to(psi.device)
    else:
        p = _marginal(psi, N)
        cdf = torch.cumsum(p, 0)
        p0 = float(p[0])
        xs = torch.searchsorted(cdf, p0 + torch.from_numpy(u).to(psi.device) * (cdf[-1] - p0), right=True)
        xs = xs.clamp_(1, (1 << N) - 1)
        del p, cdf
    xs[0] = 0
    m = _family_sums(psi, xs, N).cpu().numpy()
    n = n_x - 1
    if uniform:
        y = np.stack([N * (m[:, 0] / d) - m[:, 3] / d, m[:, 1] / d ** 2, m[:, 2] / d ** 3], 1)
        mean, std = y[1:].mean(0), y[1:].std(0)
        S = y[0] + (d - 1) * mean
        a = np.array([1.0, 2.0, 3.0])
        M = [S[0] - N] + [math.log2(S[k]) / (1 - a[k]) - N for k in (1, 2)]
        r = std * d / S
        err = [(d - 1) * std[0] / math.sqrt(n)] + [r[k] / ((a[k] - 1) * math.log(2) * math.sqrt(n_x)) for k in (1, 2)]
        M, S, err = [float(v) for v in M], [float(v) for v in S], [float(v) for v in err]
        return {"M": M, "S": S, "err_M": err, "M_rb": M, "err_rb": err, "r2": float(r[1])}
    y = np.stack([-m[:, 3], m[:, 1], m[:, 2]], 1) / m[:, :1]
    mean, std = y[1:].mean(0), y[1:].std(0)
    S, se = p0 * y[0] + (1 - p0) * mean, (1 - p0) * std / math.sqrt(n)
    M_rb = [S[0]] + [math.log2(S[k]) / -k for k in (1, 2)]
    err = [se[0]] + [se[k] / (S[k] * k * math.log(2)) for k in (1, 2)]
    # the estimate from the drawn strings has no value apart from the draws
    return {"M": None, "S": None, "err_M": None, "M_rb": [float(v) for v in M_rb], "err_rb": [float(v) for v in err],
            "xs": None, "zs": None, "c": None}


def _exact_circuit(psi, gates):
    v = psi.to(torch.complex128)
    b = torch.arange(v.numel(), device=v.device)
    for op, q0, q1 in gates.tolist():
        if op == 0:
            v = _h(v, q0)
        elif op == 3:
            v = v[b ^ (((b >> q0) & 1) << q1)]
        else:
            v.view(-1, 2, 1 << q0)[:, 1] *= 1j if op == 1 else complex(math.sqrt(0.5), math.sqrt(0.5))
    return v


def _exact_brickwall(psi, mats, pairs):
    v = psi.to(torch.complex128)
    mats = torch.from_numpy(mats).to(v.device).to(torch.complex128)
    for u, (q0, q1) in zip(mats, pairs.tolist()):
        # neighbours q1 = q0 + 1: the local index bit(q0) + 2 bit(q1) is one axis
        v = torch.einsum("oi,aib->aob", u, v.view(-1, 4, 1 << q0)).reshape(-1)
    return v


def _exact_mixed(psi, N, N_A):
    dA = 1 << N_A
    a = psi.to(torch.complex128)
    a = (a / torch.linalg.vector_norm(a)).view(-1, dA)
    rho = a.transpose(0, 1) @ a.conj()
    i = torch.arange(dA, device=psi.device)
    W = np.zeros(4)
    step = max(1, (1 << 24) >> N_A)
    for x0 in range(0, dA, step):
        x = i[x0:x0 + step]
        f = rho[i[None, :].expand(len(x), -1), i[None, :] ^ x[:, None]]
        q = _wht(f.real + f.imag).square_()
        W += [float(q.sum()), float((q ** 2).sum()), float((q ** 3).sum()), float(torch.special.xlogy(q, q).sum()) / math.log(2)]
    S2 = -math.log2(W[0] / dA)
    M = [None, -math.log2(W[1] / dA ** 2) - N_A - S2, -0.5 * math.log2(W[2] / dA ** 3) - N_A - S2]
    return {"M": M, "S2": S2, "W": [float(v) for v in W]}


def exact(case, seed):
    kind, N = case["kind"], case["N"]
    st = prepare(case, seed)
    if kind in ("exact", "nullity"):
        r = _exact_state(st["psi"], N)
        return r if kind == "exact" else {k: r[k] for k in ("nullity", "stab_count")}
    if kind == "batched":
        rs = [_exact_state(psi, n) for psi, n in zip(st["psis"], _sizes(case))]
        return {k: torch.tensor([r[k] for r in rs], dtype=torch.int64 if k in ("stab_count", "nullity") else torch.float64)
                for k in EXACT_OUT}
    if kind in ("mc_marginal", "mc_uniform"):
        return _exact_mc(case, st["psi"], seed) if N <= 26 and case["n_x"] << N <= 1 << 36 else None
    if kind == "marginal":
        return _marginal(st["psi"], N)
    if kind == "circuit":
        return _exact_circuit(st["psi"], st["gates"]) if N <= 26 else None
    if kind == "brickwall":
        return _exact_brickwall(st["psi"], st["mats"], st["pairs"])
    return _exact_mixed(st["psi"], N, case["N_A"])
