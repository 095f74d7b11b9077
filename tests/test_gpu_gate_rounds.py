"""Gate blocks in register rounds against a plain complex128 update of the state,
at the edges of the tiling: fewer qubits than a thread's five slots, one tile of
fewer than 13 qubits, one full tile, several tiles; every opcode, controls and
phases on slots and on thread bits, two-qubit matrices in both qubit orders.
Tolerance: 1e-6 per amplitude, as for the other gate tests (FP32 rounding of at
most 200 gates is about 3 * 2^-24 * sqrt(200) of an amplitude of norm at most 1)."""
import numpy as np
import pytest
import torch

import paper_2601_00761_gb300 as sre

pytestmark = pytest.mark.gpu

W = np.exp(1j * np.pi / 4)
ONE = {0: np.array([[1, 1], [1, -1]]) / np.sqrt(2), 1: np.diag([1, 1j]), 2: np.diag([1, -1j]), 4: np.diag([1, W]),
       5: np.diag([1, W.conjugate()])}


def _apply1(v, m, q):
    return np.einsum("oi,aib->aob", m, v.reshape(-1, 2, 1 << q)).reshape(-1)


def _apply2(v, m, q0, q1):
    b = np.arange(v.size)
    out = np.zeros_like(v)
    l = ((b >> q0) & 1) + 2 * ((b >> q1) & 1)
    base = b & ~((1 << q0) | (1 << q1))
    for i in range(4):
        out += m[l, i] * v[base | ((i & 1) << q0) | ((i >> 1) << q1)]
    return out


def _psi(N, r):
    v = r.standard_normal(1 << N) + 1j * r.standard_normal(1 << N)
    return (v / np.linalg.norm(v)).astype(np.complex64)


@pytest.mark.parametrize("N", [1, 2, 4, 5, 6, 8, 12, 13, 14, 16])
@pytest.mark.parametrize("n", [1, 200])
def test_gate_list(N, n):
    r = np.random.default_rng(7 * N + n)
    psi = _psi(N, r)
    ops = r.choice([0, 1, 2, 4, 5] + ([3, 3, 0] if N > 1 else []), n)
    rows = []
    v = psi.astype(np.complex128)
    for op in ops:
        q0, q1 = (int(q) for q in (r.permutation(N)[:2] if N > 1 else (0, 0)))
        rows.append((op, q0, q1))
        if op == 3:
            b = np.arange(v.size)
            v = v[b ^ (((b >> q0) & 1) << q1)]
        else:
            v = _apply1(v, ONE[int(op)], q0)
    p = torch.from_numpy(psi).cuda()
    sre.apply_clifford_tdoped_circuit(p, rows)
    assert np.abs(p.cpu().numpy() - v).max() <= 1e-6


@pytest.mark.parametrize("N", [2, 4, 5, 6, 12, 13, 15])
@pytest.mark.parametrize("n", [1, 60])
def test_two_qubit_list(N, n):
    r = np.random.default_rng(11 * N + n)
    psi = _psi(N, r)
    mats = np.linalg.qr(r.standard_normal((n, 4, 4)) + 1j * r.standard_normal((n, 4, 4)))[0].astype(np.complex64)
    pairs = np.array([r.permutation(N)[:2] for _ in range(n)], np.int32)
    v = psi.astype(np.complex128)
    for m, (q0, q1) in zip(mats.astype(np.complex128), pairs.tolist()):
        v = _apply2(v, m, q0, q1)
    p = torch.from_numpy(psi).cuda()
    sre.apply_two_qubit_gates(p, mats, pairs)
    assert np.abs(p.cpu().numpy() - v).max() <= 1e-6
