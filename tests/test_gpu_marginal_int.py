"""The integer transforms of the x-marginal against extended precision, at the
edges of its plans: one strided bit (N = 13), 5 + 5 (N = 22), nine (N = 21).

Tolerance, in units u = 2^-53 of p(0), the sum of magnitudes that every p(x) is
a signed sum of: a pass rounds its inputs to 2^-61 of the largest sum of
magnitudes it forms (6 sigma over 2^11 inputs: 0.3 u of that sum) and its
outputs to u/2. Two transforms of at most three passes, the first one doubled
by the square, the square and the normalisation (four roundings of u/2) stay
below (2 * 3 + 3) * 0.8 + 2 < 10 u; the bound is 16 u."""
import numpy as np
import pytest
import torch

import paper_2601_00761_gb300 as sre
from paper_2601_00761_gb300 import inputs

pytestmark = pytest.mark.gpu


def _wht(v):
    h = 1
    v = v.copy()
    while h < v.size:
        w = v.reshape(-1, 2, h)
        a, b = w[:, 0].copy(), w[:, 1].copy()
        w[:, 0], w[:, 1] = a + b, a - b
        h *= 2
    return v


def _state(kind, N):
    if kind == "basis":
        return inputs.basis_state(N, (1 << N) - 3)
    if kind == "product":
        return inputs.random_product_state(N, 5)
    if kind == "t":
        return inputs.t_product_state(N, N // 2)
    v = inputs.unnormalised_gaussian_state(N, 6, scale={"haar": 1.0, "large": 1e15, "small": 1e-15}[kind])
    if kind == "haar":
        v[17] = 300.0        # one amplitude far above the others
    return v


@pytest.mark.parametrize("N,kind", [(N, k) for N in (13, 14, 16) for k in ("haar", "product", "basis", "t")] +
                         [(21, "haar"), (22, "product"), (17, "large"), (17, "small")])
def test_marginal_against_extended_precision(N, kind):
    psi = _state(kind, N)
    a = psi.real.astype(np.longdouble), psi.imag.astype(np.longdouble)
    q = a[0] * a[0] + a[1] * a[1]
    q /= q.sum()
    ref = _wht(_wht(q) ** 2) / q.size
    got = sre.pauli_x_marginal(torch.from_numpy(psi).cuda()).cpu().numpy()
    assert np.abs(got - ref).max() <= 16 * 2.0 ** -53 * float(ref[0])


@pytest.mark.parametrize("bad", [float("inf"), 3e38])
def test_marginal_of_a_norm_without_a_value(bad):
    psi = torch.ones(1 << 13, dtype=torch.complex64, device="cuda")
    psi[5] = bad
    p = sre.pauli_x_marginal(psi)
    # an infinite norm gives no number, as in FP64; 3e38 has a finite one
    assert bool(torch.isnan(p).all()) if bad == float("inf") else float(p[0]) == 1.0
