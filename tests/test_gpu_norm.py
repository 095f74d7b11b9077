"""sum |psi|^2 at the edges of its kernels (one block, two launches, ragged
groups) and of the float range, against exact rational sums. Each group of eight
amplitudes loses less than 2^-53 of its sum, and there are at most 2^-53 per FP64
addition of the rest (under 100 in a row at these sizes): 1e-14 relative."""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

import paper_2601_00761_gb300 as sre

pytestmark = pytest.mark.gpu


def _exact(psi):
    v = psi.view(np.float32).astype(np.float64)
    m = max(0, -math.frexp(float(np.abs(v).max()))[1])
    w = v * 2.0 ** m                                   # exact: only the exponents move
    return Fraction(math.fsum((w * w).tolist())) / Fraction(4) ** m


@pytest.mark.parametrize("N", [1, 2, 5, 10, 13, 14, 16, 18])
@pytest.mark.parametrize("kind", ["gauss", "spread", "tiny", "large", "one"])
def test_norm2(N, kind):
    r = np.random.default_rng(N)
    v = r.standard_normal(1 << N) + 1j * r.standard_normal(1 << N)
    if kind == "spread":
        v *= 10.0 ** r.uniform(-18, 18, 1 << N)
    psi = (v * {"tiny": 1e-40, "large": 1e37}.get(kind, 1.0)).astype(np.complex64)
    if kind == "one":
        psi = np.zeros(1 << N, np.complex64)
        psi[-1] = 3.0 - 4.0j
    got = sre.sre_norm2(torch.from_numpy(psi).cuda())
    assert abs(Fraction(got) / _exact(psi) - 1) <= 1e-14


@pytest.mark.parametrize("N", [3, 15])
def test_norm2_without_a_value(N):
    psi = torch.ones(1 << N, dtype=torch.complex64, device="cuda")
    psi[1] = float("inf")
    assert sre.sre_norm2(psi) == math.inf
    psi[2] = float("nan")
    assert math.isnan(sre.sre_norm2(psi))
