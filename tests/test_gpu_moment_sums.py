"""FP32 partial sums of the family moments: no sum covers more than 32 points of a
thread before the tree over the warp, whichever row kernel runs.

psi = |0> + b |x> gives family x one value of |c| at every point, so every FP32 q^2
of the family is the same number and a running sum rounds the same way at each step.
b is chosen so that 32 additions lose almost nothing and 64 lose much: in the second
32 the sum's last place is larger, and each step drops nearly half of it."""
import numpy as np
import pytest
import torch

import paper_2601_00761_gb300 as sre

pytestmark = pytest.mark.gpu
U = 2.0 ** -24
f32 = np.float32


def _q2(b):
    """FP32 c^4 as the kernels form it, every step rounded once: s, 2 s, h = b, c, q, q^2."""
    s = f32(1.0 / (1.0 + float(b) * float(b)))
    c = f32(f32(f32(2.0) * s) * b)
    q = f32(c * c)
    return f32(q * q)


def _chain(v, n):
    t = f32(0)
    for _ in range(n):
        t = f32(t + v)
    return float(t) / (n * float(v)) - 1.0


def _find_b():
    for i in range(20000):
        b = f32(0.5 + i * 2.0 ** -16)
        v = _q2(b)
        if abs(_chain(v, 32)) < 2 * U and abs(_chain(v, 64)) > 8 * U:
            return b
    raise AssertionError("no such b")


@pytest.mark.parametrize("N", [16, 18, 20, 21, 24, 25])      # rows of 10, 12 and 13 bits
def test_no_sum_over_more_than_32_points(N):
    """Uniform estimate from x = 0 and one drawn x: S_2 = m_{2;0} + (d - 1) m_{2;x}, and
    m_{2;x} = sum c^4 / d^2 is half of d equal terms. Tree and FP64 sums of equal
    numbers are exact, so 32 additions' error (< 2 U) is all there is, and one more U
    for the FP64 arithmetic around it; 64 additions are off by more than 8 U."""
    b, d, seed = _find_b(), 2.0 ** N, 7
    probe = torch.zeros(1 << N, dtype=torch.complex64, device="cuda")
    probe[0] = 1
    x = int(sre.sre_mc(probe, sre.SRE_MC_UNIFORM, 2, seed=seed, return_samples=True)["xs"][1])
    assert x > 0
    probe[x] = float(b)
    r = sre.sre_mc(probe, sre.SRE_MC_UNIFORM, 2, seed=seed)
    n2 = 1.0 + float(b) ** 2
    c0 = (1.0 - float(b) ** 2) / n2                  # family 0: half of its c are 1, half c0
    want = (0.5 * d * (1.0 + c0 ** 4) + (d - 1) * 0.5 * d * float(_q2(b))) / d ** 2
    assert abs(r["S"][1] / want - 1.0) <= 3 * U
