"""Nullity of states whose stabilizer strings all lie in one flagged family (x = 0):
|T>^(N-m) |0>^m has the 2^m strings of Z's on the |0> qubits. m walks through the
recount's routes: one candidate, cosets of up to 6 dimensions (64 candidates),
and the overflow to the FP64 transform; N walks across the line where eight CTAs
share a family, and the totals across one block, several blocks and their limit."""
import numpy as np
import pytest
import torch

import paper_2601_00761_gb300 as sre
from paper_2601_00761_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [7, 8, 9, 12, 13, 14, 16, 17])
@pytest.mark.parametrize("m", [0, 1, 4, 5, 6, 7])
def test_one_family(N, m):
    psi = torch.from_numpy(inputs.product_state([inputs.ZERO_QUBIT] * m + [(0.6, 0.48 + 0.64j)] * (N - m))).cuda()
    r = sre.sre_exact(psi)
    assert (r["n_flagged"], r["stab_count"], r["nullity"]) == (1, 1 << m, N - m)
    # every qubit off the axes contributes the same entropies; err_M bounds the FP32 rounding
    one = sre.sre_exact(torch.tensor([0.6, 0.48 + 0.64j], dtype=torch.complex64, device="cuda"))
    assert (np.abs(np.array(r["M"]) - (N - m) * np.array(one["M"])) <= np.array(r["err_M"]) * (N + 1)).all()
