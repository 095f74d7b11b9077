"""The 10-bit strided pass from the copy of psi in tile order (64 families and
more) against the pass that reads psi itself (fewer). The amplitudes and the
arithmetic are the same, so every draw is bit-identical."""
import numpy as np
import pytest
import torch

import paper_2601_00761_gb300 as sre

pytestmark = pytest.mark.gpu


def _haar(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn(1 << n, 2, generator=g, device="cuda")) * 2.0 ** (-(n + 1) / 2)


@pytest.mark.parametrize("low", [24, 15, 14, 13, 12, 5])
def test_marginal_draws_are_the_same(low):
    """|0> on the qubits from `low` on: x < 2^low, so its top bit lies in the rows
    (13 and up), in the tile index or in the columns."""
    psi = torch.zeros(1 << 24, dtype=torch.complex64, device="cuda")
    psi[:1 << low] = _haar(low, low)
    a = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, 63, 16, seed=11, return_samples=True)
    b = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, 64, 16, seed=11, return_samples=True)
    assert int(a["xs"].max()) < 1 << low
    for k in ("xs", "zs", "c"):
        assert torch.equal(a[k], b[k][:63])


@pytest.mark.parametrize("N", [23, 24])
def test_uniform(N):
    psi = _haar(N, N)
    a = sre.sre_mc(psi, sre.SRE_MC_UNIFORM, 70, seed=4)
    b = sre.sre_mc(psi, sre.SRE_MC_UNIFORM, 70, seed=4, radix_log2=14)      # nine strided bits: never tiled
    ec = (N + 2) * 2.0 ** -24                                               # both within err_M of an exact sweep
    bound = 2 * np.array([2 * ec * (N + 2), 4 * ec / np.log(2), 3 * ec / np.log(2)])
    assert (np.abs(np.array(a["M"]) - b["M"]) <= bound).all()
