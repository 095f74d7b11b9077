"""Marginal Monte Carlo across the lines of its x and z draws: few draws on a
large state (chunk sums) against many (the whole CDF), rows of up to 2^14 ranges
against larger ones, families of few and of many tiles."""
import numpy as np
import pytest
import torch

import paper_2601_00761_gb300 as sre

pytestmark = pytest.mark.gpu


def _psi(N, kind="haar"):
    g = torch.Generator(device="cuda").manual_seed(N)
    psi = torch.view_as_complex(torch.randn(1 << N, 2, generator=g, device="cuda")) * 2.0 ** (-(N + 1) / 2)
    if kind == "sparse":                       # p(x) = 0 for most x
        psi[torch.arange(1 << N, device="cuda") % 37 != 0] = 0
    return psi


@pytest.mark.parametrize("N,kind", [(12, "haar"), (16, "haar"), (20, "haar"), (16, "sparse"), (21, "sparse")])
def test_x_draws_of_chunks_and_cdf(N, kind):
    """The first draws do not depend on how many there are; a draw from the chunk
    sums equals the CDF's unless rounding (2^-52 d of a draw's spacing) decides."""
    psi = _psi(N, kind)
    few = max(2, (1 << N) // 2048)
    a = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, few, 1, seed=3, return_samples=True)["xs"]
    b = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, few + 1, 1, seed=3, return_samples=True)["xs"][:few]
    assert torch.equal(a, b)
    p = sre.pauli_x_marginal(psi)
    assert a[0] == 0 and bool((a[1:] > 0).all()) and float(p[a].min()) > 0


@pytest.mark.parametrize("N", [24, 25, 26])
def test_z_draws_of_small_and_large_rows(N):
    """Draw k of a family does not depend on z_per_x; every drawn c is that of its
    string; the estimate agrees with the families' exact means."""
    psi = _psi(N)
    r = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, 6, 33, seed=5, return_samples=True)
    s = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, 6, 3, seed=5, return_samples=True)
    assert torch.equal(r["xs"], s["xs"]) and torch.equal(r["zs"][:, :3], s["zs"]) and torch.equal(r["c"][:, :3], s["c"])
    for i in (0, 1, 5):
        c = sre.sre_family_spectrum(psi, int(r["xs"][i]))[r["zs"][i]]
        assert float((c - r["c"][i]).abs().max()) <= 1e-6
    big = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, 4, 4096, seed=6)
    assert abs(big["M"][0] - big["M_rb"][0]) <= 6 * max(big["err_M"][0], 3.2 / 64)   # sd of -log2 c^2 is below 3.2
