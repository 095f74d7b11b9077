"""x draws of the marginal estimator where p(0) is so close to 1 that only a few
doubles lie between p(0) and the total: t = p(0) + u (total - p(0)) then rounds to
the total in a fraction of the draws. A drawn x has positive p all the same."""
import numpy as np
import pytest
import torch

import paper_2601_00761_gb300 as sre

pytestmark = pytest.mark.gpu


# x = 1 lies in the chunk (4096 x) of x = 0, 4095 and 4096 beside a chunk's edge,
# 5000 and 70000 in later chunks; N = 26 has 2^14 chunks, more than one tile of the
# scan, with x = 33558528 in the second one.
@pytest.mark.parametrize("N,other", [(12, 1), (20, 1), (20, 4095), (20, 4096), (20, 5000), (20, 70000),
                                     (26, 1), (26, 33558528)])
@pytest.mark.parametrize("b", [1e-7, 3e-8])
def test_drawn_x_have_positive_p(N, other, b):
    """a|0> + b|other>: p is positive at 0 and other alone."""
    psi = torch.zeros(1 << N, dtype=torch.complex64, device="cuda")
    psi[0], psi[other] = 1, b
    p = sre.pauli_x_marginal(psi)
    assert float(p[other]) > 0 and int((p > 0).sum()) == 2
    few = max(2, min(512, (1 << N) // 2048))
    for seed in range(4):
        r = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, few, 2, seed=seed, return_samples=True)
        assert r["xs"][0] == 0 and bool((r["xs"][1:] == other).all())
        assert np.isfinite(r["M_rb"]).all() and np.isfinite(r["M"]).all()


def test_all_mass_at_zero():
    """|0...0>: no x but 0 has positive p; the draws take x = 1, as from the CDF."""
    psi = torch.zeros(1 << 20, dtype=torch.complex64, device="cuda")
    psi[0] = 1
    for n_x in (512, 513):                  # chunk sums, the whole CDF
        r = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, n_x, 1, seed=1, return_samples=True)
        assert r["xs"][0] == 0 and bool((r["xs"][1:] == 1).all())


@pytest.mark.parametrize("N", [8, 10, 12])
@pytest.mark.parametrize("b", [1e-7, 3e-8])
def test_families_of_rounding_noise(N, b):
    """|0> + sum b_k |x_k>: 1 - p(0) is some 1e-14, so the rounding of the marginal (1e-17)
    is drawn too, and with it families without any weight. The estimates stay what
    the x = 0 stratum makes them (1e-5, the bound of every M)."""
    r = np.random.Generator(np.random.PCG64(N))
    for seed in range(8):
        at = torch.from_numpy(r.choice(np.arange(1, 1 << N), 6, replace=False)).cuda()
        psi = torch.zeros(1 << N, dtype=torch.complex64, device="cuda")
        psi[0] = 1
        psi[at] = torch.from_numpy(b * np.sqrt(r.random(6) + 0.1)).to(psi)
        got = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, 4000, 2, seed=seed)
        exact = sre.sre_exact(psi)
        for k in ("M", "M_rb"):
            assert np.abs(np.array(got[k]) - exact["M"]).max() <= 1e-5
        assert np.isfinite(got["err_M"]).all() and np.isfinite(got["err_rb"]).all()


# few draws go through the chunk sums, many through the CDF (n_x > 2^N / 2048)
@pytest.mark.parametrize("N,n_x", [(10, 4000), (12, 4000), (16, 4000), (20, 512), (20, 4000), (22, 4000)])
@pytest.mark.parametrize("b", [1e-7, 3e-8])
def test_several_x_of_little_mass(N, n_x, b):
    """|0> + sum b_k |x_k>: prefixes over several of the p(x_k) round differently from
    chunk to chunk, by as much as a p(x_k) is worth."""
    r = np.random.Generator(np.random.PCG64(N))
    for seed in range(4):
        at = torch.from_numpy(r.choice(np.arange(1, 1 << N), 6, replace=False)).cuda()
        psi = torch.zeros(1 << N, dtype=torch.complex64, device="cuda")
        psi[0] = 1
        psi[at] = torch.from_numpy(b * np.sqrt(r.random(6) + 0.1)).to(psi)
        p = sre.pauli_x_marginal(psi)
        got = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, n_x, 2, seed=seed, return_samples=True)
        assert float(p[got["xs"]].min()) > 0
        assert np.isfinite(got["M_rb"]).all()
