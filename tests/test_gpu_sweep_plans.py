"""Exact and uniform Monte Carlo sweeps in the splits they choose themselves
(rows of 10 to 13 bits, strided passes of 4 to 10) against explicit 13-bit
rows on the same state. Both are FP32 transforms of the same families, each
within err_M of the exact value, so they differ by at most twice that."""
import numpy as np
import pytest
import torch

import paper_2601_00761_gb300 as sre
from paper_2601_00761_gb300 import inputs

pytestmark = pytest.mark.gpu


def _psi(N):
    g = torch.Generator(device="cuda").manual_seed(100 + N)
    return torch.view_as_complex(torch.randn(1 << N, 2, generator=g, device="cuda")) * 2.0 ** (-(N + 1) / 2)


def _bound(N):
    # err_M of an exact sweep: relative rounding (N + 2) 2^-24 of each c, N-fold in M_1
    ec = (N + 2) * 2.0 ** -24
    return 2 * np.array([2 * ec * (N + 2), 4 * ec / np.log(2), 3 * ec / np.log(2)])


@pytest.mark.parametrize("N", [15, 16, 17])
@pytest.mark.parametrize("kind", ["haar", "product"])
def test_exact_sweep_split(N, kind):
    psi = _psi(N) if kind == "haar" else torch.from_numpy(inputs.t_product_state(N, 5)).cuda()
    a = sre.sre_exact(psi, allow_nullity_error=True)
    b = sre.sre_exact(psi, radix_log2=13, allow_nullity_error=True)
    assert (np.abs(np.array(a["M"]) - b["M"]) <= _bound(N)).all()
    assert (a["stab_count"], a["nullity"], a["n_flagged"]) == (b["stab_count"], b["nullity"], b["n_flagged"])


@pytest.mark.parametrize("N", [15, 18, 19, 20, 21, 22, 23, 24, 25, 26, 28])
def test_uniform_sweep_split(N):
    psi = _psi(N)
    n_x = 37 if N < 24 else 5
    a = sre.sre_mc(psi, sre.SRE_MC_UNIFORM, n_x, seed=9)
    b = sre.sre_mc(psi, sre.SRE_MC_UNIFORM, n_x, seed=9, radix_log2=13)
    # the same families: S is (d - 1) times a mean, so compare M; M_1's rounding is relative to S_1 <= 2 N
    assert (np.abs(np.array(a["M"]) - b["M"]) <= _bound(N)).all()


def test_workspace_of_the_13_bit_split():
    """A workspace that holds the 13-bit split (and no copy of psi) is accepted and
    runs that one; a smaller one is refused."""
    psi = _psi(17)
    n = sre.sre_workspace_bytes(17, -1, radix_log2=13)
    assert n < sre.sre_workspace_bytes(17, -1)
    ws = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
    ws = ws[-ws.data_ptr() % 256:][:n]
    a, b = sre.sre_exact(psi, workspace=ws), sre.sre_exact(psi, radix_log2=13)
    assert a["M"] == b["M"] and a["stab_count"] == b["stab_count"]
    with pytest.raises(sre.SreError):
        sre.sre_exact(psi, workspace=ws[:n // 2])
    psi = _psi(24)
    n = sre.sre_workspace_bytes(24, sre.SRE_MC_MARGINAL, 64, 4, precision=sre.SRE_BF16X3_TC)
    assert n < sre.sre_workspace_bytes(24, sre.SRE_MC_MARGINAL, 64, 4)
    ws = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
    ws = ws[-ws.data_ptr() % 256:][:n]
    a = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, 64, 4, seed=1, workspace=ws, return_samples=True)
    b = sre.sre_mc(psi, sre.SRE_MC_MARGINAL, 64, 4, seed=1, return_samples=True)
    assert all(torch.equal(a[k], b[k]) for k in ("xs", "zs", "c"))
