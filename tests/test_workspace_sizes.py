"""Workspace of a call: an intermediate for the families it runs, not for a full
launch (host only), and smaller plans where the library's own allocation of the
preferred one is refused (GPU)."""
import numpy as np
import pytest

import paper_2601_00761_gb300 as sre
from paper_2601_00761_gb300 import inputs


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2601_00761_gb300 import build
    build.build()
    sre.load()
    sre.sre_autotune_clear(0)


@pytest.mark.parametrize("mode", [sre.SRE_MC_UNIFORM, sre.SRE_MC_MARGINAL])
@pytest.mark.parametrize("N", [15, 16, 17, 18, 21, 24])
@pytest.mark.parametrize("n_x", [2, 16])
def test_few_families_take_little(N, mode, n_x):
    """Packed intermediate 8 bytes x 2^(N-1) a family, at most a tile partial (64
    bytes) per 2^10 points and a range weight (4 bytes) per 2^10 z; the marginal
    holds p, its work space and psi's copy (24 bytes per amplitude); 1 MB for the rest."""
    family = (8 << (N - 1)) + (64 << max(0, N - 11)) + (4 << max(0, N - 10))
    marg = 24 << N if mode == sre.SRE_MC_MARGINAL else 0
    assert sre.sre_workspace_bytes(N, mode, n_x, 4) <= n_x * family + marg + (1 << 20)


def test_more_families_take_more_up_to_a_launch():
    b = [sre.sre_workspace_bytes(16, sre.SRE_MC_UNIFORM, n, 1) for n in (2, 100, 5000, 16384)]
    assert b == sorted(b) and b[0] < b[-1]
    # beyond a launch only the per-family records grow (160 bytes each at most)
    assert sre.sre_workspace_bytes(16, sre.SRE_MC_UNIFORM, 20000, 1) - b[-1] <= 160 * (20000 - 16384) + 4096


def _hold_all_but(torch, leave):
    """Device memory in one tensor so that at most `leave` bytes stay free."""
    sre.sre_release_workspace()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - leave, dtype=torch.uint8, device="cuda")


@pytest.mark.gpu
@pytest.mark.parametrize("call", ["exact", "uniform", "batched"])
def test_short_memory_runs_a_smaller_plan(call):
    """Between the 13-bit split's need and the preferred plan's: the call runs, and
    gives what it gives with memory to spare (err_M of both, as in the split tests)."""
    import torch
    N = 16
    psi = torch.from_numpy(inputs.haar_state(N, 5)).cuda()
    run = {"exact": lambda: sre.sre_exact(psi),
           "uniform": lambda: sre.sre_mc(psi, sre.SRE_MC_UNIFORM, 9000, seed=2),
           "batched": lambda: sre.sre_exact_batched([psi, psi])[1]}[call]
    if call == "uniform":
        full = sre.sre_workspace_bytes(N, sre.SRE_MC_UNIFORM, 9000, 1)
        small = sre.sre_workspace_bytes(N, sre.SRE_MC_UNIFORM, 9000, 1, radix_log2=13)
    else:
        full, small = sre.sre_workspace_bytes(N, -1), sre.sre_workspace_bytes(N, -1, radix_log2=13)
    a = run()
    assert full - small > 1 << 30
    hold = _hold_all_but(torch, (full + small) // 2)
    try:
        b = run()
        c = run()                          # from the workspace that is there
    finally:
        del hold
        torch.cuda.empty_cache()
        sre.sre_release_workspace()
    ec = (N + 2) * 2.0 ** -24
    bound = 2 * np.array([2 * ec * (N + 2), 4 * ec / np.log(2), 3 * ec / np.log(2)])
    assert (np.abs(np.array(a["M"]) - b["M"]) <= bound).all()
    assert b["M"] == c["M"] and b["nullity"] == a["nullity"]
    assert run()["M"] == a["M"]            # memory is back: the preferred plan
