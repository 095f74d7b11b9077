"""The autotuner's table: entries of their own for the marginal estimator and for the
sweeps without z draws, in memory and in SRE_TUNE_FILE (host only), and no entry
where the planned tiling is the faster one (GPU)."""
import os
import subprocess
import sys

import pytest

import paper_2601_00761_gb300 as sre

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import paper_2601_00761_gb300 as sre
U, M = sre.SRE_MC_UNIFORM, sre.SRE_MC_MARGINAL
row = lambda N: sre.sre_make_plan(N)["pass_bits"][-1]
ws = lambda N, mode, **o: sre.sre_workspace_bytes(N, mode, 20000, 2, **o)
assert row(18) == 13 and row(17) == 11 and row(16) == 12
assert ws(18, U) == ws(18, U, radix_log2=12) and ws(18, -1) == ws(18, -1, radix_log2=12)
assert ws(18, M) == ws(18, M, radix_log2=13)
assert ws(17, M) == ws(17, M, radix_log2=11)
assert ws(16, U) == ws(16, U, radix_log2=12) and ws(16, M) == ws(16, M, radix_log2=12)
tuned = {N: (ws(N, U), ws(N, -1)) for N in (16, 17, 18)}
sre.sre_autotune_clear(16)
left = open(FILE).read().splitlines()
assert left == ["17 11 0 0 marginal", "18 12 0 0 sweep"], left
sre.sre_autotune_clear(0)
assert open(FILE).read() == ""
assert all(row(N) == 13 for N in (16, 17, 18))
assert (ws(17, U), ws(17, -1)) == tuned[17] and ws(18, U) != tuned[18][0] and ws(16, U) != tuned[16][0]
"""


def test_entries_by_kind(tmp_path):
    """A word after the four numbers names the kind of call; without it (files of an
    earlier version) the line holds for both. Unknown words and sizes are ignored."""
    from paper_2601_00761_gb300 import build
    build.build()
    f = tmp_path / "tune.txt"
    f.write_text("18 12 0 0 sweep\n17 11 0 0 marginal\n16 12 0 0\n17 14 0 0 else\n40 12 0 0\n\n19 12\n")
    r = subprocess.run([sys.executable, "-c", f"FILE = {str(f)!r}\n" + CHILD], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, SRE_TUNE_FILE=str(f)))
    assert r.returncode == 0, r.stderr[-2000:]


def _exact_ms(psi):
    import torch
    best = float("inf")
    for _ in range(9):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        sre.sre_exact(psi)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


@pytest.mark.gpu
@pytest.mark.parametrize("N", [15, 16])
def test_tuning_does_not_slow_the_sweep(N, tmp_path, monkeypatch):
    """Planned: 10-bit rows and launches of 16384 families, which no explicit tiling
    gets. The tuned call is that plan or a faster one (3% for the timing's scatter)."""
    import torch
    from paper_2601_00761_gb300 import inputs
    f = tmp_path / "tune.txt"
    monkeypatch.setenv("SRE_TUNE_FILE", str(f))
    sre.sre_autotune_clear(0)
    psi = torch.from_numpy(inputs.haar_state(N, 3)).cuda()
    before, planned = sre.sre_exact(psi), _exact_ms(psi)
    rows = sre.sre_make_plan(N)["pass_bits"][-1]
    best = sre.sre_autotune(psi)
    after, tuned = sre.sre_exact(psi), _exact_ms(psi)
    lines = [line.split() for line in f.read_text().splitlines()]
    row = sre.sre_make_plan(N)["pass_bits"][-1]
    sre.sre_autotune_clear(0)
    planned = max(planned, _exact_ms(psi))         # before and after, should the clocks drift
    assert tuned <= 1.03 * planned
    assert all(len(w) == 5 and w[4] in ("marginal", "sweep") for w in lines)
    marg = [w for w in lines if w[4] == "marginal"]
    assert row == (int(marg[0][1]) if marg else rows)
    assert best["radix_log2"] in (0, row)
    if not [w for w in lines if w[4] == "sweep"]:
        assert after["M"] == before["M"]
