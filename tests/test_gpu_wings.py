"""The Voigt kernel's treatment of the wings against the FP64 oracle, at the sizes where it changes
over: lines smooth on a span (Chebyshev points), multipole cells, window edges (running sums of
moments, or masked pairs where the cutoff is too short for them), batches of slow zones, spans cut by
the end of the grid, and more parts than 16 on short grids.

Tolerance per point: the profile forms' own bounds (zone forms 4e-6; far form 3.5e-6, for y >= 11.5 the
2-level fraction's 1.1e-5), the expansions' (interpolation and moments 1e-7 each of a line's value
nearby, a few 1e-7 across a span) and FP32 sums: 1.5e-5 of the cross-section where it exceeds 1e-6 of the
maximum."""
import numpy as np
import pytest

import oracle
from rox_testutil import check_sigma, q_pair, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2510_20870_gb300 as rox  # noqa: E402
from test_gpu_parity import _run_xsec, _small_lines  # noqa: E402

TOL = 1.5e-5


# (points, dnu, cutoff, lines, P, T): cutoffs below, at and above two spans (512 steps) and long ones;
# grids of one span less, exactly and one point more than whole spans; a line per cell and many
@pytest.mark.parametrize("points,dnu,cutoff,lines,P,T", [
    (255, 0.01, 25.0, 4000, 0.1, 1000.0),
    (256, 0.01, 25.0, 4000, 1e-5, 300.0),
    (257, 0.01, 25.0, 4000, 100.0, 300.0),
    (4097, 0.01, 5.1, 6000, 0.1, 1500.0),
    (4097, 0.01, 5.15, 6000, 1.0, 500.0),
    (4097, 0.01, 14.0, 6000, 3.0, 3000.0),
    (6000, 0.01, 25.0, 300, 0.3, 800.0),
    (6000, 0.01, 25.0, 9000, 1e-3, 2000.0),
    (3000, 0.05, 100.0, 9000, 10.0, 1000.0),
    (12001, 0.002, 25.0, 5000, 0.02, 296.0),
])
def test_wings_vs_oracle(points, dnu, cutoff, lines, P, T):
    lo = 3000.0
    hi = lo + dnu * (points - 1)
    w, L = _small_lines(1, lines, lo - 1.2 * cutoff, hi + 1.2 * cutoff, 61)
    grid = (lo, dnu, points)
    Qt, Qr = q_pair(w, T)
    ref = oracle.xsec_windowed(L, grid, P, T, Qt, Qr, 16.0, cutoff)
    sig, evals = _run_xsec(to_device(L, torch), grid, [(P, T, Qt)], Qr, 16.0, cutoff, flags=rox.ROX_KAHAN)
    check_sigma(sig[0], ref, rel_tol=TOL, label="%d points, cutoff %g, P=%g" % (points, cutoff, P))
    assert evals == oracle.count_evals(L["nu0"], *grid, cutoff)
    # several points of one call take the constants in the kernel instead of from the record
    two, _ = _run_xsec(to_device(L, torch), grid, [(P, T, Qt), (3 * P, T, Qt)], Qr, 16.0, cutoff, flags=rox.ROX_KAHAN)
    check_sigma(two[0], ref, rel_tol=TOL, label="with a second point")
