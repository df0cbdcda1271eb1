"""How a short grid's lines are divided among the GPU's warps, where an average over the reach of the
cutoff says little: 3,000 lines on 301 points. Cutoffs that all reach over the whole grid mean the
same work, so the longer one may not take much longer (0.20 and 0.24 ms; in parts sized by the
average it took 2.7 times as long), and the sums agree with the oracle.

Tolerance as in test_gpu_wings.py (1.5e-5); time: a factor of 1.6 between the fastest of 20 calls each."""
import numpy as np
import pytest

import oracle
import rox_synth as rs
from rox_testutil import check_sigma, q_pair, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2510_20870_gb300 as rox  # noqa: E402
from test_gpu_parity import _small_lines  # noqa: E402


def _run(dl, grid, P, T, q, mass, cutoff, reps):
    ws = torch.empty(rox.rox_xsec_workspace_size(dl["nu0"].numel(), grid, 1), dtype=torch.uint8, device="cuda")
    sigma = torch.empty((1, grid[2]), dtype=torch.float32, device="cuda")
    best = float("inf")
    for _ in range(reps):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        rox.rox_xsec(dl, grid, P, T, q[0], q[1], mass, cutoff, sigma, ws)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    rc, evals = rox.rox_ws_status(ws)
    assert rc == 0
    return sigma[0].double().cpu().numpy(), evals, best


@pytest.mark.parametrize("P", [1e-4, 100.0])
@pytest.mark.parametrize("points", [1, 255, 301, 4001])
def test_lines_gathered_on_a_short_grid(points, P):
    T, dnu, lo = 1500.0, 0.002, 12000.0
    grid = (lo, dnu, points)
    w, L = _small_lines(1, 3000, lo, lo + dnu * max(points - 1, 1), 17)
    dl, q = to_device(L, torch), q_pair(w, T)
    times = []
    for cutoff in (20.0, 100.0):
        sig, evals, t = _run(dl, grid, P, T, q, 16.0, cutoff, 20)
        assert evals == 3000 * points
        times.append(t)
        j = np.linspace(0, points - 1, min(points, 40)).astype(int)
        ref = np.array([oracle.xsec_window(L, grid, int(k), int(k) + 1, P, T, q[0], q[1], 16.0, cutoff)[0] for k in j])
        check_sigma(sig[j], ref, M=float(sig.max()), rel_tol=1.5e-5, label="%d points, cutoff %g" % (points, cutoff))
    assert times[1] < 1.6 * times[0], times
