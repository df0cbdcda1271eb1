"""A point's cross-section is the same, bit for bit, alone (per-line constants kept in a record) and in a call
of several points (constants formed in the kernel): the same cells, parts, edges and sums. Lists from
sparse to dense, narrow lines widened to the precision margin, zones of hundreds of points, wide lines;
and the (P,T) plan with one point a shard."""
import numpy as np
import pytest

from rox_testutil import q_pair, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2510_20870_gb300 as rox  # noqa: E402
from paper_2510_20870_gb300 import dist as rd  # noqa: E402
from test_gpu_parity import _run_xsec, _small_lines  # noqa: E402


@pytest.mark.parametrize("points,dnu,cutoff,lines,P,T,mass", [
    (4097, 0.01, 25.0, 60000, 0.1, 1500.0, 16.0),
    (4097, 0.01, 25.0, 2000, 1e-5, 300.0, 200.0),
    (20000, 0.05, 100.0, 200000, 1e-4, 300.0, 44.0),
    (20000, 0.01, 14.0, 90000, 3.0, 3000.0, 16.0),
    (6001, 0.001, 10.0, 50000, 20.0, 500.0, 18.0),
    (6001, 0.001, 10.0, 50000, 1e-3, 3000.0, 2.0),
    (100001, 0.01, 25.0, 300000, 0.01, 1000.0, 2.0),
    (3000, 0.05, 100.0, 20000, 100.0, 296.0, 16.0),
    (12001, 0.02, 50.0, 400000, 0.5, 800.0, 16.0),
])
def test_point_alone_and_among_others(points, dnu, cutoff, lines, P, T, mass):
    lo = 3000.0
    hi = lo + dnu * (points - 1)
    w, L = _small_lines(1, lines, lo - 1.2 * cutoff, hi + 1.2 * cutoff, 61)
    dl, grid, Qr = to_device(L, torch), (lo, dnu, points), q_pair(w, 296.0)[1]
    pts = [(P, T, q_pair(w, T)[0]), (2 * P, T, q_pair(w, T)[0]), (P, T + 100.0, q_pair(w, T + 100.0)[0])]
    several, _ = _run_xsec(dl, grid, pts, Qr, mass, cutoff, flags=rox.ROX_KAHAN)
    for k, pt in enumerate(pts):
        alone, _ = _run_xsec(dl, grid, [pt], Qr, mass, cutoff, flags=rox.ROX_KAHAN)
        assert np.array_equal(alone[0], several[k]), (k, int((alone[0] != several[k]).sum()))


def test_one_point_a_shard():
    w, L = _small_lines(1, 12000, 4990.0, 5110.0, 51)
    grid, dl, Qr = (5000.0, 0.01, 10001), to_device(L, torch), q_pair(w, 296.0)[1]
    pts = [(P, T, q_pair(w, T)[0]) for P in (1e-3, 1.0, 30.0) for T in (500.0, 2500.0)]
    full, _ = _run_xsec(dl, grid, pts, Qr, w.mass_amu, 25.0)
    parts = [_run_xsec(dl, grid, rd.point_shard(pts, 6, r)[0], Qr, w.mass_amu, 25.0)[0] for r in range(6)]
    assert np.array_equal(np.concatenate(parts), full)
