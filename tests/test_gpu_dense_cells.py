"""Compensated summation (ROX_KAHAN) where most of a cross-section is sums over many lines: one strong
line ahead of a few hundred thousand weak ones, each below half a unit in the last place of the strong
one's value, so that a plain FP32 running sum drops all of them. In turn they lie in one multipole
cell, at the window edges beyond the cells (the edge runs), at window edges taken batch by batch (a cutoff
too short for cells) or under masks (shorter still), inside their slow zones, and a few in each of
thousands of cells.

Tolerance: the profile forms' bounds (1.5e-5, see test_gpu_wings.py) plus 128 lines summed plainly
between two compensated additions (at most 128 x 2^-25 of the sum): 2e-5. The weak lines make up
1e-4 to 1e-2 of each value."""
import numpy as np
import pytest

import oracle
from rox_testutil import check_sigma, q_pair, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2510_20870_gb300 as rox  # noqa: E402
import rox_synth as rs  # noqa: E402

TOL = 2e-5
DNU, T, MASS, POINTS = 0.01, 296.0, 18.0, 2_200_001


def _list(strong, weak, rel, at=None):
    """HITRAN lines of equal widths at 296 K (so S = S_ref): the strong one and weak ones of relative
    strength rel -- with `at`, of that value at wavenumber `at` relative to the strong line's there."""
    nu0 = np.concatenate([[strong], weak])
    s = np.full(nu0.size, rel)
    if at is not None:
        s *= ((nu0 - at) / (strong - at)) ** 2
    s[0] = 1.0
    order = np.argsort(nu0, kind="stable")
    n = nu0.size
    f = lambda v: np.full(n, v, np.float32)  # noqa: E731
    return {"convention": 0, "nu0": nu0[order], "s_or_a": (1e-20 * s[order]).astype(np.float32), "g_up": None,
            "e_lower": f(0.0), "gamma_ref": f(0.07), "n_t": f(0.5)}


def _spread(lo, hi, n):
    return lo + (hi - lo) * (np.arange(n) + 0.5) / n


# name: (cutoff, strong line, weak lines, their relative strength, first point compared); the grid is long,
# so that a span is summed in one part and not in up to 128
CASES = {
    # one cell (64 steps from 1009.60), some 9 cm^-1 from the points
    "cell": (25.0, 1009.605, _spread(1009.61, 1010.23, 240_000), 2.5e-8, 0),
    # window edges, beyond the cells' reach: from above and from below
    "edge run above": (25.0, 1025.3, _spread(1025.31, 1025.9, 300_000), 9e-10, 150),
    "edge run below": (25.0, 1004.3, _spread(1003.7, 1004.29, 300_000), 9e-10, 2816),
    # no cells (under two spans), scanned in the general batches
    "edge scan": (5.1, 1006.3, _spread(1006.31, 1006.7, 300_000), 9e-10, 190),
    # too short a cutoff for the scan: masked pairs
    "edge masked": (1.0, 1001.2, _spread(1001.21, 1001.4, 300_000), 1.5e-8, 60),
    # inside the slow zones of all of them
    "zones": (25.0, 1001.2, _spread(1001.205, 1001.235, 300_000), 1.5e-8, 100),
}
REF = {}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("points_in_call", [1, 2])
def test_weak_lines_beside_a_strong_one(name, points_in_call):
    cutoff, strong, weak, rel, j0 = CASES[name]
    _check(name, POINTS, cutoff, _list(strong, weak, rel), j0, points_in_call, 0.5)


def test_weak_cells_beside_a_strong_one():
    """Ten lines a cell in thousands of cells left of a span, each cell's value there 2.9e-8 of that of the
    strong line in the farthest."""
    points, cutoff = 420_001, 2500.0
    j0 = points - 200
    at = 1000.0 + DNU * j0
    weak = _spread(at - 2480.0 + 1.0, at - 100.0, 10 * int(2380 / 0.64))
    L = _list(at - 2480.0, weak, 2.9e-9, at)
    _check("far cells", points, cutoff, L, j0, 1, 0.5)


def _check(name, points, cutoff, L, j0, points_in_call, P):
    grid = (1000.0, DNU, points)
    w = rs.CONFIGS[1]
    Qt, Qr = q_pair(w, T)
    j1 = j0 + 8
    if name not in REF:
        k = int(np.argmax(L["s_or_a"]))
        strong = {n: v[k:k + 1] if isinstance(v, np.ndarray) else v for n, v in L.items()}
        REF[name] = [oracle.xsec_window(lines, grid, j0, j1, P, T, Qt, Qr, MASS, cutoff) for lines in (L, strong)]
    ref, one = REF[name]
    assert np.all(one > 0) and np.all(1.0 - one / ref > 4 * TOL)       # what a plain sum would drop
    ps = [P, 3 * P][:points_in_call]
    ws = torch.empty(rox.rox_xsec_workspace_size(L["nu0"].size, grid, 1), dtype=torch.uint8, device="cuda")
    sigma = torch.empty((len(ps), points), dtype=torch.float32, device="cuda")
    rox.rox_xsec_batch(to_device(L, torch), grid, ps, [T] * len(ps), [Qt] * len(ps), Qr, MASS, cutoff, sigma, ws,
                       flags=rox.ROX_KAHAN)
    assert rox.rox_ws_status(ws)[0] == 0
    got = sigma[0, j0:j1].double().cpu().numpy()
    err = float((np.abs(got - ref) / ref).max())
    print("PARITY dense lists, %s: max rel err %.3e" % (name, err))
    assert err <= TOL, (name, err)


# widest Lorentz half-width in units of 64 half-cells (beyond 1 a cell's moments are not used: the powers of
# the poles would leave FP32's range)
@pytest.mark.parametrize("wide", [0.2, 0.9, 0.999, 1.001, 1.5])
def test_narrow_and_very_wide_lines_in_one_cell(wide):
    """3,000 lines of 3e-4 to 1e-3 of that width, every 50th of the full width, in cells of 0.128 cm^-1; the
    tolerance of test_gpu_wings.py."""
    dnu, points, cutoff = 0.002, 2049, 100.0
    half = 32 * dnu
    rng = np.random.default_rng(7)
    n = 3000
    nu0 = np.sort(rng.uniform(1000.0 - cutoff, 1004.0 + cutoff, n))
    gam = (wide * 64 * half) * np.where(np.arange(n) % 50 == 0, 1.0, rng.uniform(3e-4, 1e-3, n))
    f = lambda v: np.full(n, v, np.float32)  # noqa: E731
    L = {"convention": 0, "nu0": nu0, "s_or_a": np.exp(rng.uniform(np.log(1e-24), np.log(1e-20), n)).astype(np.float32),
         "g_up": None, "e_lower": f(0.0), "gamma_ref": gam.astype(np.float32), "n_t": f(0.5)}
    grid = (1000.0, dnu, points)
    w = rs.CONFIGS[1]
    Qt, Qr = q_pair(w, T)
    ref = oracle.xsec_windowed(L, grid, 1.01325, T, Qt, Qr, MASS, cutoff)
    ws = torch.empty(rox.rox_xsec_workspace_size(n, grid, 1), dtype=torch.uint8, device="cuda")
    sigma = torch.empty((1, points), dtype=torch.float32, device="cuda")
    rox.rox_xsec(to_device(L, torch), grid, 1.01325, T, Qt, Qr, MASS, cutoff, sigma, ws)
    assert rox.rox_ws_status(ws)[0] == 0
    check_sigma(sigma[0].double().cpu().numpy(), ref, rel_tol=1.5e-5, label="wide %g" % wide)
