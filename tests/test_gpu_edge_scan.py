"""Window edges inside a span where the kernel changes over between masked pairs and the scan of running
sums: clusters of 15, 16, 17 and 33 lines whose windows end in one span, from below and from above, in
lists of a span's length around the 128 lines from which it is put in order. Against the FP64 oracle at
the tolerance of test_gpu_wings.py (1.5e-5), on a uniform grid and on nodes."""
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

TOL, DNU, LO, POINTS = 1.5e-5, 0.01, 3000.0, 2561


def _list(cluster, spread, cutoff):
    """`spread` lines evenly over the grid and its reach, and clusters whose windows end at and about the
    centre of the fifth span, to its right (lines below) and to its left (lines above)."""
    centre = LO + DNU * (4 * 256 + 128)
    rng = np.random.default_rng(cluster + spread)
    near = rng.uniform(-0.25, 0.25, cluster)
    nu0 = np.concatenate([centre - cutoff + near, centre + cutoff + near,
                          np.linspace(LO - cutoff, LO + DNU * POINTS + cutoff, spread)])
    w, L = _small_lines(1, nu0.size, LO - 10.0, LO + 40.0, 5)
    L["nu0"] = np.sort(nu0)
    return w, L


@pytest.mark.parametrize("cluster", [0, 15, 16, 17, 33])
@pytest.mark.parametrize("spread", [40, 340, 360, 2000])      # some 15, 126, 132 and 720 lines a span
def test_edges_on_both_sides_of_the_scan(cluster, spread):
    cutoff, T, P = 5.1, 800.0, 0.3
    w, L = _list(cluster, spread, cutoff)
    Qt, Qr = q_pair(w, T)
    grid = (LO, DNU, POINTS)
    ref = oracle.xsec_windowed(L, grid, P, T, Qt, Qr, 16.0, cutoff)
    dl = to_device(L, torch)
    sig, evals = _run_xsec(dl, grid, [(P, T, Qt)], Qr, 16.0, cutoff, flags=rox.ROX_KAHAN)
    check_sigma(sig[0], ref, rel_tol=TOL, label="%d + %d lines" % (cluster, spread))
    assert evals == oracle.count_evals(L["nu0"], *grid, cutoff)
    nodes = LO + DNU * np.arange(POINTS)
    ws = torch.empty(rox.rox_xsec_nodes_workspace_size(L["nu0"].size, POINTS, 1), dtype=torch.uint8, device="cuda")
    out = torch.empty((1, POINTS), dtype=torch.float32, device="cuda")
    rox.rox_xsec_nodes_batch(dl, torch.from_numpy(nodes).cuda(), [P], [T], [Qt], Qr, 16.0, cutoff, out, ws,
                             flags=rox.ROX_KAHAN)
    assert rox.rox_ws_status(ws)[0] == 0
    ref = oracle.xsec_nodes(L, nodes, P, T, Qt, Qr, 16.0, cutoff)
    check_sigma(out[0].double().cpu().numpy(), ref, rel_tol=TOL, label="nodes, %d + %d lines" % (cluster, spread))
