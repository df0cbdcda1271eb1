"""Calls in a workspace without room for the per-line constants (sized for more temperatures) give the
same cross-sections bit for bit, on a uniform grid and on nodes."""
import numpy as np
import pytest

from rox_testutil import q_pair, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2510_20870_gb300 as rox  # noqa: E402
from test_gpu_parity import _small_lines  # noqa: E402


@pytest.mark.parametrize("on_nodes", [False, True])
@pytest.mark.parametrize("n_temps", [1, 2, 4])
def test_without_room_for_the_constants(on_nodes, n_temps):
    w, L = _small_lines(1, 30000, 2990.0, 3140.0, 23)
    dl, grid, n = to_device(L, torch), (3000.0, 0.01, 12001), 30000
    nodes = torch.from_numpy(3000.0 * np.exp(np.arange(12001) / 3e5)).cuda()
    T = [400.0 + 500.0 * k for k in range(n_temps)]
    P, Q, Qr = [0.1 * 4 ** k for k in range(n_temps)], [q_pair(w, t)[0] for t in T], q_pair(w, 296.0)[1]
    size = (lambda t: rox.rox_xsec_nodes_workspace_size(n, 12001, t)) if on_nodes else (
        lambda t: rox.rox_xsec_workspace_size(n, grid, t))
    out = []
    for sized in (n_temps, 5):
        if sized == 5 and on_nodes:
            assert size(5) < size(4)
        ws = torch.empty(size(sized), dtype=torch.uint8, device="cuda")
        sigma = torch.empty((n_temps, 12001), dtype=torch.float32, device="cuda")
        if on_nodes:
            rox.rox_xsec_nodes_batch(dl, nodes, P, T, Q, Qr, 16.0, 25.0, sigma, ws)
        else:
            rox.rox_xsec_batch(dl, grid, P, T, Q, Qr, 16.0, 25.0, sigma, ws)
        assert rox.rox_ws_status(ws)[0] == 0
        out.append(sigma.cpu().numpy())
    assert np.array_equal(out[0], out[1])
