"""Selection bins and node windows where their short forms hand over to the exact ones: line centres
on the edges of bins (the quotient's product form against the rounded division), lines of equal
strength (every one a candidate for its bin's maximum), and lists in which a block of lines is not
sorted (no bracket for the searches). Everything compared here is a decision: no tolerance."""
import numpy as np
import pytest

import oracle
import rox_synth as rs
from rox_testutil import q_pair, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2510_20870_gb300 as rox  # noqa: E402

GRID, CUT = (2000.0, 0.01, 50001), 25.0


def _mask_and_evals(L, w, rel, bw, T=700.0):
    dl = to_device(L, torch)
    Qt, Qr = q_pair(w, T)
    n = L["nu0"].size
    keep = torch.empty(n, dtype=torch.uint8, device="cuda")
    ws = torch.empty(rox.rox_xsec_select_workspace_size(n, GRID, 1, CUT, rel, bw), dtype=torch.uint8, device="cuda")
    rox.rox_line_select(dl, GRID, CUT, T, Qt, Qr, rel, bw, keep, ws)
    sigma = torch.empty((1, GRID[2]), dtype=torch.float32, device="cuda")
    rox.rox_xsec_select_batch(dl, GRID, [1.0], [T], [Qt], Qr, w.mass_amu, CUT, rel, bw, sigma, ws)
    rc, evals = rox.rox_ws_status(ws)
    assert rc == 0
    S = oracle.line_strength(L, T, Qt, Qr)
    jlo, jhi = oracle.window_indices(L["nu0"], *GRID, CUT)
    return keep.cpu().numpy().astype(bool), evals, S, np.maximum(np.minimum(jhi, GRID[2] - 1) - np.maximum(jlo, 0) + 1, 0)


@pytest.mark.parametrize("bw", [1.0, 0.1, 1.0 / 3.0, 7.3, 1e-3, 1e9])
def test_lines_on_bin_edges(bw):
    w = rs.CONFIGS[1]
    L = oracle.sort_lines(rs.make_lines(w, 0, 20_000))
    origin, nb = oracle.select_bins(GRID, CUT, bw)
    k = np.random.default_rng(5).integers(0, min(nb, int(560 / bw) + 1) + 1, L["nu0"].size)
    edge = origin + k * bw
    step = np.random.default_rng(6).integers(-2, 3, edge.size)
    nu0 = np.where(step == 0, edge, edge + step * np.spacing(edge))
    order = np.argsort(nu0, kind="stable")
    L = {key: np.ascontiguousarray(v[order]) if isinstance(v, np.ndarray) else v for key, v in L.items()}
    L["nu0"] = nu0[order]
    got, evals, S, win = _mask_and_evals(L, w, 0.5, bw)
    ref = oracle.select_mask(L["nu0"], S, 0.5, bw, origin, nb)
    assert np.array_equal(got, ref), int((got != ref).sum())
    assert evals == int(win[ref].sum())


@pytest.mark.parametrize("rel", [0.0, 0.3, 1.0])
def test_equal_strengths(rel):
    w = rs.CONFIGS[1]
    n = 5003
    one = rs.make_lines(w, 0, 1)
    L = {key: np.repeat(v[:1], n) if isinstance(v, np.ndarray) else v for key, v in one.items()}
    L["nu0"] = np.repeat(np.float64(2210.125), n)
    got, evals, S, win = _mask_and_evals(L, w, rel, 1.0)
    assert got.all() and evals == int(win.sum())


def test_unsorted_blocks_of_node_windows():
    nodes = rs.fixed_resolution_grid(1000.0, 5000.0, 100_000)
    rng = np.random.default_rng(8)
    nu0 = np.sort(rng.uniform(900.0, 5100.0, 4000))
    nu0[256:512] = rng.permutation(nu0[256:512])     # one block in disorder
    nu0[700], nu0[900] = nu0[3900], nu0[3]           # single lines out of their block's range
    nu0[1024:1280] = nu0[1024]                       # a block of equal centres
    nu0[1300] = nodes[5000] + CUT                    # cutoff on a node
    nd, d = torch.from_numpy(nodes).cuda(), torch.from_numpy(nu0).cuda()
    jlo = torch.empty(nu0.size, dtype=torch.int32, device="cuda")
    jhi = torch.empty_like(jlo)
    rox.rox_node_windows(d, nd, CUT, jlo, jhi)
    ol, oh = oracle.node_windows(nu0, nodes, CUT)
    assert np.array_equal(jlo.cpu().numpy(), ol) and np.array_equal(jhi.cpu().numpy(), oh)
