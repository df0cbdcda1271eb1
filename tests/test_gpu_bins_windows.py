"""Selection bins and node windows where their short forms hand over to the exact ones: line centres
on the edges of bins (the quotient's product form against the rounded division), lines of equal
strength (every one a candidate for its bin's maximum), and lists in which a block of lines is not
sorted (no bracket for the searches). Everything compared here is a decision: no tolerance."""
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
    _check_node_windows(rs.fixed_resolution_grid(1000.0, 5000.0, 100_000))


def test_node_windows_with_nodes_within_the_rounding():
    """Hundreds of nodes closer to zero than the rounding of their distance from a line."""
    nodes = np.concatenate([np.arange(1, 400) * 1e-18, np.geomspace(1e-10, 40.0, 500)])
    c = np.concatenate([CUT + np.arange(-3, 4) * np.spacing(CUT), [1e-18, 24.0, 65.0]])
    _compare(np.sort(c), nodes)


def _compare(nu0, nodes):
    nd, d = torch.from_numpy(nodes).cuda(), torch.from_numpy(nu0).cuda()
    jlo = torch.empty(nu0.size, dtype=torch.int32, device="cuda")
    jhi = torch.empty_like(jlo)
    rox.rox_node_windows(d, nd, CUT, jlo, jhi)
    ol, oh = oracle.node_windows(nu0, nodes, CUT)
    assert np.array_equal(jlo.cpu().numpy(), ol) and np.array_equal(jhi.cpu().numpy(), oh)


def _check_node_windows(nodes):
    rng = np.random.default_rng(8)
    nu0 = np.sort(rng.uniform(900.0, 5100.0, 4000))
    nu0[256:512] = rng.permutation(nu0[256:512])     # one block in disorder
    nu0[700], nu0[900] = nu0[3900], nu0[3]           # single lines out of their block's range
    nu0[1024:1280] = nu0[1024]                       # a block of equal centres
    nu0[1300] = nodes[5000] + CUT                    # cutoff on a node
    _compare(nu0, nodes)


@pytest.mark.parametrize("pts", [[(1.0, 400.0)], [(0.1, 300.0), (10.0, 1000.0), (1e-4, 2000.0), (1.0, 3000.0)],
                                 [(1e-4, 300.0), (1.0, 600.0), (1.0, 900.0), (10.0, 1200.0), (0.01, 2500.0)],
                                 [(1e-3, 700.0), (20.0, 700.0)]])
def test_nodes_points_on_both_sides_of_the_record_limit(pts):
    """Constants kept per line and point (each point its own temperature, at most four) or computed per
    span (more temperatures, or two pressures at one), both against the oracle; its usual tolerance."""
    w = rs.CONFIGS[1]
    L = oracle.sort_lines(rs.make_lines(w, 0, 4000))
    L = {key: v[(L["nu0"] > 1980.0) & (L["nu0"] < 2320.0)] if isinstance(v, np.ndarray) else v for key, v in L.items()}
    nodes = rs.fixed_resolution_grid(2000.0, 2300.0, 60_000)
    nd, dl = torch.from_numpy(nodes).cuda(), to_device(L, torch)
    qs = [q_pair(w, T) for _, T in pts]
    n_temps = len(set(T for _, T in pts))
    ws = torch.empty(rox.rox_xsec_nodes_workspace_size(L["nu0"].size, nodes.size, n_temps), dtype=torch.uint8, device="cuda")
    sigma = torch.empty((len(pts), nodes.size), dtype=torch.float32, device="cuda")
    rox.rox_xsec_nodes_batch(dl, nd, [p for p, _ in pts], [t for _, t in pts], [q for q, _ in qs], qs[0][1], w.mass_amu,
                             CUT, sigma, ws)
    assert rox.rox_ws_status(ws)[0] == 0
    got = sigma.double().cpu().numpy()
    for k, (P, T) in enumerate(pts):
        ref = oracle.xsec_nodes(L, nodes, P, T, qs[k][0], qs[k][1], w.mass_amu, CUT)
        check_sigma(got[k], ref, label="nodes point %d of %d" % (k, len(pts)))
