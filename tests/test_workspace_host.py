"""Workspace sizes: a workspace that serves more temperatures serves fewer, and the per-line constants
that a call can do without are bounded on nodes. Host only: a call whose workspace is accepted
meets the missing GPU (ROX_ECUDA) where a refused one returns ROX_ENOMEM; the pointers are
placeholders that are never dereferenced."""
import ctypes

import pytest

import paper_2510_20870_gb300._binding as b
from test_abi_host import host_only


def _lines(n):
    return b.RoxLines(nu0=8, s_or_a=8, g_up=None, e_lower=8, gamma_ref=8, n_t=8, n=n, convention=0, width_dtype=0)


def _pts(n):
    v = ctypes.c_double * n
    return v(*[1.0] * n), v(*[300.0 + k for k in range(n)]), v(*[1.0] * n)


@host_only
@pytest.mark.parametrize("n_temps", [1, 2, 3, 4, 5])
def test_more_temperatures_serve_fewer(n_temps):
    n, G, N = 100_000, b.RoxGrid(2000.0, 0.01, 50001), b.RoxNodes(8, 40_000)
    by = ctypes.byref
    P, T, Q = _pts(n_temps)
    for sized in range(n_temps, 21):
        ws = b.lib.rox_xsec_nodes_workspace_size(n, N.n, sized)
        rc = b.lib.rox_xsec_nodes_batch(by(_lines(n)), by(N), n_temps, P, T, Q, 1.0, 18.0, 25.0, 0, 8, 256, ws, None)
        assert rc == b.ROX_ECUDA, (sized, b.lib.rox_last_error())
        ws = b.lib.rox_xsec_workspace_size(n, by(G), sized)
        rc = b.lib.rox_xsec_batch(by(_lines(n)), by(G), n_temps, P, T, Q, 1.0, 18.0, 25.0, 0, 8, 256, ws, None)
        assert rc == b.ROX_ECUDA, (sized, b.lib.rox_last_error())
    few = b.lib.rox_xsec_nodes_workspace_size(n, N.n, 5) - 12 * n * (6 - n_temps)     # no room for one row less
    rc = b.lib.rox_xsec_nodes_batch(by(_lines(n)), by(N), n_temps, P, T, Q, 1.0, 18.0, 25.0, 0, 8, 256, few, None)
    assert rc == b.ROX_ENOMEM


def test_constants_on_nodes_are_bounded():
    """At most 16 GiB of them: 1e9 lines at four temperatures take 64 bytes a line, as before there
    were any, and the size grows with the number of temperatures there."""
    for n in (1_000_000, 100_000_000, 1_000_000_000):
        least = [n * (16 + 12 * t) for t in range(1, 6)]
        size = [b.lib.rox_xsec_nodes_workspace_size(n, 1_000_000, t) for t in range(1, 6)]
        for s, l in zip(size, least):
            assert l < s < l + (16 << 30) + (1 << 28), (n, s, l)
