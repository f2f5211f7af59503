"""The recursion of gg -> t t~ g g g, compiled for the host, against the
per-helicity diagram program on several events, helicity by helicity and flow
by flow (no GPU): the two programs share no currents and no order of sums, so
this is the check of the recursion that does not rest on another recursion.
Tolerance as in test_recursion_host.py (1e-11 of the helicity's largest flow)."""
import numpy as np

from test_recursion_host import _run


def test_flows_of_every_helicity_of_several_events(tmp_path):
    r = _run("g g > t t~ g g g", 2000.0, 6, tmp_path)
    for e in range(6):
        assert sorted(r[e, :, 0].astype(int)) == list(range(128))
        assert np.max(r[e, :, 1]) <= 1e-11
        assert np.max(np.abs(r[e, :, 2] - r[e, :, 3])) <= 1e-11 * r[e, :, 3].sum()
