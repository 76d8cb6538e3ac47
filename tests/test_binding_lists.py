"""Multipole lists set through Context outlive new windows and power spectra for the same number of points,
as they do in the library: the size of the outputs stays that of the lists.  The library's functions are
replaced, so this runs on CPU."""
import numpy as np

from paper_2505_22718_gb300 import api


def test_lists_outlive_new_inputs(monkeypatch):
    for f in ("swcl_create", "swcl_set_grids", "swcl_set_tracers", "swcl_set_windows", "swcl_set_power",
              "swcl_set_ell_lists", "swcl_destroy"):
        monkeypatch.setattr(api, f, lambda *a, **k: 1)
    sizes = []
    monkeypatch.setattr(api, "swcl_compute_cl", lambda ptr, precision, out: sizes.append(out.shape))
    c = api.Context()
    c.set_grids(1.0, 1e5, 64, np.ones(10), np.arange(2, 7), np.ones(1))
    c.set_tracers([0, 0], [-0.3, -0.3])
    W, P, A = np.zeros((3, 2, 64)), np.zeros((3, 10)), np.zeros((3, 2))
    c.set_windows(W)
    c.set_power(P, A)
    c.compute_cl()
    c.set_ell_lists([np.arange(5), np.arange(2), np.arange(0)])
    c.compute_cl()
    c.set_power(P, A)
    c.compute_cl()
    c.set_windows(W)
    c.compute_cl()
    c.set_ell_lists(None)
    c.compute_cl()
    c.set_ell_lists([np.arange(5), np.arange(2), np.arange(0)])
    c.set_grids(1.0, 1e5, 64, np.ones(10), np.arange(2, 6), np.ones(1))   # drops the lists
    c.set_windows(W)
    c.compute_cl()
    assert sizes == [(15, 2, 2), (7, 2, 2), (7, 2, 2), (7, 2, 2), (15, 2, 2), (12, 2, 2)]
