"""The longest window, N = 8192, with few rows (walkers x tracers x knots): the cluster form of the FFTLog
would need more shared memory than a launch has by default, so that such rows take the form with one CTA
each.  Against the FP64 oracle with the gates of each form."""
import numpy as np
import pytest

from gpu_helpers import grad_err, lib_context, norm_err, p_abs, pbar_err, wbar_err
from oracle import fftlog as O
from workloads.n5k_synth import CHI_MAX, CHI_MIN, Cosmology, Workload, clustering_window, ell_list, power_spectrum

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("prec,n_knots", [("fp64", 1), ("fp64", 3), ("bf16x9", 12)])
def test_longest_window_against_oracle(prec, n_knots):
    import paper_2505_22718_gb300 as S
    N, n_k, n_ell = 8192, 150, 6
    cosmo = Cosmology()
    chi = CHI_MIN * np.exp(np.arange(N) * np.log(CHI_MAX / CHI_MIN) / N)
    z = cosmo.z_of_chi(chi)
    W = np.array([clustering_window(cosmo, chi, m, 0.2, z) for m in (0.4, 0.8, 1.2)])
    k = np.geomspace(1e-3, 5.0, n_k)
    knots = np.geomspace(1e-3, 5.0, n_knots) if n_knots > 1 else np.array([0.1])
    lk = np.log(knots / 0.1)
    D = (1.0 / (1.0 + z))[None, :] * (1.0 + 0.02 * lk)[:, None]
    if n_knots == 3:
        D = D + 0.01 * np.sin(lk)[:, None] * (z / (1.0 + z))[None, :]
    w = Workload("long", N, CHI_MIN, CHI_MAX, k, ell_list(2, 300, n_ell), knots, np.zeros(3, np.int32),
                 np.full(3, -0.3), W, D, None, power_spectrum(k, 3.5e6), np.array([1.3, 0.8, 1.0]))
    Cb = np.random.default_rng(9).standard_normal((n_ell, 3, 3))
    ctx = lib_context(w)
    C = ctx.compute_cl(S.PRECISIONS[prec])
    g = ctx.vjp(Cb, S.PRECISIONS[prec])
    ctx.close()
    gr = O.Grids(w.N, w.chi_min, w.chi_max, w.k, w.ells, w.knots, w.kind, w.fft_bias, fft="numpy")
    f = O.forward(gr, w.W, w.D, w.P, w.amp)
    Pb, Ab, Wb, _ = O.vjp(gr, f, Cb, w.W, w.D, w.P, w.amp)
    e = (norm_err(C, f["C"]), pbar_err(g[0][0], Pb, p_abs(f["delta"], Cb, w.amp, w.k)), grad_err(g[1][0], Ab),
         wbar_err(g[2][0], Wb))
    print("C %.2e  P_bar %.2e  amp_bar %.2e  W_bar %.2e" % e)
    tol = (1e-10, 1e-9) if prec == "fp64" else (1e-4, 5e-5)
    assert e[0] < tol[0] and max(e[1:]) < tol[1]
