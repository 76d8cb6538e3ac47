"""The FP64 k-quadrature with Delta u staged beside Delta (up to 55 tracers) and without, and amp_bar with
few and with many terms per tracer, against the FP64 oracle with the gates of the FP64 path."""
import numpy as np
import pytest

from gpu_helpers import grad_err, lib_context, norm_err
from oracle import fftlog as O
from workloads.n5k_synth import CHI_MAX, CHI_MIN, Cosmology, Workload, clustering_window, ell_list, power_spectrum

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


# 253 and 276 pairs: one and two turns of 256 threads; 256 and 257 k points: one and two chunks
@pytest.mark.parametrize("n_tr,n_ell,n_k", [(2, 4, 257), (22, 3, 256), (23, 3, 257), (55, 3, 70), (56, 80, 70), (64, 2, 300)])
def test_quadrature_against_oracle(n_tr, n_ell, n_k):
    import paper_2505_22718_gb300 as S
    N = 128
    rng = np.random.default_rng(n_tr)
    cosmo = Cosmology()
    chi = CHI_MIN * np.exp(np.arange(N) * np.log(CHI_MAX / CHI_MIN) / N)
    z = cosmo.z_of_chi(chi)
    W = np.array([clustering_window(cosmo, chi, m, 0.25, z) for m in np.linspace(0.4, 1.4, n_tr)])
    k = np.geomspace(1e-3, 5.0, n_k)
    w = Workload("quad", N, CHI_MIN, CHI_MAX, k, ell_list(2, 300, n_ell), np.array([0.1]), np.zeros(n_tr, np.int32),
                 np.full(n_tr, -0.3), W, (1.0 / (1.0 + z))[None, :], None, power_spectrum(k, 3.5e6),
                 rng.uniform(1.0, 2.0, n_tr))
    Cb = rng.standard_normal((n_ell, n_tr, n_tr))
    ctx = lib_context(w)
    C = ctx.compute_cl(S.SWCL_FP64)
    g = ctx.vjp(Cb, S.SWCL_FP64)
    ctx.close()
    gr = O.Grids(w.N, w.chi_min, w.chi_max, w.k, w.ells, w.knots, w.kind, w.fft_bias, fft="numpy")
    f = O.forward(gr, w.W, w.D, w.P, w.amp)
    _, Ab, _, _ = O.vjp(gr, f, Cb, w.W, w.D, w.P, w.amp)
    e = norm_err(C, f["C"]), grad_err(g[1][0], Ab)
    print("C %.2e  amp_bar %.2e" % e)
    assert max(e) < 1e-10
    assert np.array_equal(C, np.swapaxes(C, 1, 2))
