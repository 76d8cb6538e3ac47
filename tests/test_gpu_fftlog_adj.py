"""W_bar through the FFTLog adjoint that gives each CTA a share of a row's knots: one, several with a
short last share, the most (16), and all of them, and a tracer whose window is zero (FP64 chirp
transforms write zeros for it).  Against the FP64 oracle with the gates of the FP64 path: the
transforms are FP64 FFTs of N/2 points, and the sums over the knots have at most 30 terms."""
import numpy as np
import pytest

from gpu_helpers import grad_err, lib_context, norm_err, wbar_err
from oracle import fftlog as O
from workloads.n5k_synth import CHI_MAX, CHI_MIN, Cosmology, Workload, clustering_window, ell_list, power_spectrum

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def _case(N, n_k, n_ell, n_knots, nw, seed=1):
    rng = np.random.default_rng(seed)
    cosmo = Cosmology()
    chi = CHI_MIN * np.exp(np.arange(N) * np.log(CHI_MAX / CHI_MIN) / N)
    z = cosmo.z_of_chi(chi)
    W = np.array([clustering_window(cosmo, chi, m, 0.2, z) for m in (0.4, 0.8, 1.2)]) * rng.uniform(0.8, 1.2, (nw, 3, 1))
    k = np.geomspace(1e-3, 5.0, n_k)
    knots = np.geomspace(1e-3, 5.0, n_knots) if n_knots > 1 else np.array([0.1])
    lk = np.log(knots / 0.1)
    D = (1.0 / (1.0 + z))[None, :] * (1.0 + 0.02 * lk + 0.003 * lk ** 2)[:, None]
    P = power_spectrum(k, 3.5e6) * rng.uniform(0.9, 1.1, (nw, 1))
    amp = rng.uniform(1.0, 2.0, (nw, 3))
    Cb = rng.standard_normal((nw * n_ell, 3, 3))
    return Workload("adj", N, CHI_MIN, CHI_MAX, k, ell_list(2, 300, n_ell), knots, np.zeros(3, np.int32),
                    np.full(3, -0.3), W, D, None, P, amp), Cb


def _check(w, Cb, C, g, t, n):
    gr = O.Grids(w.N, w.chi_min, w.chi_max, w.k, w.ells, w.knots, w.kind, w.fft_bias, fft="numpy")
    f = O.forward(gr, w.W[t], w.D, w.P[t], w.amp[t])
    o = slice(t * n, (t + 1) * n)
    Pb, Ab, Wb, _ = O.vjp(gr, f, Cb[o], w.W[t], w.D, w.P[t], w.amp[t])
    live = w.W[t].any(axis=1)
    e = (norm_err(C[o][:, live][:, :, live], f["C"][:, live][:, :, live]), grad_err(g[1][t][live], Ab[live]),
         wbar_err(g[2][t], Wb))
    print("walker %d: C %.2e  amp_bar %.2e  W_bar %.2e" % ((t,) + e))
    assert e[0] < 1e-10 and e[1] < 1e-10 and e[2] < 1e-9
    assert not C[o][:, ~live].any() and not g[1][t][~live].any()


# walkers x 3 rows x knots over 8 x 152 gives the knots per CTA
@pytest.mark.parametrize("N,n_knots,nw,per_cta", [(256, 30, 1, 1), (512, 30, 35, 2), (256, 24, 100, 5),
                                                  (64, 20, 330, 16), (64, 3, 410, 3), (128, 1, 20, 1)])
def test_knot_shares_against_oracle(N, n_knots, nw, per_cta, monkeypatch):
    import paper_2505_22718_gb300 as S
    assert per_cta == max(1, min(3 * nw * n_knots // (8 * 152), n_knots, 16))
    monkeypatch.setenv("SWCL_PER_KNOT_FFT", "1")
    w, Cb = _case(N, 70, 2, n_knots, nw)
    ctx = lib_context(w)
    C = ctx.compute_cl(S.SWCL_FP64)
    g = ctx.vjp(Cb, S.SWCL_FP64)
    ctx.close()
    for t in sorted({0, nw // 2, nw - 1}):
        _check(w, Cb, C, g, t, 2)


@pytest.mark.parametrize("N,n_k", [(256, 256), (512, 700)])   # half and whole windows of the FFT
def test_zero_windows_against_oracle(N, n_k):
    import paper_2505_22718_gb300 as S
    w, Cb = _case(N, n_k, 5, 1, 2)
    w.W[0, 1] = 0.0
    ctx = lib_context(w)
    S.swcl_profile_enable(ctx.ptr, True)
    C = ctx.compute_cl(S.SWCL_FP64)
    g = ctx.vjp(Cb, S.SWCL_FP64)
    assert "chirp fwd fp64" in S.swcl_profile_read(ctx.ptr)
    ctx.close()
    for t in range(2):
        _check(w, Cb, C, g, t, 5)
