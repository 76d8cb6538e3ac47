"""The k-quadrature that streams the rows of many walkers and multipoles through a ring of stages
(mixed form, more than 16 tracers, from 304 rows on, where a row's k points are more than one CTA stages
at once) against the form with one CTA per row and chunk, which a single walker takes.

Both sum the same FP32 products; a product carries two roundings, a sum of four at most three more, and
the sums above are compensated, so that either result is within 6 x 2^-24 sum_q u |Delta_i Delta_j| <=
6 x 2^-24 sqrt(U_ii U_jj) of the exact sum: the two differ by at most 7.2e-7 sqrt(C_ii C_jj).  Gate 1e-6."""
import numpy as np
import pytest

from gpu_helpers import lib_context
from workloads.n5k_synth import CHI_MAX, CHI_MIN, Cosmology, Workload, clustering_window, ell_list, power_spectrum

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


# tracers: the first size, one, two and seven parts of up to twenty blocks; k points: just more than a
# chunk, not a multiple of 4, of 64 or of a stage; with lists the rows keep their own CTAs
@pytest.mark.parametrize("n_tr,n_k,n_ell,ragged", [
    (17, 1030, 8, False), (20, 1500, 8, False), (21, 1025, 19, False), (30, 1100, 9, False), (30, 600, 9, True),
    (33, 577, 8, False), (64, 322, 8, False), (4, 1090, 8, True)])
def test_stream_against_one_row_per_cta(n_tr, n_k, n_ell, ragged):
    import paper_2505_22718_gb300 as S
    N, nw = 1024, 39
    rng = np.random.default_rng(n_tr)
    cosmo = Cosmology()
    chi = CHI_MIN * np.exp(np.arange(N) * np.log(CHI_MAX / CHI_MIN) / N)
    z = cosmo.z_of_chi(chi)
    k = np.geomspace(1e-4, 8.0, n_k)
    W0 = np.array([clustering_window(cosmo, chi, m, 0.1, z) for m in np.linspace(0.3, 1.6, n_tr)])
    W = W0 * rng.uniform(0.8, 1.2, (nw, n_tr, 1))
    P = power_spectrum(k, 3.5e6) * rng.uniform(0.9, 1.1, (nw, 1))
    amp = rng.uniform(1.0, 2.0, (nw, n_tr))
    knots = np.geomspace(1e-4, 8.0, 12)
    D = (1.0 / (1.0 + z))[None, :] * (1.0 + 0.02 * np.log(knots / 0.1))[:, None]
    ells = ell_list(2, 800, n_ell)
    every = np.arange(n_ell, dtype=np.int32)
    lists = [np.sort(rng.choice(n_ell, int(rng.integers(0, n_ell + 1)), replace=False)).astype(np.int32) if ragged
             else every for _ in range(nw)]
    lists[nw - 1] = every

    def spectra(sel):
        w = Workload("rows", N, CHI_MIN, CHI_MAX, k, ells, knots, np.zeros(n_tr, np.int32), np.full(n_tr, -0.3),
                     W[sel], D, None, P[sel], amp[sel], None, [lists[t] for t in sel], None)
        ctx = lib_context(w)
        C = ctx.compute_cl(S.SWCL_SPLIT_BF16)
        ctx.close()
        return C

    C = spectra(list(range(nw)))
    at = np.concatenate([[0], np.cumsum([len(v) for v in lists])])
    for t in (0, 1, nw // 2, nw - 1):
        if len(lists[t]) == 0:
            continue
        one, many = spectra([t]), C[at[t]:at[t + 1]]
        dg = np.sqrt(np.einsum("lii->li", one))
        err = np.max(np.abs(many - one) / (dg[:, :, None] * dg[:, None, :]))
        print("walker %d: %.2e" % (t, err))
        assert err < 1e-6
        assert np.array_equal(many, np.swapaxes(many, 1, 2))
