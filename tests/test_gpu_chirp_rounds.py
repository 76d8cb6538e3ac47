"""Mixed form with chirp transforms: how many of a row's lowest frequencies stay in the tensor-core
products (64 to 256, from the row's own coefficients, kHeadRest), over windows from wide to narrow.

Accuracy where Delta is far below its largest value: P_bar weighted to the largest k by a bias that grows as
k^2.  Both routes compute the same sums with FP32 rounding errors of the same size, so the norm of
P_bar's error may differ by chance, but not by more than a factor of 2 (with 64 frequencies for every row
it is 4.7 to 5.5 times that of the GEMMs).  Elsewhere the gates of the mixed form against the FP64 oracle,
1e-4 (C) and 5e-5 (gradients).  The gate of C does not hold for every pair of windows as narrow as
sigma_z = 0.01: where two of them cancel to 4e-10 of their own spectra (l = 2500, N = 4096), both routes are off by
1.2e-3 of the gate's scale.  There C has to come as near as the GEMMs do, within the same factor of 2."""
import numpy as np
import pytest

from gpu_helpers import grad_err, lib_context, norm_err, p_abs, pbar_err, wbar_err
from oracle import fftlog as O
from workloads.n5k_synth import (CHI_MAX, CHI_MIN, Cosmology, Workload, clustering_window, ell_list,
                                 lensing_window, power_spectrum)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def _case(N, n_k, k_max, n_ell, sigmas, rank=1, bias=False, n_walk=1, chi_lo=CHI_MIN, chi_hi=CHI_MAX, seed=7):
    rng = np.random.default_rng(seed)
    cosmo = Cosmology()
    chi = chi_lo * np.exp(np.arange(N) * np.log(chi_hi / chi_lo) / N)
    z = cosmo.z_of_chi(chi)
    mu = np.linspace(0.25, 1.8, len(sigmas))
    W = np.array([clustering_window(cosmo, chi, m, s, z) for m, s in zip(mu, sigmas)] +
                 [lensing_window(cosmo, chi, 0.6, 1.4, 0.0, z)])
    W = W * rng.uniform(0.9, 1.1, (n_walk, len(W), 1))
    n_tr = W.shape[1]
    k = np.geomspace(1e-4, k_max, n_k)
    knots = np.geomspace(1e-4, k_max, 24)
    lk = np.log(knots / 0.1)
    f = [1.0 / (1.0 + z), 0.02 * z / (1.0 + z), 0.01 * np.sin(2.0 * z) * np.exp(-z), 0.01 * np.exp(-2.0 * z)]
    h = [np.ones_like(lk), lk, np.sin(lk), np.cos(0.7 * lk)]
    D = sum(np.outer(h[t], f[t]) for t in range(rank))
    B = None
    if bias:
        B = np.ones((n_tr, len(knots), N))
        B[:-1] = (np.sqrt(1.0 + z) * (1.0 + 0.1 * knots[:, None] ** 2))[None]
    kind = np.array([0] * (n_tr - 1) + [1], dtype=np.int32)
    P = power_spectrum(k, 3.5e6) * rng.uniform(0.9, 1.1, (n_walk, 1))
    w = Workload("rounds", N, chi_lo, chi_hi, k, ell_list(2, 2500, n_ell), knots, kind,
                 np.where(kind == 0, -0.3, -1.5), W, D, B, P, rng.uniform(1.0, 2.0, (n_walk, n_tr)))
    return w, rng


# the last two: another range of chi, so that 64 frequencies reach less far in 2 pi n / ln(chi_max/chi_min)
@pytest.mark.parametrize("N,n_k,k_max,chi_lo,chi_hi", [
    (1024, 700, 10.0, CHI_MIN, CHI_MAX), (1024, 512, 20.0, CHI_MIN, CHI_MAX), (2048, 1024, 10.0, CHI_MIN, CHI_MAX),
    (2048, 700, 10.0, 1e-2, 1e6), (1024, 600, 20.0, 10.0, 2e4)])
def test_pbar_at_the_largest_k_against_the_gemms(N, n_k, k_max, chi_lo, chi_hi, monkeypatch):
    import paper_2505_22718_gb300 as S
    w, rng = _case(N, n_k, k_max, 40, [0.03] * 5, bias=True, chi_lo=chi_lo, chi_hi=chi_hi)
    Cb = rng.standard_normal((len(w.ells),) + (w.n_tr,) * 2)

    def pbar(precision):
        ctx = lib_context(w)
        S.swcl_profile_enable(ctx.ptr, True)
        ctx.compute_cl(precision)
        out = ctx.vjp(Cb, precision)[0][0]
        names = set(S.swcl_profile_read(ctx.ptr))
        ctx.close()
        return out, names

    want, _ = pbar(S.SWCL_FP64)
    mine, names = pbar(S.SWCL_SPLIT_BF16)
    assert {"basis head", "chirp fwd f32"} <= names
    monkeypatch.setenv("SWCL_BASIS_GEMM", "1")
    gemm, names = pbar(S.SWCL_SPLIT_BF16)
    assert "basis gemm fwd" in names
    a, b = (np.linalg.norm(x - want) / np.linalg.norm(want) for x in (mine, gemm))
    print("P_bar error %.2e, GEMMs over all frequencies %.2e" % (a, b))
    assert a < 2.0 * b


# wide and narrow windows in one tile of columns, few multipoles (many rows per tile) and many, profile
# ranks that leave columns of a tile unused, k points beside tile edges, lists with an empty one
@pytest.mark.parametrize("N,n_k,n_ell,rank,n_walk,ragged", [
    (1024, 129, 3, 1, 1, False), (1024, 640, 70, 3, 1, False), (2048, 257, 33, 2, 1, False),
    (2048, 300, 1, 4, 3, False), (4096, 200, 9, 1, 1, False), (1024, 333, 21, 1, 4, True), (1024, 200, 12, 3, 3, True)])
def test_rounds_against_oracle(N, n_k, n_ell, rank, n_walk, ragged, monkeypatch):
    import paper_2505_22718_gb300 as S
    w, rng = _case(N, n_k, 8.0, n_ell, [0.02, 0.3, 0.05, 0.01, 0.1, 0.03], rank=rank, n_walk=n_walk)
    every = np.arange(n_ell, dtype=np.int32)
    lists = [every] * n_walk
    if ragged:
        lists = [every, every[:0], every[1::3], every[::2]][:n_walk]
        w.ell_lists = lists
    Cb = rng.standard_normal((sum(map(len, lists)),) + (w.n_tr,) * 2)
    ctx = lib_context(w)
    C = ctx.compute_cl(S.SWCL_SPLIT_BF16)
    g = ctx.vjp(Cb, S.SWCL_SPLIT_BF16)
    ctx.close()
    monkeypatch.setenv("SWCL_BASIS_GEMM", "1")
    ctx = lib_context(w)
    C_gemm = ctx.compute_cl(S.SWCL_SPLIT_BF16)
    ctx.close()
    o = 0
    for t, lst in enumerate(lists):
        n = len(lst)
        if n == 0:
            assert not any(a[t].any() for a in g)
            continue
        gr = O.Grids(w.N, w.chi_min, w.chi_max, w.k, w.ells[lst], w.knots, w.kind, w.fft_bias, fft="numpy")
        f = O.forward(gr, w.W[t], w.D, w.P[t], w.amp[t], w.B)
        Pb, Ab, Wb, _ = O.vjp(gr, f, Cb[o:o + n], w.W[t], w.D, w.P[t], w.amp[t], w.B)
        e = (norm_err(C[o:o + n], f["C"]), pbar_err(g[0][t], Pb, p_abs(f["delta"], Cb[o:o + n], w.amp[t], w.k)),
             grad_err(g[1][t], Ab), wbar_err(g[2][t], Wb))
        print("walker %d: C %.2e  P_bar %.2e  amp_bar %.2e  W_bar %.2e" % ((t,) + e))
        assert e[0] < max(1e-4, 2.0 * norm_err(C_gemm[o:o + n], f["C"])) and max(e[1:]) < 5e-5
        o += n
