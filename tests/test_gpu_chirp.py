"""The chirp transforms of the contraction (k grids uniform in ln k) against the FP64 oracle, at the
sizes where their split into FFT points, halves and passes changes, and the rule that chooses them:
a grid that is uniform to rounding takes them, any other the direct sums, with the same results.  In the mixed form the transforms take the frequencies n >= 64
and the tensor-core GEMM those below.

Gates: those of the FP64 path, 1e-10 (C, P_bar, amp_bar) and 1e-9 (W_bar): the transforms are FP64
FFTs of at most 8192 points, whose rounding errors are below 1e-13 of a row.  Mixed form: its gates,
1e-4 (C) and 5e-5 (gradients)."""
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


def _case(N, k, n_ell, n_knots, curved=True, rank=0):
    """Two density tracers and a lensing one, one of them with its own bias; with few knots the
    growth is curved in ln k, so that every knot carries weight."""
    cosmo = Cosmology()
    chi = CHI_MIN * np.exp(np.arange(N) * np.log(CHI_MAX / CHI_MIN) / N)
    z = cosmo.z_of_chi(chi)
    W = np.array([clustering_window(cosmo, chi, 0.5, 0.2, z), clustering_window(cosmo, chi, 1.1, 0.3, z),
                  lensing_window(cosmo, chi, 0.6, 1.4, 0.0, z)])
    knots = np.geomspace(k[0], k[-1], n_knots) if n_knots > 1 else np.array([0.1])
    lk = np.log(knots / 0.1)
    D = (1.0 / (1.0 + z))[None, :] * (1.0 + 0.02 * lk + (0.003 * lk ** 2 if curved else 0.0))[:, None]
    if curved:
        D = D + 0.002 * np.sin(lk)[:, None] * (z / (1.0 + z))[None, :]
    if rank:
        # growth of that rank in (k, z), for basis mode
        f = [1.0 / (1.0 + z), 0.02 * z / (1.0 + z), 0.01 * np.sin(2.0 * z) * np.exp(-z), 0.01 * np.exp(-2.0 * z)]
        h = [np.ones_like(lk), lk, np.sin(lk), np.cos(0.7 * lk)]
        D = sum(np.outer(h[t], f[t]) for t in range(rank))
    P = power_spectrum(k, 3.5e6)
    kind = np.array([0, 0, 1], dtype=np.int32)
    bias = np.array([-0.3, -0.45, -1.5])
    return Workload("chirp", N, CHI_MIN, CHI_MAX, k, ell_list(2, 900, n_ell), knots, kind, bias, W, D, None, P,
                    np.array([1.3, 0.8, 1.0]))


def _kernels(w, precision, Cb):
    """(C, gradients, names of the kernels that ran)"""
    import paper_2505_22718_gb300 as S
    ctx = lib_context(w)
    p = S.PRECISIONS[precision]
    S.swcl_profile_enable(ctx.ptr, True)
    C = ctx.compute_cl(p)
    g = ctx.vjp(Cb, p)
    names = set(S.swcl_profile_read(ctx.ptr))
    ctx.close()
    return C, g, names


def _errors(w, C, g, Cb):
    gr = O.Grids(w.N, w.chi_min, w.chi_max, w.k, w.ells, w.knots, w.kind, w.fft_bias, fft="numpy")
    f = O.forward(gr, w.W, w.D, w.P, w.amp)
    Pbo, Abo, Wbo, _ = O.vjp(gr, f, Cb, w.W, w.D, w.P, w.amp)
    e = (norm_err(C, f["C"]), pbar_err(g[0][0], Pbo, p_abs(f["delta"], Cb, w.amp, w.k)), grad_err(g[1][0], Abo),
         wbar_err(g[2][0], Wbo))
    print("C %.2e  P_bar %.2e  amp_bar %.2e  W_bar %.2e" % e)
    return e


def _check(w, C, g, Cb, tol, tol_w):
    e = _errors(w, C, g, Cb)
    assert max(e[:3]) < tol and e[3] < tol_w


# (N, N_k, multipoles, knots): both halves and whole windows of every FFT size, the last size that
# fits one (N/2 + N_k - 1 or N/2 + N_k points) and the first of the next, one to four transforms per
# multipole, few and many multipoles
@pytest.mark.parametrize("N,n_k,n_ell,n_knots", [
    (256, 256, 20, 1), (256, 385, 7, 2), (512, 256, 5, 3), (512, 333, 37, 23), (512, 768, 9, 1), (512, 769, 9, 4),
    (2048, 1024, 11, 1), (2048, 1025, 3, 2), (1024, 2500, 4, 3), (4096, 4096, 3, 1), (4096, 6144, 2, 1)])
def test_fp64_sizes_against_oracle(N, n_k, n_ell, n_knots):
    w = _case(N, np.geomspace(1e-4, 8.0, n_k), n_ell, n_knots, curved=n_knots <= 4)
    Cb = np.random.default_rng(3).standard_normal((n_ell, 3, 3))
    C, g, names = _kernels(w, "fp64", Cb)
    # the transforms where they take fewer FP64 operations than the direct sum: about 75 per FFT point
    # and profile row (here one row per knot up to four, one in basis mode) against 2 n_h N_k
    M = 1 << (N // 2 + n_k - 1).bit_length()
    rows = n_knots if n_knots <= 4 else 1
    assert ("chirp fwd fp64" in names) == (75 * rows * M < 2 * (N // 2 + 1) * n_k)
    assert ("chirp adj fp64" in names) == ("chirp fwd fp64" in names) == ("contract fp64" not in names)
    _check(w, C, g, Cb, 1e-10, 1e-9)


@pytest.mark.parametrize("grid", ["geomspace", "logspace", "exp", "wide", "perturbed", "linear", "rounded"])
def test_rule_on_the_k_grid(grid):
    """Grids uniform in ln k to rounding, however they were computed, take the transforms; others the
    direct sums.  Both meet the FP64 gates."""
    n = 400
    k = {"geomspace": np.geomspace(1e-4, 10.0, n), "logspace": np.logspace(-4, 1, n),
         "exp": np.exp(np.linspace(np.log(1e-4), np.log(10.0), n)),
         "wide": np.geomspace(1e-12, 1e6, n), "linear": np.linspace(1e-4, 10.0, n),
         "perturbed": np.geomspace(1e-4, 10.0, n) * (1.0 + 1e-12 * np.cos(np.arange(n))),
         "rounded": np.array([float("%.7g" % x) for x in np.geomspace(1e-4, 10.0, n)])}[grid]
    w = _case(512, k, 9, 1)
    Cb = np.random.default_rng(4).standard_normal((9, 3, 3))
    C, g, names = _kernels(w, "fp64", Cb)
    assert ("chirp fwd fp64" in names) == (grid in ("geomspace", "logspace", "exp", "wide"))
    _check(w, C, g, Cb, 1e-10, 1e-9)


# (N, N_k, multipoles, rank of the growth): the smallest N, both halves and whole windows, the last size
# that fits an FFT forward (N/2 - 63 + N_k - 1 points) and transposed, one to four transforms per
# multipole, more multipoles than one CTA sums (16)
@pytest.mark.parametrize("N,n_k,n_ell,rank", [
    (1024, 200, 37, 1), (1024, 576, 18, 2), (1024, 512, 17, 3), (2048, 1024, 33, 1), (2048, 1088, 5, 4),
    (2048, 2500, 9, 2), (4096, 2049, 3, 1), (4096, 6144, 2, 1)])
def test_mixed_sizes_against_oracle(N, n_k, n_ell, rank):
    w = _case(N, np.geomspace(1e-4, 8.0, n_k), n_ell, 24, rank=rank)
    Cb = np.random.default_rng(5).standard_normal((n_ell, 3, 3))
    C, g, names = _kernels(w, "bf16x9", Cb)
    assert {"chirp fwd f32", "chirp adj f32"} <= names and "basis gemm adj" not in names
    _check(w, C, g, Cb, 1e-4, 5e-5)


@pytest.mark.parametrize("N", [512, 1024])
@pytest.mark.parametrize("n_walk", [1, 3])
def test_mixed_ragged_walkers_against_the_gemms(n_walk, N, monkeypatch):
    """Lists of 1, 0 and many multipoles per walker; N = 512 keeps the GEMMs over all frequencies.  A
    single multipole's P_bar has no accurate digits where every Delta of that multipole is at its
    FP32 noise (the largest k), by either route: the transforms have to meet the gates or come as near
    to the oracle as the GEMMs over all frequencies do on the same inputs."""
    import paper_2505_22718_gb300 as S
    w = _case(N, np.geomspace(1e-4, 8.0, 333), 21, 24, rank=1)
    rng = np.random.default_rng(6)
    one = (w.W, w.P, w.amp)
    w.W, w.P, w.amp = (np.stack([a * (1.0 + 0.1 * t) for t in range(n_walk)]) for a in one)
    lists = [np.array([3], np.int32), np.array([], np.int32), np.arange(0, 21, 2, dtype=np.int32)][-n_walk:]
    w.ell_lists = lists
    Cb = rng.standard_normal((sum(map(len, lists)), 3, 3))
    found = []
    for gemm in (False, True):
        if gemm:
            monkeypatch.setenv("SWCL_BASIS_GEMM", "1")
        ctx = lib_context(w)
        S.swcl_profile_enable(ctx.ptr, True)
        C = ctx.compute_cl(S.SWCL_SPLIT_BF16)
        g = ctx.vjp(Cb, S.SWCL_SPLIT_BF16)
        assert ("chirp fwd f32" in S.swcl_profile_read(ctx.ptr)) == (N == 1024 and not gemm)
        errs, o = [], 0
        for t, lst in enumerate(lists):
            n = len(lst)
            if n == 0:
                assert not any(a[t].any() for a in g)
                continue
            v = _case(N, w.k, 21, 24, rank=1)
            v.W, v.P, v.amp, v.ells = w.W[t], w.P[t], w.amp[t], w.ells[lst]
            errs += _errors(v, C[o:o + n], [a[t:t + 1] for a in g], Cb[o:o + n])
            o += n
        found.append(errs)
        ctx.close()
    for j, (mine, theirs) in enumerate(zip(*found)):
        assert mine < max((1e-4, 5e-5, 5e-5, 5e-5)[j % 4], 1.5 * theirs)
