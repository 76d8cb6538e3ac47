"""Ragged multipole lists of the mixed form, with lists of one, no and many multipoles, through the chirp
transforms (N = 1024) and through the GEMMs over all frequencies (N = 512 and SWCL_BASIS_GEMM=1): each
route by itself within the absolute gates of the form against the FP64 oracle, 1e-4 (C) and 5e-5
(gradients).  P_bar of a single multipole has no gate: where every Delta of that multipole is at its FP32
noise (the largest k) it has no accurate digits by either route."""
import numpy as np
import pytest

from gpu_helpers import grad_err, lib_context, norm_err, p_abs, pbar_err, wbar_err
from oracle import fftlog as O
from test_gpu_chirp import _case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("N,gemm", [(512, False), (1024, False), (1024, True)])
@pytest.mark.parametrize("n_walk", [1, 3])
def test_lists_within_absolute_gates(n_walk, N, gemm, monkeypatch):
    import paper_2505_22718_gb300 as S
    if gemm:
        monkeypatch.setenv("SWCL_BASIS_GEMM", "1")
    w = _case(N, np.geomspace(1e-4, 8.0, 333), 21, 24, rank=1)
    w.W, w.P, w.amp = (np.stack([a * (1.0 + 0.1 * t) for t in range(n_walk)]) for a in (w.W, w.P, w.amp))
    lists = [np.array([3], np.int32), np.array([], np.int32), np.arange(0, 21, 2, dtype=np.int32)][-n_walk:]
    w.ell_lists = lists
    Cb = np.random.default_rng(6).standard_normal((sum(map(len, lists)), 3, 3))
    ctx = lib_context(w)
    S.swcl_profile_enable(ctx.ptr, True)
    C = ctx.compute_cl(S.SWCL_SPLIT_BF16)
    g = ctx.vjp(Cb, S.SWCL_SPLIT_BF16)
    assert ("chirp fwd f32" in S.swcl_profile_read(ctx.ptr)) == (N == 1024 and not gemm)
    ctx.close()
    o = 0
    for t, lst in enumerate(lists):
        n = len(lst)
        if n == 0:
            assert not any(a[t].any() for a in g)
            continue
        gr = O.Grids(w.N, w.chi_min, w.chi_max, w.k, w.ells[lst], w.knots, w.kind, w.fft_bias, fft="numpy")
        f = O.forward(gr, w.W[t], w.D, w.P[t], w.amp[t])
        Pb, Ab, Wb, _ = O.vjp(gr, f, Cb[o:o + n], w.W[t], w.D, w.P[t], w.amp[t])
        e = (norm_err(C[o:o + n], f["C"]), grad_err(g[1][t], Ab), wbar_err(g[2][t], Wb),
             pbar_err(g[0][t], Pb, p_abs(f["delta"], Cb[o:o + n], w.amp[t], w.k)))
        print("walker %d: C %.2e  amp_bar %.2e  W_bar %.2e  P_bar %.2e" % ((t,) + e))
        assert e[0] < 1e-4 and max(e[1:3]) < 5e-5
        assert n == 1 or e[3] < 5e-5
        o += n
