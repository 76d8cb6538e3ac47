"""swcl_vjp after a replayed host step: it takes Delta as that step left it, in multipole chunks under a
memory budget, also when a pass that holds Delta whole (the FP64 form, which needs less beside Delta on k
grids that are not uniform in ln k) ran between the capture and the replay."""
import numpy as np
import pytest

from gpu_helpers import lib_context, max_rel
from workloads.n5k_synth import CHI_MAX, CHI_MIN, Cosmology, Workload, clustering_window, ell_list, power_spectrum

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def test_vjp_after_a_replayed_step_in_chunks():
    import torch
    import paper_2505_22718_gb300 as S
    N, n_k, n_ell, n_tr = 1024, 400, 60, 3
    rng = np.random.default_rng(12)
    cosmo = Cosmology()
    chi = CHI_MIN * np.exp(np.arange(N) * np.log(CHI_MAX / CHI_MIN) / N)
    z = cosmo.z_of_chi(chi)
    W = np.array([clustering_window(cosmo, chi, m, 0.2, z) for m in (0.4, 0.8, 1.2)])[None]
    k = np.geomspace(1e-4, 8.0, n_k) * (1.0 + 1e-4 * np.cos(np.arange(n_k)))
    knots = np.geomspace(1e-4, 8.1, 12)
    D = (1.0 / (1.0 + z))[None, :] * (1.0 + 0.02 * np.log(knots / 0.1))[:, None]
    w = Workload("chunks", N, CHI_MIN, CHI_MAX, k, ell_list(2, 900, n_ell), knots, np.zeros(n_tr, np.int32),
                 np.full(n_tr, -0.3), W, D, None, power_spectrum(k, 3.5e6)[None], np.array([[1.3, 0.8, 1.0]]))
    Cb = rng.standard_normal((n_ell, n_tr, n_tr))

    def run(budget):
        """(VJP after a replayed step, chunks of the mixed pass, of the FP64 pass) or None"""
        ctx = None
        try:
            ctx = lib_context(w, budget=budget)
            pin = lambda a: torch.as_tensor(np.ascontiguousarray(a)).pin_memory()  # noqa: E731
            ins = [pin(a) for a in (w.W, w.P, w.amp, Cb)]
            outs = [pin(np.zeros(s)) for s in (Cb.shape, w.P.shape, w.amp.shape, w.W.shape)]
            step = S.HostStep(ctx.ptr, S.SWCL_SPLIT_BF16, outs[0], *ins, *outs[1:])
            for _ in range(3):   # the first rounds may grow buffers and capture anew
                ctx.compute_cl(S.SWCL_FP64)
                whole64 = ctx.query(S.SWCL_Q_RECOMPUTE) == 0
                step()
                chunked = ctx.query(S.SWCL_Q_RECOMPUTE) == 1
            return ctx.vjp(Cb, S.SWCL_SPLIT_BF16), chunked, whole64, ctx.query(S.SWCL_Q_WORKSPACE_BYTES)
        except S.SwiftClError as e:
            assert "budget" in str(e)
            return None
        finally:
            if ctx is not None:
                ctx.close()

    want, _, _, held = run(0)
    met = 0
    for b in np.linspace(0.3, 1.0, 15) * held:
        got = run(int(b))
        if got is None:
            continue
        met += got[1] and got[2]
        assert np.array_equal(got[0][0], want[0]) and np.array_equal(got[0][1], want[1])
        assert max_rel(got[0][2], want[2]) < 1e-5   # as in the other tests of budgets
    assert met   # some budget holds the FP64 pass whole and the mixed one in chunks
