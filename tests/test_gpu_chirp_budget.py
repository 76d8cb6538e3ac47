"""The chirp transforms in a context with a memory budget: what happens when their tables or partial
sums do not fit.  Budgets are found by bisection on fresh contexts, so that they lie within 4 KB of
where a call begins to fit, whatever the sizes of the buffers are."""
import numpy as np
import pytest

from gpu_helpers import lib_context, max_rel
from workloads.n5k_synth import CHI_MAX, CHI_MIN, Cosmology, Workload, clustering_window, ell_list, power_spectrum

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def _case(N, n_k, n_ell, n_tr=3, n_walk=1, seed=2):
    rng = np.random.default_rng(seed)
    cosmo = Cosmology()
    chi = CHI_MIN * np.exp(np.arange(N) * np.log(CHI_MAX / CHI_MIN) / N)
    z = cosmo.z_of_chi(chi)
    W = np.array([clustering_window(cosmo, chi, m, 0.2, z) for m in np.linspace(0.4, 1.2, n_tr)])
    W = W * rng.uniform(0.8, 1.2, (n_walk, n_tr, 1))
    k = np.geomspace(1e-4, 8.0, n_k)
    knots = np.geomspace(1e-4, 8.0, 12)
    D = (1.0 / (1.0 + z))[None, :] * (1.0 + 0.02 * np.log(knots / 0.1))[:, None]
    P = power_spectrum(k, 3.5e6) * rng.uniform(0.9, 1.1, (n_walk, 1))
    w = Workload("budget", N, CHI_MIN, CHI_MAX, k, ell_list(2, 900, n_ell), knots, np.zeros(n_tr, np.int32),
                 np.full(n_tr, -0.3), W, D, None, P, rng.uniform(1.0, 2.0, (n_walk, n_tr)))
    return w, rng


class _Step:
    """swcl_compute_batched (a captured graph) into its own device arrays."""

    def __init__(self, w, seed=4):
        import torch
        n_walk, n_tr, _ = w.W.shape
        self.Cb = torch.tensor(np.random.default_rng(seed).standard_normal((n_walk * len(w.ells), n_tr, n_tr)), device="cuda")
        self.out = [torch.zeros_like(self.Cb)] + [torch.zeros(a.shape, dtype=torch.float64, device="cuda")
                                                  for a in (w.P, w.amp, w.W)]

    def __call__(self, ctx, precision):
        import paper_2505_22718_gb300 as S
        for t in self.out:
            t.zero_()
        import torch
        torch.cuda.synchronize()
        S.swcl_compute_batched(ctx.ptr, precision, self.out[0], self.Cb, *self.out[1:])
        ctx.sync()
        return [t.cpu().numpy() for t in self.out]


def _over_budget(call):
    """Whether call() was refused for the memory budget (any other error is raised)."""
    import paper_2505_22718_gb300 as S
    try:
        call()
    except S.SwiftClError as e:
        assert "budget" in str(e)
        return True
    return False


def _context(w, budget):
    """A context, or None where its inputs and tables alone exceed the budget."""
    got = []
    return None if _over_budget(lambda: got.append(lib_context(w, budget=budget))) else got[0]


def _smallest_budget(fits, hi):
    """The smallest budget, to 4 KB, for which fits(budget) holds (it holds for hi)."""
    assert fits(hi)
    lo = 0
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        if fits(mid):
            hi = mid
        else:
            lo = mid
    return hi


def _routes(ctx, call):
    """Names of the kernels that call() runs (outside a graph)."""
    import paper_2505_22718_gb300 as S
    S.swcl_profile_enable(ctx.ptr, True)
    S.swcl_profile_reset(ctx.ptr)
    call()
    names = set(S.swcl_profile_read(ctx.ptr))
    S.swcl_profile_enable(ctx.ptr, False)
    return names


def _same(a, b, tol):
    for x, y in zip(a, b):
        assert max_rel(x, y) < tol


def test_graph_after_the_tables_were_freed():
    """A batched FP64 step captured with the chirp transforms; then a forward-mode call that fits the
    budget only without their tables (they are freed), or does not fit at all; then the step
    again: it must not replay the graph that holds the freed addresses.  FP64 results by either route
    agree to 1e-10 (the gate of the FP64 path)."""
    import paper_2505_22718_gb300 as S
    w, rng = _case(512, 400, 40)
    step, W_dot = _Step(w), rng.standard_normal((8,) + w.W.shape[1:]) * w.W[0]
    free = lib_context(w)
    want = step(free, S.SWCL_FP64)
    J = free.jvp(W_dot=W_dot)
    most = free.query(S.SWCL_Q_WORKSPACE_BYTES)
    free.close()

    def run(budget, check):
        """None (the step does not fit), else whether the JVP fits"""
        ctx = _context(w, budget)
        if ctx is None:
            return None
        try:
            if not check and _over_budget(lambda: step(ctx, S.SWCL_FP64)):
                return None
            if check:
                for _ in range(2):
                    _same(step(ctx, S.SWCL_FP64), want, 1e-10)
            S.swcl_profile_enable(ctx.ptr, True)
            got = []
            fits = not _over_budget(lambda: got.append(ctx.jvp(W_dot=W_dot)))
            names = set(S.swcl_profile_read(ctx.ptr))
            S.swcl_profile_enable(ctx.ptr, False)
            if check:
                if fits:
                    assert max_rel(got[0], J) < 1e-10 and "contract fp64" in names   # the tables were given up
                for _ in range(2):
                    _same(step(ctx, S.SWCL_FP64), want, 1e-10)
                assert ctx.query(S.SWCL_Q_WORKSPACE_BYTES) <= budget
            return fits
        finally:
            ctx.close()

    b = _smallest_budget(lambda x: bool(run(x, False)), most + (64 << 20))
    assert run(b, True) is True
    assert run(b - 65536, True) is False


def test_tables_given_up_for_one_call_only():
    """The same forward-mode call that leaves no room for the tables: the FP64 passes of one point that
    follow have it, and take the transforms again."""
    import paper_2505_22718_gb300 as S
    w, rng = _case(512, 400, 40)
    W_dot = rng.standard_normal((8,) + w.W.shape[1:]) * w.W[0]

    def fits(budget):
        ctx = _context(w, budget)
        if ctx is None:
            return False
        try:
            return not _over_budget(lambda: ctx.jvp(W_dot=W_dot))
        finally:
            ctx.close()

    free = lib_context(w)
    want = free.compute_cl(S.SWCL_FP64)
    free.jvp(W_dot=W_dot)
    most = free.query(S.SWCL_Q_WORKSPACE_BYTES)
    free.close()
    ctx = lib_context(w, budget=_smallest_budget(fits, most + (64 << 20)))
    got = []
    assert "contract fp64" in _routes(ctx, lambda: ctx.jvp(W_dot=W_dot))
    assert "chirp fwd fp64" in _routes(ctx, lambda: got.append(ctx.compute_cl(S.SWCL_FP64)))
    assert max_rel(got[0], want) < 1e-10
    ctx.close()


def test_mixed_step_between_calls_that_do_not_fit():
    """A mixed step under a budget that it just fits.  Calls that find no room there (forward mode along
    eight windows, the FP64 form beside the FP32 tables) leave its route and its results as they were: C,
    P_bar and amp_bar bit for bit; W_bar, whose partial sums are as many as the budget has room for, to the
    1e-5 of the other tests of budgets."""
    import paper_2505_22718_gb300 as S
    w, rng = _case(1024, 400, 40)
    W_dot = rng.standard_normal((8,) + w.W.shape[1:]) * w.W[0]
    step = _Step(w)
    free = lib_context(w)
    want = step(free, S.SWCL_SPLIT_BF16)
    want64 = free.compute_cl(S.SWCL_FP64)
    most = free.query(S.SWCL_Q_WORKSPACE_BYTES)
    free.close()

    def fits(budget):
        ctx = _context(w, budget)
        if ctx is None:
            return False
        try:
            return not _over_budget(lambda: step(ctx, S.SWCL_SPLIT_BF16)) and ctx.query(S.SWCL_Q_RECOMPUTE) == 0
        finally:
            ctx.close()

    def check(got):
        assert all(np.array_equal(a, b) for a, b in zip(got[:3], want)) and max_rel(got[3], want[3]) < 1e-5

    ctx = lib_context(w, budget=_smallest_budget(fits, most + (64 << 20)))
    C = np.empty_like(want[0])
    for _ in range(2):
        check(step(ctx, S.SWCL_SPLIT_BF16))
        assert _over_budget(lambda: ctx.jvp(W_dot=W_dot, precision=S.SWCL_SPLIT_BF16))
        if not _over_budget(lambda: ctx.compute_cl(S.SWCL_FP64, C)):
            assert max_rel(C, want64) < 1e-10
        assert {"basis head", "chirp fwd f32"} <= _routes(ctx, lambda: ctx.compute_cl(S.SWCL_SPLIT_BF16))
    check(step(ctx, S.SWCL_SPLIT_BF16))
    ctx.close()


@pytest.mark.parametrize("prec", ["bf16x9", "fp64"])
def test_partial_sums_that_do_not_all_fit(prec):
    """600 multipoles of two tracers, whose partial sums take more memory than 250 multipoles of Delta and
    Delta bar: just below the budget that holds them all beside 8 multipoles, longer chunks are planned
    with one partial sum per row.  In the mixed form no FP32 sum may cover more than 16 multipoles:
    the transpose then runs in groups, several launches per Delta bar."""
    import paper_2505_22718_gb300 as S
    p = S.PRECISIONS[prec]
    w, rng = _case(1024, 512, 600, n_tr=2)
    Cb = rng.standard_normal((600, 2, 2))
    free = lib_context(w)
    C = free.compute_cl(p)
    P, A, W = free.vjp(Cb, p)
    most = free.query(S.SWCL_Q_WORKSPACE_BYTES)
    free.close()

    def run(budget):
        """(results, chunks of multipoles, launches of the transpose) or None"""
        ctx = _context(w, budget)
        if ctx is None:
            return None
        got = []
        try:
            if _over_budget(lambda: got.append(ctx.compute_cl(p))):
                return None
            S.swcl_profile_enable(ctx.ptr, True)
            if _over_budget(lambda: got.extend(ctx.vjp(Cb, p))):
                return None
            n = S.swcl_profile_read(ctx.ptr)
            assert ctx.query(S.SWCL_Q_WORKSPACE_BYTES) <= budget
            k = "fp64" if prec == "fp64" else "f32"
            return got, n["delta_bar " + k][0], n.get("chirp adj " + k, (0,))[0]
        finally:
            ctx.close()

    least = _smallest_budget(lambda b: run(b) is not None, most + (64 << 20))
    groups = 0
    for b in np.linspace(least, most, 12).astype(int):   # from 8 multipoles to all, one partial sum to all
        got, n_delta, n_adj = run(int(b))
        if prec == "fp64":   # the direct sums at the smallest budgets
            _same(got, (C, P, A, W), 1e-10)
            continue
        assert np.array_equal(got[0], C) and np.array_equal(got[1], P) and np.array_equal(got[2], A)
        assert max_rel(got[3], W) < 1e-5   # as in the other tests of budgets
        groups = max(groups, n_adj - n_delta)
    assert groups > 0 or prec == "fp64"


def test_forward_mode_pays_for_no_transpose():
    """Forward mode of the FP64 form has no transpose: the smallest budget under which its multipoles stay in
    one chunk is what it holds, the cotangent's arrays that every plan counts, and no partial sums
    (44 MB here)."""
    import paper_2505_22718_gb300 as S
    n_ell, n_dir, n_tr, N, n_k = 600, 8, 2, 1024, 512
    w, rng = _case(N, n_k, n_ell, n_tr=n_tr)
    W_dot = rng.standard_normal((n_dir,) + w.W.shape[1:]) * w.W[0]
    free = lib_context(w)
    J = free.jvp(W_dot=W_dot)
    most = free.query(S.SWCL_Q_WORKSPACE_BYTES)
    free.close()

    def run(budget):
        ctx = _context(w, budget)
        if ctx is None:
            return None
        try:
            got = []
            if _over_budget(lambda: got.append(ctx.jvp(W_dot=W_dot))) or ctx.query(S.SWCL_Q_RECOMPUTE):
                return None
            return got[0]
        finally:
            ctx.close()

    b = _smallest_budget(lambda x: run(x) is not None, most + (256 << 20))
    assert np.array_equal(run(b), J)
    nw, n_h = 1 + n_dir, N // 2 + 1
    rows = nw * n_tr
    counted = (8 * rows * n_ell * n_k            # Delta bar
               + 16 * rows * n_h                 # cbar
               + 8 * nw * n_k * n_ell            # the parts of P_bar
               + 3 * 8 * nw * n_ell * n_tr ** 2  # U and the cotangent of every walker, the staging of C
               + 8 * nw * n_ell * 2 * 3          # pair sums of the quadrature, of every walker
               + 8 * (rows * N + nw * n_k + rows))
    assert b < most + counted + (4 << 20)


def test_partial_sums_give_way():
    """A VJP whose partial sums (10 MB) fill the budget, then a call that needs 2 MB more: it has them, and
    the VJP after it works with what is left."""
    import paper_2505_22718_gb300 as S
    w, rng = _case(1024, 512, 600, n_tr=2)
    Cb, X = rng.standard_normal((600, 2, 2)), rng.standard_normal((50, 600, 2, 2))
    modes, noise = np.ones(600), np.full(2, 1e-8)
    free = lib_context(w)
    C = free.compute_cl(S.SWCL_FP64)
    g = free.vjp(Cb, S.SWCL_FP64)
    held = free.query(S.SWCL_Q_WORKSPACE_BYTES)
    F = free.gaussian_fisher(X, modes, noise)
    free.close()
    ctx = lib_context(w, budget=held + (1 << 20))
    for _ in range(2):
        _same([ctx.compute_cl(S.SWCL_FP64)], [C], 1e-10)
        _same(ctx.vjp(Cb, S.SWCL_FP64), g, 1e-10)
        _same([ctx.gaussian_fisher(X, modes, noise)], [F], 1e-9)
    assert ctx.query(S.SWCL_Q_WORKSPACE_BYTES) <= held + (1 << 20)
    ctx.close()
