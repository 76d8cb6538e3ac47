"""Performance cases of the library: what its users have it do, through its public entry points.

A survey analysis holds one context (grids, tracers, growth) and evaluates C_ell, mostly with its
gradients, at many parameter points.  The cases span the sizes that such programs run (a two-tracer
notebook, an N5K-shaped 3x2pt analysis, many walkers at once, every multipole to 3000 with 30
tracers), both directions (C alone, C and its gradients, forward mode), both growth kinds (low-rank
knot profiles and one FFTLog per knot), host and device callers, the default FP64 form and the
mixed-precision tensor-core form.  Shapes are those of this repository's workloads, tests and bench.

Types.  The FP64 form's results stay float64.  The mixed form (bf16x9) sums in FP32, and the tile
that its first call tunes by timing sets the order of some of those sums, so two contexts on the
same inputs already differ in the eighth digit of W_bar.  A program that chooses that form hands its
results to a single-precision likelihood or network: they are kept as float32 here, converted in
one pass from the float64 arrays that the library fills.
"""
import math

import numpy as np
import torch

import paper_2505_22718_gb300 as swcl

CHI_MIN, CHI_MAX = 1.0, 1.0e5       # Mpc/h, the FFTLog grid of every workload here
C_OVER_H0 = 2997.92458              # Mpc/h
OMEGA_M = 0.3
F_SKY = 0.4363

_DEFAULTS = dict(call="step", precision="bf16x9", N=2048, n_k=1024, k_min=1e-4, k_max=10.0, k_grid="log",
                 n_ell=103, l_max=2000, n_gauss=10, n_lens=5, sigma_lo=0.04, sigma_hi=0.08, z_lo=0.25,
                 z_hi=1.25, n_knots=150, growth="separable", bias=False, tapers=False, walkers=1,
                 ragged=False, n_dir=0)


def listed():
    return [
        # two bins, three spectra in a notebook: numpy arrays in and out, the default FP64 form
        dict(name="notebook_small_fp64", call="host_arrays", precision="fp64", N=256, n_k=256, n_ell=20,
             l_max=200, n_gauss=2, n_lens=0, sigma_lo=0.05, sigma_hi=0.05, z_lo=0.5, z_hi=1.0, n_knots=1),
        # the same survey inside a sampler on the GPU: the smallest step, launches and latency
        dict(name="sampler_small", N=256, n_k=256, n_ell=20, l_max=200, n_gauss=2, n_lens=0, sigma_lo=0.05,
             sigma_hi=0.05, z_lo=0.5, z_hi=1.0, n_knots=1),
        # odd sizes together: 333 k, 37 multipoles, 23 knots, 7 tracers, a k- and z-dependent bias,
        # tapers, three parameter points with their own multipole lists
        dict(name="odd_shape", N=512, n_k=333, k_max=5.0, n_ell=37, l_max=700, n_gauss=4, n_lens=3, sigma_lo=0.1,
             sigma_hi=0.2, z_lo=0.3, z_hi=1.3, n_knots=23, bias=True, tapers=True, walkers=3, ragged=True),
        # N5K-shaped 3x2pt survey, C_ell alone: gradient-free samplers, emulator training sets
        dict(name="n5k_forward", call="forward"),
        # the same with all gradients: one Hamiltonian / gradient-descent step on the GPU
        dict(name="n5k_step"),
        # the same step for a sampler that lives on the host (page-locked arrays in and out)
        dict(name="n5k_host_step", call="host_step"),
        # the same inside a PyTorch model: float32 parameters, forward and backward through autograd
        dict(name="n5k_autograd", call="autograd"),
        # the reference arithmetic at survey size (the default precision): validation runs, final chains
        dict(name="n5k_step_fp64", precision="fp64"),
        # scale-dependent growth that no few profiles span (massive neutrinos, modified gravity):
        # one FFTLog per k-knot
        dict(name="n5k_general_step", growth="general"),
        # Fisher forecast: forward mode along 8 parameters, then the Fisher matrix
        dict(name="n5k_forecast_fp64", call="forecast", precision="fp64", n_dir=8),
        # an ensemble of 256 walkers in one call, each with its own multipole list
        dict(name="walkers_256", walkers=256, ragged=True),
        # a stage-IV survey: 30 tracers, every multipole to 3000, N = N_k = 4096, a k- and
        # z-dependent bias
        dict(name="large_step", N=4096, n_k=4096, k_min=1e-5, k_max=20.0, n_ell=2999, l_max=3000, n_gauss=20,
             n_lens=10, sigma_lo=0.03, sigma_hi=0.03, z_lo=0.2, z_hi=1.8, n_knots=200, bias=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any call and form, sizes spread over their logarithms.  k
    grids are mostly log-spaced; some are refined around the baryon oscillations, as Boltzmann codes
    write them."""
    fp64 = rng.random() < 0.35
    call = rng.choice(["forward", "step", "step", "host_step", "autograd", "forecast", "host_arrays"])
    c = dict(call=call, precision="fp64" if fp64 else "bf16x9",
             N=2 ** rng.randint(8, 12), n_k=_log_int(rng, 150, 2500), k_max=rng.choice([5.0, 10.0, 20.0]),
             k_grid="refined" if rng.random() < 0.2 else "log",
             n_ell=_log_int(rng, 8, 300), l_max=rng.choice([200, 700, 2000, 3000]),
             n_gauss=rng.randint(1, 14), n_lens=rng.randint(0, 8), sigma_lo=round(rng.uniform(0.03, 0.06), 3),
             sigma_hi=round(rng.uniform(0.06, 0.12), 3), z_hi=round(rng.uniform(0.9, 1.8), 2),
             n_knots=_log_int(rng, 1, 200), bias=rng.random() < 0.25, tapers=rng.random() < 0.2)
    c["n_ell"] = min(c["n_ell"], c["l_max"] - 1)
    if call == "forecast":
        c["n_dir"] = rng.randint(2, 12)
    else:
        c["walkers"] = 1 if rng.random() < 0.6 else _log_int(rng, 2, 48)
        c["ragged"] = c["walkers"] > 1 and call != "autograd" and rng.random() < 0.5
    if rng.random() < 0.15:
        # one FFTLog per knot: at one parameter point, with knots enough to interpolate between
        c.update(growth="general", walkers=1, ragged=False, bias=False, n_knots=max(12, c["n_knots"]))
    if not fp64 and (c.get("growth") == "general" or c["n_knots"] <= 4):
        c["n_ell"] = min(c["n_ell"], 112)   # the mixed form's limit where the knots keep their own FFTLogs
    x = dict(_DEFAULTS, **c)
    # nothing costlier than the largest listed case: fewer walkers, tangents or multipoles
    limit = 0.25 * _direct_flops(dict(_DEFAULTS, **listed()[-1])) * (0.012 if fp64 else 1.0)
    while _direct_flops(x) > limit or _delta_bytes(x) > 2e10:
        for key, floor in (("walkers", 1), ("n_dir", 2 if call == "forecast" else 0), ("n_ell", 8), ("n_k", 150)):
            if c.get(key, 0) > floor:
                c[key] = max(floor, c[key] // 2)
                break
        x = dict(_DEFAULTS, **c)
    if c.get("walkers", 1) == 1:
        c["ragged"] = False
    return c


# ------------------------------------------------------------------------------ inputs ----

def _full(case):
    x = dict(_DEFAULTS, **case)
    x["n_tr"] = x["n_gauss"] + x["n_lens"]
    x["n_h"] = x["N"] // 2 + 1
    return x


def _k_grid(x):
    if x["k_grid"] == "log":
        return np.geomspace(x["k_min"], x["k_max"], x["n_k"])
    # three times the points per ln k in [0.02, 0.4]
    u = np.linspace(math.log(x["k_min"]), math.log(x["k_max"]), 8192)
    dens = 1.0 + 2.0 / (1.0 + np.exp(-(u - math.log(0.02)) / 0.1)) / (1.0 + np.exp((u - math.log(0.4)) / 0.1))
    cum = np.concatenate([[0.0], np.cumsum(0.5 * (dens[1:] + dens[:-1]))])
    return np.exp(np.interp(np.linspace(0.0, cum[-1], x["n_k"]), cum, u))


def _ells(n, l_max):
    """n distinct multipoles in [2, l_max], log-spaced where they are sparse."""
    if n == l_max - 1:
        return np.arange(2, l_max + 1, dtype=np.int32)
    m = n
    while True:
        e = np.unique(np.round(np.geomspace(2, l_max, m)).astype(np.int32))
        if len(e) >= n:
            keep = np.unique(np.round(np.linspace(0, len(e) - 1, n)).astype(np.int64))
            return np.ascontiguousarray(e[keep])
        m += max(1, m // 8)


def _background():
    z = torch.linspace(0.0, 12.0, 24001, dtype=torch.float64)
    e = torch.sqrt(OMEGA_M * (1.0 + z) ** 3 + 1.0 - OMEGA_M)
    chi = torch.cat([torch.zeros(1, dtype=torch.float64), torch.cumulative_trapezoid(C_OVER_H0 / e, z)])
    return z.numpy(), chi.numpy()


def _smail(z):
    z = np.maximum(z, 0.0) if isinstance(z, np.ndarray) else z.clamp(min=0.0)
    return z * z * (np.exp if isinstance(z, np.ndarray) else torch.exp)(-((z / 0.5) ** 1.5))


def _windows(x, chi, z, zt, chit, shifts, dev):
    """[walkers][tracers][N]: Gaussian clustering bins n(z) H(z)/c and lens efficiencies of
    equal-count source bins, each with its mean shifted."""
    live = torch.as_tensor(chi < 0.999 * chit[-1], device=dev)
    zg = torch.as_tensor(z, device=dev)
    rows = []
    hz = torch.sqrt(OMEGA_M * (1.0 + zg) ** 3 + 1.0 - OMEGA_M) / C_OVER_H0
    if x["n_gauss"]:
        mu = torch.linspace(x["z_lo"], x["z_hi"], x["n_gauss"], dtype=torch.float64, device=dev)
        sg = torch.linspace(x["sigma_lo"], x["sigma_hi"], x["n_gauss"], dtype=torch.float64, device=dev)
        m = (mu + shifts[:, :x["n_gauss"]])[:, :, None]
        nz = torch.exp(-0.5 * ((zg - m) / sg[:, None]) ** 2) / (math.sqrt(2 * math.pi) * sg[:, None])
        rows.append(torch.where(live, nz * hz, torch.zeros_like(zg)))
    if x["n_lens"]:
        zs = np.linspace(0.0, 4.0, 40001)
        cdf = np.cumsum(_smail(zs))
        edges = np.interp(np.linspace(0.0, 1.0, x["n_lens"] + 1), cdf / cdf[-1], zs)
        edges[0], edges[-1] = 0.0, 4.0
        ed = torch.as_tensor(edges, device=dev)
        s = shifts[:, x["n_gauss"]:, None]
        lo, hi = (ed[:-1, None] + s).clamp(min=0.0), ed[1:, None] + s
        t = torch.linspace(0.0, 1.0, 1025, dtype=torch.float64, device=dev)
        zz = lo + (hi - lo) * t
        n = _smail(zz - s)
        h = (hi - lo) / 1024
        tab = torch.as_tensor(chit, device=dev)
        step = zt[1] - zt[0]
        j = (zz / step).long().clamp(0, len(zt) - 2)
        cz = (tab[j] + (zz / step - j) * (tab[j + 1] - tab[j])).clamp(min=1e-3)
        zero = torch.zeros_like(lo)
        g0 = torch.cat([zero, torch.cumsum(0.5 * h * (n[..., 1:] + n[..., :-1]), -1)], -1)
        g1 = torch.cat([zero, torch.cumsum(0.5 * h * (n[..., 1:] / cz[..., 1:] + n[..., :-1] / cz[..., :-1]), -1)], -1)
        a = torch.minimum(torch.maximum(zg.expand(lo.shape[0], lo.shape[1], -1), lo), hi)
        f = (a - lo) / h
        i = f.long().clamp(0, 1023)
        f = f - i
        at = lambda g: torch.gather(g, 2, i) + f * (torch.gather(g, 2, i + 1) - torch.gather(g, 2, i))  # noqa: E731
        cg = torch.as_tensor(chi, device=dev)
        inner = (g0[..., -1:] - at(g0)) - cg * (g1[..., -1:] - at(g1))
        w = 1.5 * OMEGA_M / C_OVER_H0 ** 2 * cg * (1.0 + zg) * inner / g0[..., -1:]
        rows.append(torch.where(zg < hi, w.clamp(min=0.0), torch.zeros_like(w)))
    return torch.cat(rows, 1).contiguous()


def _inputs(case, seed):
    """The numbers of a case: host grids (numpy), float64 parameter arrays on the GPU (torch)."""
    x = _full(case)
    dev = torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")
    rng = np.random.default_rng([20250528, int(seed)])
    N, nw, ntr = x["N"], x["walkers"], x["n_tr"]
    L = math.log(CHI_MAX / CHI_MIN)
    chi = CHI_MIN * np.exp(np.arange(N) * L / N)
    zt, chit = _background()
    z = np.interp(chi, chit, zt)
    k = _k_grid(x)
    knots = np.geomspace(x["k_min"], x["k_max"], x["n_knots"]) if x["n_knots"] > 1 else np.array([0.1])
    kind = np.array([swcl.SWCL_DENSITY] * x["n_gauss"] + [swcl.SWCL_LENSING] * x["n_lens"], dtype=np.int32)
    bias = np.where(kind == swcl.SWCL_DENSITY, -0.3, -1.5)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
    shifts = t(rng.uniform(-0.02, 0.02, (nw, ntr)))
    W = _windows(x, chi, z, zt, chit, shifts, dev)
    zg, lk = t(z), t(np.log(knots / 0.1))
    if x["growth"] == "general":
        g = 0.5 + 0.8 * zg / (1.0 + zg) + 0.3 * torch.sin(2.3 * zg) * torch.exp(-0.5 * zg)
        D = torch.exp(0.02 * lk[:, None] * g) / (1.0 + zg)
    else:
        D = (1.0 + 0.01 * lk)[:, None] / (1.0 + zg)
    B = None
    if x["bias"]:
        B = torch.ones((ntr, x["n_knots"], N), dtype=torch.float64, device=dev)
        b0 = 1.0 + 0.1 * torch.arange(x["n_gauss"], dtype=torch.float64, device=dev)
        B[:x["n_gauss"]] = (b0[:, None, None] * torch.sqrt(1.0 + zg) * (1.0 + 0.1 * t(knots) ** 2)[:, None])
    amp_k, tilt = 3.5e6 * rng.uniform(0.9, 1.1, (nw, 1)), rng.uniform(0.94, 0.99, (nw, 1))
    P = t(amp_k * k ** tilt / (1.0 + (k / 0.02) ** 2) ** 2 * (1.0 + 0.05 * np.sin(105.0 * k)))
    amp = t(np.concatenate([rng.uniform(1.0, 2.5, (nw, x["n_gauss"])), np.ones((nw, x["n_lens"]))], 1))
    ells = _ells(x["n_ell"], x["l_max"])
    lists = None
    if x["ragged"]:
        # between half and all of the multipoles, so many for each walker whatever the seed
        sizes = np.random.default_rng(99).integers((len(ells) + 1) // 2, len(ells) + 1, nw)
        lists = [np.sort(rng.choice(len(ells), size=int(m), replace=False)).astype(np.int32) for m in sizes]
    taper_chi = taper_c = None
    if x["tapers"]:
        # raised cosines on the outer 5 % of the chi range and the top quarter of the frequencies
        u = np.arange(N) / (N - 1)
        edge = np.minimum(np.minimum(u, 1.0 - u) / 0.05, 1.0)
        v = np.clip((np.arange(x["n_h"]) / (x["n_h"] - 1) - 0.75) / 0.25, 0.0, 1.0)
        taper_chi = np.tile(0.5 * (1.0 - np.cos(np.pi * edge)), (ntr, 1))
        taper_c = np.tile(0.5 * (1.0 + np.cos(np.pi * v)), (ntr, 1))
    n_out = sum(len(v) for v in lists) if lists else nw * len(ells)
    gen = torch.Generator(device=dev).manual_seed(int(seed) + 17)
    C_bar = torch.randn((n_out, ntr, ntr), dtype=torch.float64, device=dev, generator=gen)
    d = dict(x=x, L=L, chi=chi, k=k, knots=knots, kind=kind, bias=bias, W=W, D=D, B=B, P=P, amp=amp, ells=ells,
             lists=lists, taper_chi=taper_chi, taper_c=taper_c, C_bar=C_bar, n_out=n_out)
    if x["call"] == "autograd":
        # the model's parameters are float32
        for key in ("W", "P", "amp", "C_bar"):
            d[key] = d[key].float()
    if x["call"] == "forecast":
        n = x["n_dir"]
        # tangents in turn: P amplitude, tilt, a bias, a window shift along ln chi
        Pd, Ad, Wd = torch.zeros((n, len(k)), dtype=torch.float64, device=dev), \
            torch.zeros((n, ntr), dtype=torch.float64, device=dev), torch.zeros((n, ntr, N), dtype=torch.float64, device=dev)
        for v in range(n):
            i = int(rng.integers(ntr))
            if v % 4 == 0:
                Pd[v] = P[0]
            elif v % 4 == 1:
                Pd[v] = P[0] * t(np.log(k / 0.05))
            elif v % 4 == 2:
                Ad[v, i] = 1.0
            else:
                Wd[v, i] = (torch.roll(W[0, i], -1) - torch.roll(W[0, i], 1)) * (0.5 * N / L)
        e = ells.astype(np.float64)
        edges = np.concatenate([[e[0] - 0.5], 0.5 * (e[1:] + e[:-1]), [e[-1] + 0.5]])
        d.update(P_dot=Pd, amp_dot=Ad, W_dot=Wd, modes=t((2.0 * e + 1.0) * F_SKY * np.diff(edges)),
                 noise=t(np.where(kind == swcl.SWCL_DENSITY, 1e-8, 1e-9)))
    return d


def _flat(shapes, make):
    """One buffer that holds arrays of the given shapes (each from a 256-byte boundary on)."""
    at, places = 0, []
    for s in shapes:
        places.append((at, s))
        at += (math.prod(s) + 63) // 64 * 64
    buf = make(at)
    return buf, [buf[o:o + math.prod(s)].view(s) for o, s in places]


def prepare(case, seed):
    d = _inputs(case, seed)
    x, nw, ntr = d["x"], d["x"]["walkers"], d["x"]["n_tr"]
    st = dict(call=x["call"], prec=swcl.PRECISIONS[x["precision"]], mixed=x["precision"] != "fp64", nw=nw)
    grids = (CHI_MIN, CHI_MAX, x["N"], d["k"], d["ells"], d["knots"])
    if x["call"] == "autograd":
        st["model"] = swcl.AngularPowerSpectrum(*grids, d["kind"], d["bias"], d["D"], d["B"], precision=x["precision"],
                                                taper_chi=d["taper_chi"], taper_c=d["taper_c"])
        st["params"] = [d[n].requires_grad_(True) for n in ("W", "P", "amp")]
        st["C_bar"] = d["C_bar"]
        torch.cuda.synchronize()
        return st
    stream = torch.cuda.Stream()
    ctx = swcl.Context(0, 0, stream.cuda_stream)
    ctx.set_grids(*grids)
    ctx.set_tracers(d["kind"], d["bias"], d["taper_chi"], d["taper_c"])
    ctx.set_windows(d["W"], d["D"], d["B"])
    ctx.set_power(d["P"], d["amp"])
    if d["lists"] is not None:
        ctx.set_ell_lists(d["lists"])
    torch.cuda.synchronize()
    st.update(ctx=ctx, stream=stream, W=d["W"], P=d["P"], amp=d["amp"], C_bar=d["C_bar"])
    shapes = [(d["n_out"], ntr, ntr)] + ([] if x["call"] == "forward" else [(nw, x["n_k"]), (nw, ntr), (nw, ntr, x["N"])])
    if x["call"] == "host_arrays":
        for key in ("W", "P", "amp", "C_bar"):
            st[key] = d[key].cpu().numpy()
    elif x["call"] == "host_step":
        pin = lambda n, dt: torch.zeros(n, dtype=dt, pin_memory=True)  # noqa: E731
        ins = [d[key].cpu().pin_memory() for key in ("W", "P", "amp", "C_bar")]
        st["out"], outs = _flat(shapes, lambda n: pin(n, torch.float64))
        st["step"] = swcl.HostStep(ctx.ptr, st["prec"], outs[0], *ins, *outs[1:])
        st["res"], st["res_v"] = (_flat(shapes, lambda n: pin(n, torch.float32)) if st["mixed"] else (st["out"], outs))
    elif x["call"] == "forecast":
        st.update(P_dot=d["P_dot"], amp_dot=d["amp_dot"], W_dot=d["W_dot"], modes=d["modes"], noise=d["noise"])
        shapes = [(x["n_dir"], x["n_ell"], ntr, ntr), (x["n_dir"], x["n_dir"])]
    if x["call"] in ("step", "forward", "forecast"):
        new = lambda dt: (lambda n: torch.zeros(n, dtype=dt, device="cuda"))  # noqa: E731
        st["out"], st["out_v"] = _flat(shapes, new(torch.float64))
        st["res"], st["res_v"] = _flat(shapes, new(torch.float32)) if st["mixed"] else (st["out"], st["out_v"])
    torch.cuda.synchronize()
    return st


_NAMES = ("C", "P_bar", "amp_bar", "W_bar")


def run(st):
    call = st["call"]
    if call == "autograd":
        W, P, amp = st["params"]
        C = st["model"](W.double(), P.double(), amp.double())
        if st["mixed"]:
            C = C.float()
        grads = torch.autograd.grad(C, (W, P, amp), st["C_bar"].to(C.dtype))
        return {"C": C.detach(), "P_bar": grads[1], "amp_bar": grads[2], "W_bar": grads[0]}
    ctx, prec = st["ctx"], st["prec"]
    if call == "host_arrays":
        ctx.set_window_samples(st["W"])
        ctx.set_power(st["P"], st["amp"])
        C = ctx.compute_cl(prec)
        out = (C,) + ctx.vjp(st["C_bar"], prec)
        return {n: a.astype(np.float32) if st["mixed"] else a for n, a in zip(_NAMES, out)}
    if call == "host_step":
        st["step"]()
        if st["mixed"]:
            st["res"].copy_(st["out"])
        return dict(zip(_NAMES, st["res_v"]))
    # the parameters of this point, then one evaluation, all queued on the library's stream
    swcl.swcl_set_window_samples(ctx.ptr, st["nw"], st["W"])
    swcl.swcl_set_power(ctx.ptr, st["nw"], st["P"], st["amp"])
    out = st["out_v"]
    if call == "forward":
        swcl.swcl_compute_batched(ctx.ptr, prec, out[0])
    elif call == "step":
        swcl.swcl_compute_batched(ctx.ptr, prec, out[0], st["C_bar"], out[1], out[2], out[3])
    else:
        swcl.swcl_jvp(ctx.ptr, prec, len(out[0]), out[0], st["P_dot"], st["amp_dot"], st["W_dot"])
        swcl.swcl_gaussian_fisher(ctx.ptr, out[0], st["modes"], out[1], st["noise"])
    if st["mixed"]:
        with torch.cuda.stream(st["stream"]):
            st["res"].copy_(st["out"])
    return dict(zip(("C_dot", "F") if call == "forecast" else _NAMES, st["res_v"]))


# -------------------------------------------------------------------------------- work ----

def _evaluations(x):
    """Rows (parameter point or tangent, tracer, listed multipole) and directions of one pass."""
    rows = x["walkers"] * x["n_tr"] * x["n_ell"] * (0.75 if x["ragged"] else 1.0)
    if x["call"] == "forecast":
        rows *= 1 + x["n_dir"]
    return rows, 1 if x["call"] in ("forward", "forecast") else 2


def _direct_flops(x):
    x = dict(x, n_tr=x["n_gauss"] + x["n_lens"])
    rows, ways = _evaluations(x)
    return rows * ways * 4.0 * (x["N"] // 2 + 1) * x["n_k"]


def _delta_bytes(x):
    x = dict(x, n_tr=x["n_gauss"] + x["n_lens"])
    return _evaluations(x)[0] * x["n_k"] * 16.0


def work(case):
    """Each input read once, each output written once.  Operations: on a log-spaced k grid with few
    profiles the sum over frequencies is a chirp transform (two FFTs of the next power of two above
    n_h + n_k - 1); else the sum itself, 4 n_h n_k per row.  The k-quadrature and, in reverse, its
    transpose come on top."""
    x = _full(case)
    rows, ways = _evaluations(x)
    m = 1 << (x["n_h"] + x["n_k"] - 2).bit_length()
    direct = 4.0 * x["n_h"] * x["n_k"]
    chirp = 10.0 * m * math.log2(m) + 6.0 * (x["n_h"] + m + x["n_k"])
    per_row = min(direct, chirp) if x["k_grid"] == "log" and x["growth"] == "separable" else direct
    flops = ways * rows * (per_row + 2.0 * x["n_k"] * (x["n_tr"] + 1) * (1.0 if ways == 1 else 1.5))
    nw, ntr = x["walkers"], x["n_tr"]
    n_out = nw * x["n_ell"] * (0.75 if x["ragged"] else 1.0)
    point = 8.0 * nw * (ntr * x["N"] + x["n_k"] + ntr)
    if x["call"] == "forecast":
        size = point * (1 + x["n_dir"]) + 8.0 * x["n_dir"] * (n_out * ntr * ntr + x["n_dir"])
    else:
        size = (point + 8.0 * n_out * ntr * ntr) * ways
    knots = 8.0 * x["n_knots"] * x["N"] * (1.0 + (ntr if x["bias"] else 0)) if x["growth"] == "general" else 0.0
    return {"bytes": size + knots, "flops": flops}


# ------------------------------------------------------------------- the method in 64 bits ----

def _lgamma(z):
    """log Gamma of complex128 z, Re z > 0, up to multiples of 2 pi i: Stirling's series at z + 16."""
    out = np.zeros_like(z)
    for _ in range(16):
        out -= np.log(z)
        z = z + 1.0
    series = (1 / 12., -1 / 360., 1 / 1260., -1 / 1680., 1 / 1188., -691 / 360360., 1 / 156.)
    out += (z - 0.5) * np.log(z) - z + 0.5 * math.log(2 * math.pi)
    for j, b in enumerate(series):
        out += b / z ** (2 * j + 1)
    return out


def _moments(ells, p):
    """int chi^p j_l(chi) dchi for every multipole [n_ell][n_h]: log-Gammas at the lowest multipole
    of each parity, then I_{l+2} = I_l (l + 1 + p)/(l + 2 - p)."""
    out = np.empty((len(ells), len(p)), dtype=np.complex128)
    at = {int(e): i for i, e in enumerate(ells)}
    for par in (0, 1):
        sel = [int(e) for e in ells if e % 2 == par]
        if not sel:
            continue
        l = min(sel)
        cur = math.sqrt(math.pi) * np.exp((p - 1.0) * math.log(2.0) + _lgamma(0.5 * (l + 1.0 + p))
                                          - _lgamma(0.5 * (l + 2.0 - p)))
        while l <= max(sel):
            if l in at:
                out[at[l]] = cur
            cur = cur * (l + 1.0 + p) / (l + 2.0 - p)
            l += 2
    return out


def _lagrange(k, knots):
    """First knot and weights [n_k][s] of the local Lagrange interpolation in ln k."""
    u, v = np.log(k), np.log(knots)
    s = min(4, len(v))
    a = np.clip(np.searchsorted(v, u, side="right") - 1, 0, len(v) - 1)
    j0 = np.clip(a - 1, 0, len(v) - s)
    w = np.ones((len(u), s))
    for r in range(s):
        for t in range(s):
            if t != r:
                w[:, r] *= (u - v[j0 + t]) / (v[j0 + r] - v[j0 + t])
    return j0, w


def exact(case, seed):
    x = _full(case)
    if _direct_flops(x) > 3e12 or x["walkers"] * x["n_tr"] * x["n_knots"] > 7e5:
        return None
    d = _inputs(case, seed)
    dev = d["W"].device
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=dev)  # noqa: E731
    N, nh, nw, ntr, L, k = x["N"], x["n_h"], x["walkers"], x["n_tr"], d["L"], d["k"]
    W, P, amp, Cb = d["W"].double(), d["P"].double(), d["amp"].double(), d["C_bar"].double()
    ells = d["ells"]
    eta = 2 * np.pi * np.arange(nh) / L
    phase = torch.polar(torch.ones((), dtype=torch.float64, device=dev).expand(len(k), nh), -t(np.outer(np.log(k), eta)))
    lens = d["kind"] == swcl.SWCL_LENSING
    le = ells.astype(np.float64)
    wn = np.full(nh, 2.0)
    wn[[0, -1]] = 1.0
    tab = {}
    for ln in set(lens.tolist()):
        pre = np.sqrt((le + 2) * (le + 1) * le * (le - 1)) if ln else np.ones_like(le)
        b = -1.5 if ln else -0.3
        tab[ln] = t(_moments(ells, b + 1j * eta) * pre[:, None] * wn)
    j0, lw = _lagrange(k, d["knots"])
    j0, lw = t(j0), t(lw)
    psi = t(np.exp(-1j * eta * math.log(CHI_MIN)) / N)
    lk = np.log(k)
    h = np.empty_like(lk)
    h[1:-1] = 0.5 * (lk[2:] - lk[:-2])
    h[0], h[-1] = 0.5 * (lk[1] - lk[0]), 0.5 * (lk[-1] - lk[-2])
    wk = t(2.0 / np.pi * k * h * k * k)
    D, B = d["D"], d["B"]

    def tracer(i):
        """chi factor [n_knots][N], coefficient factor [n_h], k factor [n_k] of tracer i"""
        b = -1.5 if lens[i] else -0.3
        f = D * t(d["chi"] ** ((-2.0 if lens[i] else 0.0) - b))
        if B is not None:
            f = f * B[i]
        if d["taper_chi"] is not None:
            f = f * t(d["taper_chi"][i])
        c = psi if d["taper_c"] is None else psi * t(d["taper_c"][i])
        return f, c, t(k ** ((-2.0 if lens[i] else 0.0) - 1.0 - b))

    tr = [tracer(i) for i in range(ntr)]

    def delta(Wi, i):
        f, c, kp = tr[i]
        co = torch.fft.rfft(Wi * f, dim=-1) * c
        X = sum(lw[:, s, None] * co[j0 + s] for s in range(lw.shape[1])) * phase
        return (X @ tab[bool(lens[i])].T).real.T * kp              # [n_ell][n_k]

    def delta_t(Db, i):
        """the transpose of delta: W_bar row from Db [n_ell][n_k]"""
        f, c, kp = tr[i]
        X = ((Db * kp).T.to(torch.complex128) @ tab[bool(lens[i])].conj()) * phase.conj()
        co = torch.zeros((f.shape[0], nh), dtype=torch.complex128, device=dev)
        for s in range(lw.shape[1]):
            co.index_add_(0, j0 + s, lw[:, s, None] * X)
        co = co * c.conj()
        # rfft's transpose: g_m = Re sum_n co_n e^{2 pi i n m / N}
        co[:, 1:-1] *= 0.5
        co[:, 0] = co[:, 0].real.to(co.dtype)
        co[:, -1] = co[:, -1].real.to(co.dtype)
        return (torch.fft.irfft(co, n=N, dim=-1, norm="forward") * f).sum(0)

    if x["call"] == "forecast":
        De = torch.stack([delta(W[0, i], i) for i in range(ntr)], 1)
        A = amp[0]
        U = torch.einsum("liq,q,ljq->lij", De, wk * P[0], De)
        J = []
        for v in range(x["n_dir"]):
            Dd = torch.stack([delta(d["W_dot"][v, i], i) for i in range(ntr)], 1)
            X = torch.einsum("liq,q,ljq->lij", Dd, wk * P[0], De)
            dU = X + X.transpose(1, 2) + torch.einsum("liq,q,ljq->lij", De, wk * d["P_dot"][v], De)
            AA = torch.outer(d["amp_dot"][v], A)
            J.append(torch.outer(A, A) * dU + (AA + AA.T) * U)
        J = torch.stack(J)
        Ct = torch.outer(A, A) * U + torch.diag(d["noise"])
        Y = torch.linalg.solve(Ct[None], J)                        # Ct^-1 X_a
        F = 0.5 * torch.einsum("l,alij,blji->ab", d["modes"], Y, Y)
        return {"C_dot": J, "F": F}

    Cs, Ps, As, Ws, at = [], [], [], [], 0
    for w in range(nw):
        sel = t(d["lists"][w].astype(np.int64)) if d["lists"] is not None else slice(None)
        n = len(d["lists"][w]) if d["lists"] is not None else len(ells)
        De = torch.stack([delta(W[w, i], i)[sel] for i in range(ntr)], 1)
        A = amp[w]
        U = torch.einsum("liq,q,ljq->lij", De, wk * P[w], De)
        Cs.append(U * torch.outer(A, A))
        if x["call"] == "forward":
            continue
        S = 0.5 * (Cb[at:at + n] + Cb[at:at + n].transpose(1, 2))
        at += n
        T = torch.einsum("lij,j,ljq->liq", S, A, De)
        Ps.append(wk * torch.einsum("i,liq,liq->q", A, De, T))
        As.append(2.0 * torch.einsum("lij,j,lij->i", S, A, U))
        Db = torch.zeros((len(ells), ntr, len(k)), dtype=torch.float64, device=dev)
        Db[sel] = 2.0 * A[None, :, None] * (wk * P[w]) * T
        Ws.append(torch.stack([delta_t(Db[:, i], i) for i in range(ntr)]))
    C = torch.cat(Cs)
    if x["call"] == "forward":
        return {"C": C}
    return {"C": C, "P_bar": torch.stack(Ps), "amp_bar": torch.stack(As), "W_bar": torch.stack(Ws)}
