"""Timed cases of the implicit radiation / ionization / gas-energy step.

A case is one pass of what a program does with this library through its Python binding or C
entry points: whole implicit steps as an operator-split host runs them (state in, steps, state
out), an adaptive run, the linearisation of a step, the residual norm, and the learned guess's
training and inference.  Sizes and physical set-ups are those of the package's own workload
recipes, tests and benchmark; inputs are drawn on the GPU from the seed alone.
"""
import ctypes
import math

import numpy as np
import torch

import paper_0901_1110_gb300 as rhi

MPC, KPC = 3.0857e24, 3.0857e21
C_LIGHT, K_BOLTZ, M_H, EV = 2.99792458e10, 1.380649e-16, 1.67262192e-24, 1.602176634e-12
SIGMA_SB = 5.670374419e-5
CELL = MPC / 256                       # cell width of the 256^3, 1 Mpc workload
SOURCES_PER_CELL = 64 / 256 ** 3       # and its point-source density
U_E = 1e-16                            # radiation scaling of the source-driven runs
DEV = "cuda"


# ---- the cases -----------------------------------------------------------------------------------

def listed():
    """Twelve or fewer fixed cases, from single small calls to the 256^3 benchmark step."""
    return [
        # convergence measure of a 32^3, 5-unknown residual, called by hosts that own all memory
        dict(name="norm_32", kind="norm", n=5 * 32 ** 3),
        # matter-radiation equilibration (4^3 periodic LTE box, doubling steps): the smallest steps
        dict(name="lte_4", kind="lte", nx=4, ny=4, nz=4, steps=8),
        # the 32^3 hydrogen benchmark with default parameters (lagged D: CG, FP64 multigrid)
        dict(name="uniform_32", kind="uniform", nx=32, ny=32, nz=32, steps=2),
        # adaptive steps of the HII-region test (held temperature, exact matrix, FP32 multigrid)
        dict(name="advance_hii_32", kind="advance", nx=32, ny=32, nz=32, t_over_trec=0.002),
        # a ragged periodic H + He sub-box, mixed precision
        dict(name="ragged_mixed", kind="lognormal", nx=45, ny=52, nz=61, cell=1.0, form="mixed",
             periodic=True, steps=2),
        # the 128^3 plain FP64 configuration (16 sources in 1 Mpc)
        dict(name="plain_128", kind="lognormal", nx=128, ny=128, nz=128, cell=2.0, form="plain",
             periodic=False, steps=2),
        # learned guess + mixed precision at the benchmark's cell size; five steps hold one
        # evaluation of a network whose guess loses to U^n and the four steps that skip it
        dict(name="learned_128", kind="lognormal", nx=128, ny=128, nz=128, cell=1.0,
             form="learned", periodic=False, steps=5),
        # the benchmark's 256^3 workload, mixed precision: the first steps of a run, as it grows harder
        dict(name="mixed_256", kind="lognormal", nx=256, ny=256, nz=256, cell=1.0, form="mixed",
             periodic=False, steps=4),
        # residual, Newton matrix, right-hand side and multigrid hierarchy at a state with
        # ionised regions, as a host that brings its own Krylov method takes them
        dict(name="linearize_128", kind="linearize", nx=128, ny=128, nz=128, form="plain",
             periodic=False),
        # network outputs for the cells of a 128^3 state
        dict(name="mlp_forward_128", kind="mlp_forward", rows=128 ** 3),
        # loss gradient of one validation set
        dict(name="mlp_grad_12k", kind="mlp_grad", rows=12000),
        # minibatch training, the benchmark's batch size
        dict(name="mlp_train_128k", kind="mlp_train", rows=131072, batch=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["norm", "lte", "uniform", "advance", "lognormal", "lognormal", "lognormal",
                       "linearize", "mlp_forward", "mlp_grad", "mlp_train"])
    if kind == "norm":
        return dict(kind=kind, n=_log_int(rng, 1000, 2 ** 25))
    if kind == "lte":
        n = [rng.randint(2, 9) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], steps=rng.randint(3, 10))
    if kind == "uniform":
        n = _log_int(rng, 10, 72)
        return dict(kind=kind, nx=n, ny=max(8, n + rng.randint(-5, 5)),
                    nz=max(8, n + rng.randint(-5, 5)), steps=rng.randint(1, 3))
    if kind == "advance":
        n = rng.randint(14, 40)
        return dict(kind=kind, nx=n, ny=n, nz=n, t_over_trec=round(rng.uniform(0.001, 0.004), 5))
    if kind == "lognormal":
        n = _log_int(rng, 28, 200)
        ext = [max(24, int(n * rng.uniform(0.75, 1.25))) for _ in range(3)]
        if rng.random() < 0.4:                     # extents a multigrid user would choose
            ext = [max(32, 16 * round(e / 16)) for e in ext]
        return dict(kind=kind, nx=ext[0], ny=ext[1], nz=ext[2], cell=rng.choice([1.0, 2.0]),
                    form=rng.choice(["plain", "mixed", "mixed"]), periodic=rng.random() < 0.3,
                    steps=rng.randint(1, 3))
    if kind == "linearize":
        n = _log_int(rng, 24, 150)
        return dict(kind=kind, nx=n, ny=max(16, n + rng.randint(-9, 9)),
                    nz=max(16, n + rng.randint(-9, 9)), form=rng.choice(["plain", "mixed"]),
                    periodic=rng.random() < 0.5)
    if kind == "mlp_forward":
        return dict(kind=kind, rows=_log_int(rng, 500, 2 ** 24))
    if kind == "mlp_grad":
        return dict(kind=kind, rows=_log_int(rng, 64, 100000))
    return dict(kind=kind, rows=_log_int(rng, 3000, 200000), batch=rng.choice([256, 512, 1000, 4096]))


# ---- inputs --------------------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _gaussian_field(shape, gen):
    """Unit-variance Gaussian field with P(k) ~ k^-2 (k = 0 removed)."""
    w = torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64)
    ks = [torch.fft.fftfreq(n, device=DEV, dtype=torch.float64) for n in shape[:2]]
    kx = torch.fft.rfftfreq(shape[2], device=DEV, dtype=torch.float64)
    k2 = ks[0][:, None, None] ** 2 + ks[1][None, :, None] ** 2 + kx[None, None, :] ** 2
    amp = torch.where(k2 > 0, k2.clamp_min(1e-30) ** -0.5, torch.zeros_like(k2))
    g = torch.fft.irfftn(torch.fft.rfftn(w) * amp, s=shape)
    g -= g.mean()
    return g / g.std()


def _energy(T, nH, nHe, nHII, nHeII, nHeIII):
    """Specific energy of an ideal gas (gamma = 5/3) at temperature T."""
    ne = nHII + nHeII + 2.0 * nHeIII
    return 1.5 * K_BOLTZ * T * (nH + nHe + ne) / (M_H * (nH + 4.0 * nHe))


def _solver(case, dx, ns, y_he, u, spectrum, periodic=False, **over):
    p = rhi.rhi_params_default(ns)
    p.y_he, p.theta = y_he, 1.0
    p.u_e, p.u_n, p.u_E = u
    if ns:
        g = rhi.rhi_grey_constants(spectrum[0], spectrum[1], ns)
        for X in range(3):
            p.sk[X], p.pgam[X], p.ph[X] = g["sk"][X], g["pgam"][X], g["ph"][X]
        p.photon_energy = g["eps"]
    for k, v in over.items():
        setattr(p, k, v)
    kind = rhi.RHI_BC_PERIODIC if periodic else rhi.RHI_BC_ZERO_FLUX
    return rhi.Solver(case["nx"], case["ny"], case["nz"], dx, p, bc=(kind,) * 6)


def _form(case):
    """Parameters of the benchmark's forms: exact Newton matrix, FP64 or FP32 multigrid."""
    f = case["form"]
    return dict(limiter_jacobian=2, max_newton=200,
                precond=rhi.RHI_PRECOND_MG_FP64 if f == "plain" else rhi.RHI_PRECOND_MG_FP32,
                guess=rhi.RHI_GUESS_LEARNED if f == "learned" else rhi.RHI_GUESS_PREVIOUS)


def _outputs(s):
    N = s.N
    return [torch.empty(m * N, dtype=torch.float64, device=DEV) for m in (1, 1, s.ns)]


def _sources(case, seed, cell):
    rng = np.random.default_rng(seed + 7919)
    N = case["nx"] * case["ny"] * case["nz"]
    # the recipe's number in its box, whatever the cell width
    nsrc = max(1, round(N * SOURCES_PER_CELL * (2.0 if cell == 2.0 else 1.0)))
    ijk = np.stack([rng.integers(0, case[q], nsrc) for q in ("nx", "ny", "nz")], axis=1)
    return ijk.astype(np.int32), 1e49 * np.exp(rng.standard_normal(nsrc))


def _lognormal(case, seed):
    """Neutral H + He gas of the lognormal recipe: Y = 0.24, mean n_H = 1e-3, 100 K."""
    shape = (case["nz"], case["ny"], case["nx"])
    nH = (1e-3 * torch.exp(_gaussian_field(shape, _generator(seed)) - 0.5)).ravel()
    y_he = 0.24 / (4.0 * 0.76)
    nHe = y_he * nH
    x0 = 1e-4
    fr = torch.full_like(nH, x0), torch.full_like(nH, x0), torch.full_like(nH, 1e-4 * x0)
    return nH, y_he, nHe, fr


def _state(nH, nHe, T, fr, E):
    xHII, fHeII, fHeIII = fr
    e = _energy(T, nH, nHe, xHII * nH, fHeII * nHe, fHeIII * nHe)
    n = torch.stack([nH - xHII * nH, nHe - fHeII * nHe - fHeIII * nHe, fHeII * nHe])
    return E, e, n.ravel().contiguous()


def _weights(rng, mean, scale):
    """He-initialised weights in the library's layout."""
    I, H, O = rhi.RHI_MLP_IN, rhi.RHI_MLP_HID, rhi.RHI_MLP_OUT
    parts = []
    for rows, cols in ((H, I), (H, H), (H, H), (O, H)):
        parts += [rng.standard_normal(rows * cols) * math.sqrt(2.0 / cols),
                  0.1 * rng.standard_normal(rows)]
    return np.concatenate(parts + [mean, scale]).astype(np.float32)


def _no_change_weights(rng):
    """A network that predicts little change of the neutral initial gas."""
    w = _weights(rng, np.zeros(13), np.full(13, 4.0))
    # small hidden-to-output rows, output biases of the neutral state (log10 ratios 0, logits)
    O = 13 * 64 + 64 + 2 * (64 * 64 + 64)
    w[O:O + 384] *= 0.1
    w[O + 384:O + 390] = [0.0, 0.0, 9.2, 9.2, 0.0, -9.2]
    return w


def _samples(rows, seed):
    """Training samples with the features' spread: a few decades each, and smooth targets."""
    rng = np.random.default_rng(seed)
    mean = rng.uniform(-4.0, 4.0, 13)
    scale = rng.uniform(0.5, 3.0, 13)
    w = _weights(rng, mean, scale)
    gen = _generator(seed + 1)
    X = torch.randn((rows, 13), generator=gen, device=DEV, dtype=torch.float64)
    A = torch.as_tensor(rng.standard_normal((13, 6)) / 2.0, device=DEV)
    Y = torch.tanh(X @ A) + 0.05 * torch.randn((rows, 6), generator=gen, device=DEV, dtype=torch.float64)
    X = X * torch.as_tensor(scale, device=DEV) + torch.as_tensor(mean, device=DEV)
    return X.float().contiguous(), Y.float().contiguous(), w


def _tiny_solver():
    """A handle whose grid plays no part (the network entry points work on rows)."""
    return rhi.Solver(2, 2, 2, CELL, rhi.rhi_params_default(1))


def prepare(case, seed):
    k = case["kind"]
    st = dict(case=case)
    if k == "norm":
        gen = _generator(seed)
        st["v"] = torch.randn(case["n"], generator=gen, device=DEV, dtype=torch.float64) * 10.0 ** (
            6.0 * torch.rand(case["n"], generator=gen, device=DEV, dtype=torch.float64) - 8.0)
        st["out"] = torch.empty(1, dtype=torch.float64, device=DEV)
        return st
    if k in ("mlp_forward", "mlp_grad", "mlp_train"):
        s = _tiny_solver()
        X, Y, w = _samples(case["rows"], seed)
        s.mlp_set_weights(w)
        st.update(s=s, X=X, Y=Y, w=w)
        if k == "mlp_forward":
            st["out"] = torch.empty_like(Y)
        return st
    N = case["nx"] * case["ny"] * case["nz"]
    if k == "lte":
        rng = np.random.default_rng(seed)
        e_vol, kap = 10.0 ** rng.uniform(9.5, 10.5), 4e-8 * rng.uniform(0.8, 1.25)
        rho, E0 = 1e-7, 1e12 * rng.uniform(0.8, 1.25)
        full = lambda v: torch.full((N,), v, dtype=torch.float64, device=DEV)  # noqa: E731
        st.update(s=_solver(case, 1.0 / case["nx"], 0, 0.0, (1e17, 1.0, 1e12), None, True,
                            model=rhi.RHI_MODEL_LTE, kappa_total=kap, kappa_planck=kap, mu=0.6,
                            limiter_jacobian=2, precond=rhi.RHI_PRECOND_MG_FP32, mg_levels=2),
                  fields=(full(E0), full(e_vol / rho), None, full(rho / M_H)),
                  steps=[1e-12 * 2.0 ** q for q in range(case["steps"])], tol=(1e-10, 1e-9),
                  lte=(E0, e_vol / rho, rho, kap))
        st["out"] = _outputs(st["s"])
        return st
    if k in ("uniform", "advance"):
        gen = _generator(seed)
        # nearly uniform hydrogen: each realisation has its own small density noise
        nH = 1e-3 * (1.0 + 1e-2 * torch.rand(N, generator=gen, device=DEV, dtype=torch.float64))
        hii = k == "advance"
        x0, T0 = (0.0012, 1e4) if hii else (1e-4, 100.0)
        z = torch.zeros_like(nH)
        e = _energy(T0, nH, z, x0 * nH, z, z)
        E = torch.full_like(nH, 1e-20)
        u_e = float(_energy(T0, torch.tensor(1e-3), torch.tensor(0.0), torch.tensor(x0 * 1e-3),
                            torch.tensor(0.0), torch.tensor(0.0)))
        dims = (case["nx"], case["ny"], case["nz"])
        if hii:
            dx, over, u = 6.6 * KPC / dims[0], dict(
                isothermal=1, dt_norm=2, dt_tau_tol=0.01, precond=rhi.RHI_PRECOND_MG_FP32,
                mg_levels=4, limiter_jacobian=2), (u_e, 1e-3, 1e-17)
            ijk, rate = np.zeros((1, 3), dtype=np.int32), np.array([5e48 / 8])
            t_rec = 1.0 / (2.59e-13 * 1e-3)
            st["t_end"] = case["t_over_trec"] * t_rec
        else:
            dx, over, u = MPC / dims[0], {}, (u_e, 1e-3, 1e-20)
            mid = [[m // 2 - 1, m // 2] if m % 2 == 0 else [m // 2] for m in dims]
            ijk = np.array([(i, j, q) for q in mid[2] for j in mid[1] for i in mid[0]], dtype=np.int32)
            rate = np.full(len(ijk), 5e48 / len(ijk))
            st["steps"], st["tol"] = [1e12] * case["steps"], (1e-8, 1e-10)
        s = _solver(case, dx, 1, 0.0, u, (rhi.RHI_SPECTRUM_MONO, 13.6 * EV), False, **over)
        st.update(s=s, fields=(E, e, (nH - x0 * nH).contiguous(), nH), ijk=ijk, rate=rate,
                  out=_outputs(s))
        return st
    nH, y_he, nHe, fr = _lognormal(case, seed)
    bb = (rhi.RHI_SPECTRUM_BLACKBODY, 1e5)
    if k == "lognormal":
        E, e, n = _state(nH, nHe, torch.full_like(nH, 100.0), fr, torch.full_like(nH, 1e-20))
        s = _solver(case, CELL * case["cell"], 3, y_he, (float(e.mean()), float(nH.mean()), U_E), bb,
                    case["periodic"], **_form(case))
        if case["form"] == "learned":
            s.mlp_set_weights(_no_change_weights(np.random.default_rng(seed)))
        ijk, rate = _sources(case, seed, case["cell"])
        st.update(s=s, fields=(E, e, n, nH), ijk=ijk, rate=rate, out=_outputs(s),
                  steps=[5e12] * case["steps"], tol=(1e-8, 1e-10))
        return st
    # linearize: the same gas with an ionised, heated region around each source
    ijk, rate = _sources(case, seed, 1.0)
    eps = rhi.rhi_grey_constants(*bb, 3)["eps"]
    shape = (case["nz"], case["ny"], case["nx"])
    ax = [torch.arange(m, device=DEV, dtype=torch.float64) for m in shape]
    E = torch.full(shape, 1e-20, dtype=torch.float64, device=DEV)
    for (i, j, q), r in zip(ijk, rate):
        r2 = ((ax[0] - float(q)) ** 2)[:, None, None] + ((ax[1] - float(j)) ** 2)[None, :, None] \
            + ((ax[2] - float(i)) ** 2)[None, None, :] + 0.3
        E += float(r) * eps / (4 * math.pi * C_LIGHT * CELL ** 2) / r2 * torch.exp(-torch.sqrt(r2) / 6.0)
    E = E.ravel()
    y = (E / 1e-18) ** 1.5
    x = 1e-4 + (1.0 - 1e-4 - 1e-6) * y / (1.0 + y)
    fr = x, 1e-4 + 0.8 * (x - 1e-4), 1e-8 + 0.15 * x * x
    E, e, n = _state(nH, nHe, 100.0 + 2e4 * x, fr, E)
    u = (1e12, float(nH.mean()), U_E)
    s = _solver(case, CELL, 3, y_he, u, bb, case["periodic"], **_form(case))
    src = torch.zeros_like(nH)
    flat = torch.as_tensor(ijk[:, 0] + case["nx"] * (ijk[:, 1] + case["ny"] * ijk[:, 2].astype(np.int64)), device=DEV)
    src.index_add_(0, flat, torch.as_tensor(rate * eps / CELL ** 3, device=DEV))
    s.set_state(E, e, n, nH, src)
    st.update(s=s, fields=(E, e, n, nH, src), y_he=y_he, u=u, grey=rhi.rhi_grey_constants(*bb, 3),
              out=[torch.empty(m * N, dtype=torch.float64, device=DEV) for m in (5, 1, 3, 3, 1)])
    return st


# ---- one pass ------------------------------------------------------------------------------------

def run(state):
    k = state["case"]["kind"]
    if k == "norm":
        v, out = state["v"], state["out"]
        rc = rhi.rhi_rms_norm_noalloc(v.data_ptr(), v.numel(), v.numel(), out.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream)
        if rc:
            raise RuntimeError(rhi.rhi_status_string(rc))
        return out
    s = state["s"]
    if k == "mlp_forward":
        return s.mlp_forward(state["X"], out=state["out"])
    if k == "mlp_grad":
        loss, grad = s.mlp_loss_grad(state["X"], state["Y"])
        return dict(loss=loss, grad=grad)
    if k == "mlp_train":
        s.mlp_set_weights(state["w"])
        loss = s.mlp_train(state["X"], state["Y"], epochs=1, batch=state["case"]["batch"], lr=1e-3)
        return dict(loss=loss, weights=s.mlp_get_weights())
    if k == "linearize":
        f, d, lo, hi, r = state["out"]
        rc = rhi.lib().rhi_linearize(s.h, 5e12, 1.0, 0.0, *(ctypes.c_void_p(t.data_ptr()) for t in (f, d, lo, hi, r)), 1)
        if rc:
            raise RuntimeError(rhi.rhi_status_string(rc))
        return dict(f=f, diag=d, lo=lo, hi=hi, rhs=r)
    E, e, n, nH = state["fields"]
    s.set_state(E, e, n, nH)
    if k != "lte":
        s.set_sources(state["ijk"], state["rate"])
    out = {}
    if k == "advance":
        out["t"], out["steps"] = s.advance(state["t_end"], 1e10, dt_min=1e6, newton_tol=1e-7, lin_tol=1e-8)
    else:
        for dt in state["steps"]:
            s.step(dt, newton_tol=state["tol"][0], lin_tol=state["tol"][1])
    oE, oe, on = state["out"]
    s.get_state(oE, oe, on)
    out.update(E=oE, e=oe)
    if k != "lte":
        out["n"] = on
    return out


def work(case):
    """Inputs read once, outputs written once; operations of the formulas themselves (for the
    steps: four Newton evaluations of the local model and faces and thirty products with the
    7-point matrix per step, the least the listed workloads take)."""
    k = case["kind"]
    if k == "norm":
        return dict(bytes=8 * case["n"] + 8, flops=2 * case["n"])
    mac = 13 * 64 + 2 * 64 * 64 + 64 * 6
    if k == "mlp_forward":
        return dict(bytes=4 * 19 * case["rows"] + 4 * 9632, flops=2 * mac * case["rows"])
    if k in ("mlp_grad", "mlp_train"):
        return dict(bytes=4 * 19 * case["rows"] + 8 * 9632, flops=(6 * mac - 2 * 13 * 64) * case["rows"])
    N = case["nx"] * case["ny"] * case["nz"]
    if k == "linearize":
        return dict(bytes=8 * N * (7 + 13), flops=900 * N)
    ns = {"lte": 0, "uniform": 1, "advance": 1, "lognormal": 3}[k]
    per = {0: 400, 1: 1200, 3: 3800}[ns]
    steps = case.get("steps", 8)
    return dict(bytes=8 * N * (5 + 2 * ns), flops=per * N * steps)


# ---- what the outputs are in 64 bits ---------------------------------------------------------------

def exact(case, seed):
    """The network and the norm in 64 bits, the LTE steps' backward-Euler root, and the
    linearisation by automatic differentiation.  A step of the ionization model stops at the
    iterate its tolerances ask for, which no closed computation gives: None."""
    k = case["kind"]
    if k in ("uniform", "advance", "lognormal"):
        return None
    st = prepare(case, seed)
    if k == "norm":
        return torch.linalg.vector_norm(st["v"]).reshape(1) / math.sqrt(case["n"])
    if k == "lte":
        return _exact_lte(st)
    if k == "linearize":
        return _exact_linearize(st)
    X, Y, w = st["X"].double(), st["Y"].double(), torch.as_tensor(st["w"].astype(np.float64), device=DEV)
    if k == "mlp_forward":
        return torch.cat([_mlp(w, x) for x in X.split(1 << 20)])
    if k == "mlp_grad":
        loss, grad = _mlp_loss_grad(w, X, Y)
        return dict(loss=loss, grad=grad)
    n, m1, m2, se = w.numel() - 26, torch.zeros_like(w), torch.zeros_like(w), 0.0
    for t, (x, y) in enumerate(zip(X.split(case["batch"]), Y.split(case["batch"])), 1):
        loss, g = _mlp_loss_grad(w, x, y)
        se += loss * x.shape[0]
        m1 = 0.9 * m1 + 0.1 * g
        m2 = 0.999 * m2 + 0.001 * g * g
        up = 1e-3 * (m1 / (1 - 0.9 ** t)) / (torch.sqrt(m2 / (1 - 0.999 ** t)) + 1e-8)
        w = torch.cat([w[:n] - up[:n], w[n:]])
    return dict(loss=se / X.shape[0], weights=w)


def _mlp(w, X):
    at, h = 0, (X - w[-26:-13]) / w[-13:]
    for layer, (rows, cols) in enumerate(((64, 13), (64, 64), (64, 64), (6, 64))):
        W = w[at:at + rows * cols].reshape(rows, cols)
        b = w[at + rows * cols:at + rows * cols + rows]
        at += rows * cols + rows
        h = h @ W.T + b
        if layer < 3:
            h = h * torch.sigmoid(h)
    return h


def _mlp_loss_grad(w, X, Y):
    w = w.detach().clone().requires_grad_(True)
    loss = ((_mlp(w, X) - Y) ** 2).mean()
    loss.backward()
    g = w.grad.clone()
    g[-26:] = 0.0                                  # the normalisation is held
    return float(loss), g


def _exact_lte(st):
    """Backward Euler of a uniform box, E' + rho e' held: one equation per step in e'."""
    E, e, rho, kap = st["lte"]
    cT = (5.0 / 3.0 - 1.0) * 0.6 * M_H / K_BOLTZ
    for dt in st["steps"]:
        tot, e0, x = E + rho * e, e, e
        for _ in range(100):
            f = rho * (x - e0) - dt * (C_LIGHT * kap * (tot - rho * x) - 4 * kap * SIGMA_SB * (cT * x) ** 4)
            df = rho + dt * (C_LIGHT * kap * rho + 16 * kap * SIGMA_SB * cT ** 4 * x ** 3)
            x -= f / df
        E, e = tot - rho * x, x
    N = st["s"].N
    return dict(E=torch.full((N,), E, dtype=torch.float64), e=torch.full((N,), e, dtype=torch.float64))


def _rates():
    """Node values and slopes of the 11 coefficients: 64 bins per octave of [1, 2^30) K."""
    i = np.arange(30 * 64 + 1)
    T = np.ldexp(1.0 + (i % 64) / 64.0, i // 64)
    sq, d5 = np.sqrt(T), 1.0 + np.sqrt(T / 1e5)
    brem = 1.42e-27 * (1.1 + 0.34 * np.exp(-(5.5 - np.log10(T)) ** 2 / 3.0)) * sq
    lam = lambda th: 2.0 * th / T                                                   # noqa: E731
    rate = lambda th: 2.753e-14 * lam(th) ** 1.5 / (1 + (lam(th) / 2.740) ** 0.407) ** 2.242       # noqa: E731
    cool = lambda th: 3.435e-30 * T * lam(th) ** 1.970 / (1 + (lam(th) / 2.250) ** 0.376) ** 3.720  # noqa: E731
    he2 = 1.26e-14 * lam(285335.0) ** 0.75
    diel = T ** -1.5 * np.exp(-470000.0 / T) * (1 + 0.3 * np.exp(-94000.0 / T))
    k = np.stack([
        rate(157807.0), 5.85e-11 * sq * np.exp(-157809.1 / T) / d5, he2 + 1.90e-3 * diel,
        2.38e-11 * sq * np.exp(-285335.4 / T) / d5, 2.0 * rate(631515.0),
        5.68e-12 * sq * np.exp(-631515.0 / T) / d5,
        7.50e-19 * np.exp(-118348.0 / T) / d5 + 1.27e-21 * sq * np.exp(-157809.1 / T) / d5,
        cool(157807.0) + brem, 9.38e-22 * sq * np.exp(-285335.4 / T) / d5,
        4.95e-22 * sq * np.exp(-631515.0 / T) / d5 + 5.54e-17 * T ** -0.397 * np.exp(-473638.0 / T) / d5
        + K_BOLTZ * T * he2 + 1.24e-13 * diel + brem,
        8.0 * cool(631515.0) + 4.0 * brem], axis=1)
    slope = np.diff(k, axis=0) / np.diff(T)[:, None]
    return torch.as_tensor(T, device=DEV), torch.as_tensor(k, device=DEV), torch.as_tensor(slope, device=DEV)


def _exact_linearize(st):
    """f, the exact Newton matrix reduced to E, and its right-hand side at U^n (theta = 1, a = 1,
    adot = 0), all derivatives by forward-mode differentiation of the operators themselves."""
    case, dt, u = st["case"], 5e12, st["u"]
    E, e, n, nH, src = st["fields"]
    n = n.reshape(3, -1)
    nHe = st["y_he"] * nH
    rho = M_H * (nH + 4.0 * nHe)
    sk, pg, ph = (st["grey"][q] for q in ("sk", "pgam", "ph"))
    nodes, tab, slope = _rates()

    def temperature(ec, n0, n1, n2):
        ne = (nH - n0) + n2 + 2.0 * (nHe - n1 - n2)
        return (2.0 / 3.0) * rho * (e + ec) / (K_BOLTZ * (nH + nHe + ne)), ne

    b = (torch.searchsorted(nodes, temperature(0.0, *n)[0], right=True) - 1).clamp(0, 30 * 64 - 1)

    def local(ec, n0, n1, n2, E):
        T, ne = temperature(ec, n0, n1, n2)
        k = [tab[b, r] + slope[b, r] * (T - nodes[b]) for r in range(11)]
        nHII, nHeIII = nH - n0, nHe - n1 - n2
        cE = C_LIGHT * E
        return (-cE * (ph[0] * n0 + ph[1] * n1 + ph[2] * n2) / rho
                + ne * (k[6] * n0 + k[7] * nHII + k[8] * n1 + k[9] * n2 + k[10] * nHeIII) / rho,
                cE * pg[0] * n0 + ne * (k[1] * n0 - k[0] * nHII),
                cE * pg[1] * n1 + ne * (k[3] * n1 - k[2] * n2),
                cE * (pg[2] * n2 - pg[1] * n1) + ne * ((k[5] + k[2]) * n2 - k[3] * n1 - k[4] * nHeIII),
                cE * (sk[0] * n0 + sk[1] * n1 + sk[2] * n2) - src)

    U = (torch.zeros_like(E), n[0], n[1], n[2], E)
    zero, one = torch.zeros_like(E), torch.ones_like(E)
    cols = []
    for q in range(5):
        L, J = torch.func.jvp(local, U, tuple(one if p == q else zero for p in range(5)))
        cols.append(J)
    # faces: flux W (E_c - E_lower) through each lower face and its derivatives
    shape = (case["nz"], case["ny"], case["nx"])
    kap = sk[0] * n[0] + sk[1] * n[1] + sk[2] * n[2]
    Rmin = 1.0 / (max(shape) * CELL)

    def flux(Ea, Eb, ka, kb):
        R = torch.abs(Eb - Ea) / (CELL * 0.5 * (Ea + Eb))
        R = torch.where(R > Rmin, R, torch.full_like(R, Rmin))
        k = 0.5 * (ka + kb)
        return C_LIGHT * (2 * k + R) / (6 * k * k + 3 * k * R + R * R) / CELL ** 2 * (Eb - Ea)

    def shift(x, ax, by):                          # the neighbour's value along x, y, z
        return torch.roll(x.reshape(shape), by, dims=2 - ax).ravel()

    faces, D = [], torch.zeros_like(E)
    for ax in range(3):
        has = torch.ones(shape, dtype=torch.float64, device=DEV)
        if not case["periodic"]:
            has.select(2 - ax, 0).zero_()
        has = has.ravel()
        at = (shift(E, ax, 1), E, shift(kap, ax, 1), kap)
        d = [torch.func.jvp(flux, at, tuple(one if p == q else zero for p in range(4))) for q in range(3)]
        F, P, Q, K = d[0][0] * has, d[1][1] * has, -d[0][1] * has, d[2][1] * has
        D += F - shift(F, ax, -1)
        faces.append((P, Q, K))
    scale = (u[0], u[1], u[1], u[1], u[2])
    Lf = list(L[:4]) + [L[4] + D]
    f = [dt * Lf[q] / scale[q] for q in range(5)]          # theta = 1: f(U^n) = dt L(U^n)
    M = torch.stack([torch.stack([dt * cols[s][r] * (scale[s] / scale[r]) + (1.0 if r == s else 0.0)
                                  for s in range(4)], dim=-1) for r in range(4)], dim=-2)
    rhs2 = torch.stack([torch.stack(f[:4], dim=-1),
                        torch.stack([dt * cols[4][r] * (scale[4] / scale[r]) for r in range(4)], dim=-1)], dim=-1)
    y, z = torch.linalg.solve(M, rhs2).unbind(-1)
    Lrow = torch.stack([dt * cols[r][4] * (scale[r] / scale[4]) for r in range(4)], dim=-1)
    skt = torch.as_tensor([0.0] + [float(v) for v in sk[:3]], dtype=torch.float64, device=DEV) * (u[1] / u[2])
    rho_c, phi_c = z @ skt, y @ skt
    diag = 1.0 + dt * cols[4][4] - (Lrow * z).sum(-1)
    rhs = (Lrow * y).sum(-1) - f[4]
    lo, hi = [], []
    for ax, (P, Q, K) in enumerate(faces):
        Kh = shift(K, ax, -1)
        diag = diag + dt * (P + shift(Q, ax, -1) - K * rho_c + Kh * rho_c)
        rhs = rhs + dt * (K * (shift(phi_c, ax, 1) + phi_c) - Kh * (phi_c + shift(phi_c, ax, -1)))
        lo.append(dt * (Q + K * shift(rho_c, ax, 1)))
        hi.append(dt * shift(P - K * rho_c, ax, -1))
    return dict(f=torch.cat(f), diag=diag, lo=torch.cat(lo), hi=torch.cat(hi), rhs=rhs)
