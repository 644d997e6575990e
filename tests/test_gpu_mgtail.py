"""The V-cycle's coarse end as one cluster launch (`k_mg_tail`) against the numpy restatement of the
cycle, at the shapes where its split over blocks and threads can go wrong: chunks that do not
divide the level, levels next to the sizes where it starts (32768 FP32 cells, 8192 FP64 cells,
one cell per thread on the second level) or turns narrow (512, 128 cells), grids of one row,
one level alone, periodic wraps across chunks, and odd and even numbers of sweeps.

Tolerances as for the level kernels: FP64 differs by the order of sums only (1e-12); FP32 carries
single-precision rounding through the cycle (1e-4)."""
import numpy as np
import pytest

import mg_reference as mgr
from paper_0901_1110_gb300 import inputs

pytestmark = pytest.mark.gpu
KPC = inputs.KPC

# (nz, ny, nx), levels, (pre, post, coarse) sweeps, periodic
CASES = [((32, 32, 32), 4, (2, 2, 16), False), ((33, 31, 32), 5, (2, 2, 16), True),
         ((33, 32, 32), 3, (2, 2, 16), False), ((16, 32, 16), 6, (1, 2, 5), False),
         ((16, 33, 16), 3, (3, 1, 4), True), ((8, 8, 8), 2, (2, 2, 16), True),
         ((9, 8, 8), 3, (2, 0, 16), False), ((4, 8, 4), 3, (1, 1, 1), False),
         ((5, 9, 3), 1, (2, 2, 7), True), ((23, 19, 17), 1, (2, 2, 6), False),
         ((1, 1, 700), 8, (2, 2, 16), False), ((1, 300, 1), 4, (2, 3, 16), True),
         ((1, 130, 127), 5, (2, 2, 16), False), ((1, 1, 1), 2, (2, 2, 16), False)]


@pytest.mark.parametrize("shape,levels,sweeps,periodic", CASES)
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-4)])
@pytest.mark.parametrize("matrix", [0, 2])
def test_vcycle_matches_numpy_restatement(shape, levels, sweeps, periodic, precision, tol, matrix):
    import paper_0901_1110_gb300 as rhi
    w = inputs.lognormal_hhe(shape, box=4 * KPC * shape[2], nsrc=2, dt=5e12, seed=3,
                             bc=("periodic" if periodic else "zero_flux",) * 6)
    w.theta, w.u_E = 1.0, 1e-18
    rng = np.random.default_rng(1)
    w.E = w.E * np.exp(3.0 * rng.standard_normal(w.E.shape))
    w.n = w.n * rng.uniform(0.01, 0.9, w.n.shape)
    pre, post, coarse = sweeps
    s = rhi.solver_for_workload(w, mg_levels=levels, mg_pre=pre, mg_post=post, mg_coarse_sweeps=coarse,
                                precond=rhi.RHI_PRECOND_MG_FP64 if precision == "fp64" else rhi.RHI_PRECOND_MG_FP32,
                                limiter_jacobian=matrix)
    lin = s.linearize(w.dt)
    r = rng.standard_normal(s.N)
    z = s.precond_apply(r)
    s.close()
    W = [lin["face"][ax].reshape(shape) for ax in range(3)]
    Wp = [np.roll(lin["face_hi"][ax].reshape(shape), 1, axis=2 - ax) for ax in range(3)] if matrix else None
    ops = mgr.hierarchy(lin["diag"].reshape(shape), W, levels, Wp)
    zr = mgr.vcycle(ops, r.reshape(shape), 0.9, pre, post, coarse).ravel()
    assert np.linalg.norm(z - zr) <= tol * np.linalg.norm(zr)
