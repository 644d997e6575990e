"""The V-cycle's level kernels at the sizes where their forms change (the small levels of these
grids are one launch, which has a test of its own): the first two sweeps in one launch (plain, marching
along z, rows staged in shared memory; FP64 up to 64^3), the restriction with eight lanes to a parent (up
to 65536 parents) and the one with a thread to a parent, at odd extents (only children at the
far ends, parents that do not fill a warp), periodic wraps, one and more sweeps before, none to
three after, and one level alone, whose sweeps end in either of their two vectors.

Tolerances as for the other V-cycle tests: FP64 differs by the order of sums only (1e-12); FP32
carries single-precision rounding through the cycle (1e-4)."""
import numpy as np
import pytest

import mg_reference as mgr
from paper_0901_1110_gb300 import inputs

pytestmark = pytest.mark.gpu
KPC = inputs.KPC

# (nz, ny, nx), levels, (pre, post, coarse) sweeps, periodic
CASES = [((33, 35, 31), 4, (2, 2, 16), False), ((33, 35, 31), 4, (2, 1, 16), True),
         ((34, 33, 35), 3, (1, 2, 8), True), ((34, 33, 35), 1, (2, 2, 3), False),
         ((34, 33, 35), 1, (2, 2, 2), True), ((16, 9, 257), 2, (3, 0, 4), False),
         ((16, 11, 256), 3, (2, 2, 16), True), ((32, 7, 260), 3, (2, 3, 5), False),
         ((64, 64, 64), 4, (2, 2, 16), False), ((64, 65, 64), 4, (2, 2, 16), True),
         ((80, 81, 80), 4, (2, 2, 16), False), ((81, 81, 81), 4, (1, 1, 4), True)]


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
    again = s.precond_apply(r)
    s.close()
    assert np.array_equal(z, again)
    W = [lin["face"][ax].reshape(shape) for ax in range(3)]
    Wp = [np.roll(lin["face_hi"][ax].reshape(shape), 1, axis=2 - ax) for ax in range(3)] if matrix else None
    ops = mgr.hierarchy(lin["diag"].reshape(shape), W, levels, Wp)
    zr = mgr.vcycle(ops, r.reshape(shape), 0.9, pre, post, coarse).ravel()
    assert np.linalg.norm(z - zr) <= tol * np.linalg.norm(zr)
