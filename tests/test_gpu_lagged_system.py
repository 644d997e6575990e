"""The lagged-D system of a solver that keeps dD/dE: as its preconditioner (mg_matrix 0, Jacobi) it is the
matrix of limiter_jacobian 0 at the same state, its storage is part of the handle, and where BiCGStab
breaks down the Newton iteration takes its direction.

Tolerances: the two forms of the matrix add its terms in another order, a few units of 2^-52 of the largest
(here up to 1e3 times the diagonal), so 1e-12 of z's maximum for FP64; an FP32 hierarchy may round a
coefficient to the next FP32 number, 6e-8, through some tens of sweeps: 1e-5.  A fallback's direction
solves the same system to lin_tol = 1e-8 of the residual: 1e-6 over five iterations."""
import numpy as np
import pytest

from paper_0901_1110_gb300 import inputs

pytestmark = pytest.mark.gpu
KPC = inputs.KPC
MIXED = ("dirichlet", "zero_flux", "periodic", "periodic", "dirichlet", "dirichlet")


def _flat(a):
    return np.ascontiguousarray(a).ravel()


def _solver(rhi, shape, bc=("zero_flux",) * 6, decades=4.0, box=None, **over):
    """Nearly ionised hydrogen with a steep radiation field (free streaming at its faint end)."""
    w = inputs.uniform_h(4, shape=shape, box=box or KPC * shape[2], x0=1 - 1e-4, T0=1e4, E0=1e-16, bc=bc)
    w.bc_value = (1e-16, 0.0, 0.0, 0.0, 1e-17, 1e-18)
    w.theta, w.u_E = 1.0, 1e-18
    s = rhi.solver_for_workload(w, sources=False, **over)
    z, y, x = np.meshgrid(*[np.arange(n) / max(n - 1, 1) for n in shape], indexing="ij")
    st = w.state()
    s.set_state(_flat(1e-16 * 10.0 ** (-decades * (x + 0.3 * y + 0.1 * z))), _flat(st["e"]), _flat(st["n"]),
                _flat(w.nH))
    return s


@pytest.mark.parametrize("shape", [(5, 6, 7), (33, 34, 37)])
@pytest.mark.parametrize("ljac,bc", [(1, MIXED), (1, ("periodic",) * 6), (2, ("zero_flux",) * 6)])
@pytest.mark.parametrize("precond", ["JACOBI", "MG_FP64", "MG_FP32"])
def test_lagged_preconditioner_is_that_of_the_lagged_solver(shape, ljac, bc, precond):
    import paper_0901_1110_gb300 as rhi
    r = np.random.default_rng(3).standard_normal(int(np.prod(shape)))
    z = []
    for lj in (0, ljac):
        s = _solver(rhi, shape, bc, limiter_jacobian=lj, precond=getattr(rhi, "RHI_PRECOND_" + precond),
                    mg_matrix=0, mg_levels=4)
        s.linearize(2e11)
        z.append(s.precond_apply(r))
        s.close()
    tol = 1e-5 if precond == "MG_FP32" else 1e-12
    assert np.abs(z[1] - z[0]).max() <= tol * np.abs(z[0]).max()


@pytest.mark.parametrize("ljac", [1, 2])
@pytest.mark.parametrize("precond,matrix", [("JACOBI", 1), ("MG_FP64", 0), ("MG_FP32", 0)])
def test_no_device_memory_is_taken_by_a_call(ljac, precond, matrix):
    """rhi_create allocates every buffer: neither the linearisation nor a step takes any (the first of
    the two handles loads the kernels; no graphs, which hold memory of their own)."""
    import torch

    import paper_0901_1110_gb300 as rhi
    n = 64
    for _ in range(2):
        s = _solver(rhi, (n, n, n), limiter_jacobian=ljac, precond=getattr(rhi, "RHI_PRECOND_" + precond),
                    mg_matrix=matrix, krylov_graph=0, vcycle_graph=0, max_newton=1)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        s.linearize(1e11)
        s.step(1e11, check=False)
        taken = before - torch.cuda.mem_get_info()[0]
        s.close()
    assert taken < 8 * n ** 3, f"{taken / (8 * n ** 3):.1f} fields"


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("precond,sweeps", [("MG_FP64", 1500), ("MG_FP32", 300)])
@pytest.mark.parametrize("decades", [8.0, 12.0])
def test_breakdown_takes_the_lagged_direction(graph, precond, sweeps, decades):
    """Jacobi sweeps of the advective Newton matrix grow without bound, so many of them overflow and every
    BiCGStab solve breaks down, from U^n on; the lagged-D matrix's sweeps converge.  The residuals
    are then those of limiter_jacobian 0."""
    import paper_0901_1110_gb300 as rhi
    out = []
    for lj, nsweep in ((0, 16), (1, sweeps)):
        s = _solver(rhi, (1, 1, 96), decades=decades, limiter_jacobian=lj, krylov_graph=graph, mg_levels=1,
                    precond=getattr(rhi, "RHI_PRECOND_" + precond), mg_coarse_sweeps=nsweep, max_newton=5)
        s.step(5.0 * KPC / 3e10, newton_tol=1e-10, lin_tol=1e-8, check=False)
        out.append(s.stats())
        s.close()
    assert out[1]["krylov_fallbacks"] == out[1]["newton_its"] == 5, out[1]
    np.testing.assert_allclose(out[1]["res_history"], out[0]["res_history"], rtol=1e-6)
