"""stats.vcycles counts preconditioner applications with every preconditioner.  CG applies it once per
iteration, so the count equals pcg_its exactly, Jacobi included, with the solves as graphs or as direct
launches."""
import pytest

from paper_0901_1110_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("precond", ["JACOBI", "MG_FP64", "MG_FP32"])
def test_cg_counts_every_application(precond, graph):
    import paper_0901_1110_gb300 as rhi
    w = inputs.uniform_h(12, box=inputs.MPC)
    w.theta = 1.0
    s = rhi.solver_for_workload(w, precond=getattr(rhi, "RHI_PRECOND_" + precond), krylov_graph=graph)
    s.step(1e12, newton_tol=1e-8, lin_tol=1e-10)
    st = s.stats()
    s.close()
    assert st["pcg_its"] > 0 and st["vcycles"] == st["pcg_its"], st
