"""CG on the lagged-D matrix as one CUDA graph launch per solve against the same kernels launched from
the host with one read per iteration (krylov_graph 0; there with the FP32 cycle as a graph of its own or
not): the steps agree bit for bit with the same counts, also after a change of step size, at grids whose
cycle is one launch and at grids with levels of their own kernels; with the graph a step makes one host
read per Newton iteration.  And the solve of a system that is already converged, or has a limit of
one iteration, ends where the direct one does."""
import numpy as np
import pytest

from paper_0901_1110_gb300 import inputs

pytestmark = pytest.mark.gpu


def _steps(rhi, shape, code, **over):
    w = inputs.uniform_h(8, shape=shape, box=inputs.MPC)
    w.theta = 1.0
    s = rhi.solver_for_workload(w, precond=code, **over)
    stats = []
    for dt in (1e12, 1e12, 4e11):
        s.step(dt, newton_tol=1e-8, lin_tol=1e-10)
        stats.append(s.stats())
    st = s.get_state()
    s.close()
    return st, stats


@pytest.mark.parametrize("shape", [(12, 9, 14), (36, 40, 33)])
@pytest.mark.parametrize("precond", ["RHI_PRECOND_JACOBI", "RHI_PRECOND_MG_FP64", "RHI_PRECOND_MG_FP32"])
def test_cg_graph_matches_direct_launches(shape, precond):
    import paper_0901_1110_gb300 as rhi
    code = getattr(rhi, precond)
    ref, refs = _steps(rhi, shape, code, krylov_graph=1)
    for vg in (0, 1):
        st, stats = _steps(rhi, shape, code, krylov_graph=0, vcycle_graph=vg)
        for key in ("E", "e", "n"):
            assert np.array_equal(np.asarray(st[key]), np.asarray(ref[key])), key
        for a, b in zip(stats, refs):
            for k in ("newton_its", "pcg_its", "vcycles", "backtracks"):
                assert a[k] == b[k], (k, a[k], b[k])
    for b in refs:
        assert b["pcg_its"] > 0
        assert b["host_syncs"] <= b["newton_its"] + b["backtracks"] + b["final_missed"] + 2, b


def test_cg_iteration_limit_is_kept():
    import paper_0901_1110_gb300 as rhi
    out = []
    for graph in (0, 1):
        w = inputs.uniform_h(8, shape=(10, 11, 12), box=inputs.MPC)
        w.theta = 1.0
        s = rhi.solver_for_workload(w, krylov_graph=graph, max_pcg=1, max_newton=3)
        rc = s.step(1e12, newton_tol=1e-14, lin_tol=1e-14, check=False)
        out.append((rc, s.stats()["pcg_its"], s.stats()["newton_its"], s.stats()["res_final"]))
        s.close()
    assert out[0] == out[1] and out[0][1] == out[0][2], out
