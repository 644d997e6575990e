"""Device memory of a handle, and the steps of a solver whose learned guess shares it.

A handle's fields (8 bytes per cell, at 128^3) may not exceed those of the layout with separate face
arrays for both work iterates and one diagonal more, which the solver once had and the sizes of users' grids
may rest on.  Where a learned guess loses to U^n, U^n's face arrays have lain in the Krylov vectors: the
step is then that of RHI_GUESS_PREVIOUS, bit for bit."""
import numpy as np
import pytest

from paper_0901_1110_gb300 import inputs

pytestmark = pytest.mark.gpu
# (n_species, limiter_jacobian): fields with Jacobi, FP64 and FP32 multigrid
FIELDS = {(0, 0): (32.2, 36.4, 36.7), (0, 1): (52.2, 56.8, 58.5), (0, 2): (58.2, 62.8, 64.5),
          (1, 0): (43.2, 47.4, 47.7), (1, 1): (63.2, 67.8, 69.5), (1, 2): (69.2, 73.8, 75.5),
          (3, 0): (61.2, 65.4, 65.7), (3, 1): (81.2, 85.8, 87.5), (3, 2): (87.2, 91.8, 93.5)}
ALLOCATOR = 4 * 2 ** 20                     # the small buffers' slab and the allocator's granularity


@pytest.mark.parametrize("guess", ["PREVIOUS", "LEARNED"])
@pytest.mark.parametrize("ns,ljac", sorted(FIELDS))
def test_fields_of_a_handle(ns, ljac, guess):
    import torch

    import paper_0901_1110_gb300 as rhi
    if ns == 0 and guess == "LEARNED":
        pytest.skip("the learned guess needs the ionization model")
    n = 128
    for precond, most in enumerate(FIELDS[ns, ljac]):
        p = rhi.rhi_params_default(ns)
        p.y_he = 0.08 if ns == 3 else 0.0
        p.limiter_jacobian, p.precond, p.guess = ljac, precond, getattr(rhi, "RHI_GUESS_" + guess)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        s = rhi.Solver(n, n, n, 1e22, p)
        taken = before - torch.cuda.mem_get_info()[0]
        s.close()
        assert taken <= 8 * n ** 3 * most + ALLOCATOR, (precond, taken / (8 * n ** 3), most)


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("ljac", [0, 1, 2])
@pytest.mark.parametrize("shape,precond", [((7, 9, 11), "MG_FP32"), ((20, 21, 23), "MG_FP64"), ((9, 8, 7), "JACOBI"),
                                           ((34, 35, 37), "MG_FP32")])
def test_lost_guess_leaves_the_step_of_the_previous_state(shape, ljac, graph, precond):
    import paper_0901_1110_gb300 as rhi
    w = inputs.lognormal_hhe(shape, box=10 * inputs.KPC * shape[2], nsrc=2, dt=2e12, seed=2)
    w.theta, w.u_E = 1.0, 1e-18
    weights = np.zeros(rhi.RHI_MLP_NWEIGHTS, dtype=np.float32)
    weights[-13:] = 1e3                            # features in range ...
    weights[-32:-26] = [3.0, 1.0, -4.0, 2.0, 0.0, 0.0]  # ... and one far-off output for every cell
    out = []
    for guess in (rhi.RHI_GUESS_PREVIOUS, rhi.RHI_GUESS_LEARNED):
        s = rhi.solver_for_workload(w, limiter_jacobian=ljac, krylov_graph=graph, mg_levels=4, guess=guess,
                                    mlp_retry=0, precond=getattr(rhi, "RHI_PRECOND_" + precond))
        s.mlp_set_weights(weights)
        for _ in range(3):
            s.step(w.dt, newton_tol=1e-9, lin_tol=1e-9)
            st = s.stats()
            assert st["guess_used"] == rhi.RHI_GUESS_PREVIOUS and st["newton_its"] > 0
            assert (st["res_guess_prev"] > 0) == (guess == rhi.RHI_GUESS_LEARNED)
        out.append(s.get_state())
        s.close()
    for k in ("E", "e", "n"):
        assert np.array_equal(out[0][k], out[1][k]), k


def test_small_handles_stay_small():
    """A 4^3 handle's buffers are 0.4 MB (most of it the rate table): 20 of them within 1 MB each."""
    import torch

    import paper_0901_1110_gb300 as rhi
    p = rhi.rhi_params_default(1)
    rhi.Solver(4, 4, 4, 1e22, p).close()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    handles = [rhi.Solver(4, 4, 4, 1e22, p) for _ in range(20)]
    taken = before - torch.cuda.mem_get_info()[0]
    for s in handles:
        s.close()
    assert taken <= 20 * 2 ** 20, taken / 20
