"""The FP64 V-cycle of the symmetric matrix on both sides of the size up to which its restriction has eight
lanes to a parent (24576 parents), at even and odd extents, against the numpy restatement; tolerance as
for the other FP64 V-cycle tests, the order of sums (1e-12)."""
import numpy as np
import pytest

import mg_reference as mgr
from paper_0901_1110_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(48, 64, 64), (47, 64, 63), (50, 64, 64), (49, 63, 65), (57, 58, 57), (60, 58, 58)])
@pytest.mark.parametrize("bc", ["zero_flux", "periodic"])
def test_symmetric_fp64_vcycle(shape, bc):
    import paper_0901_1110_gb300 as rhi
    w = inputs.lognormal_hhe(shape, box=4 * inputs.KPC * shape[2], nsrc=2, dt=5e12, seed=3, bc=(bc,) * 6)
    w.theta, w.u_E = 1.0, 1e-18
    rng = np.random.default_rng(1)
    w.E = w.E * np.exp(3.0 * rng.standard_normal(w.E.shape))
    s = rhi.solver_for_workload(w, mg_levels=4, precond=rhi.RHI_PRECOND_MG_FP64)
    lin = s.linearize(w.dt)
    r = rng.standard_normal(s.N)
    z = s.precond_apply(r)
    s.close()
    ops = mgr.hierarchy(lin["diag"].reshape(shape), [lin["face"][ax].reshape(shape) for ax in range(3)], 4)
    zr = mgr.vcycle(ops, r.reshape(shape), 0.9, 2, 2, 16).ravel()
    assert np.linalg.norm(z - zr) <= 1e-12 * np.linalg.norm(zr)
