"""The allocation-free norm at the sizes where its kernels change: single values and odd ends, one block
more or less, the most blocks, where every thread's four-fold turns end, the largest input, and an address
that is not a multiple of 16 bytes.  Point sources: batches of 128 with several sources in one cell.

Tolerance of the norm: chains of at most n / 8192 + 32 additions, each rounding 2^-53 of a sum of
squares."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 511, 1023, 1024, 1025, 8191, 608 * 1024 - 1, 608 * 1024 + 1, 608 * 256 * 8 - 1,
                               608 * 256 * 8, 608 * 256 * 8 + 3, 2 ** 25])
@pytest.mark.parametrize("offset", [0, 1])
def test_norm_at_kernel_edges(n, offset):
    import torch

    import paper_0901_1110_gb300 as rhi
    g = torch.Generator(device="cuda").manual_seed(n)
    v = torch.randn(n + offset, generator=g, device="cuda", dtype=torch.float64)[offset:]
    out = torch.full((1,), -1.0, device="cuda", dtype=torch.float64)
    for count in (n, 3 * n):
        rc = rhi.rhi_rms_norm_noalloc(v.data_ptr(), n, count, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == rhi.RHI_OK
        ref = float(np.sqrt(np.sum(v.cpu().numpy().astype(np.longdouble) ** 2) / count))
        assert abs(out.item() / ref - 1.0) <= (n / 8192 + 32) * 2.0 ** -53
        assert v.numel() == n


@pytest.mark.parametrize("nsrc", [0, 1, 127, 128, 129, 300])
def test_sources_add_up_in_order(nsrc):
    import paper_0901_1110_gb300 as rhi
    rng = np.random.default_rng(nsrc)
    shape = (5, 4, 3)
    N = 60
    p = rhi.rhi_params_default(1)
    s = rhi.Solver(3, 4, 5, 1e20, p)
    one = np.ones(N)
    src = rng.uniform(0.0, 1e-27, N)
    s.set_state(one * 1e-20, one * 1e11, one * 5e-4, one * 1e-3, src.copy())
    ijk = np.stack([rng.integers(0, 3, nsrc), rng.integers(0, 4, nsrc), rng.integers(0, 5, nsrc)], axis=1)
    rate = rng.uniform(1e47, 1e49, nsrc)
    s.set_sources(ijk, rate)
    # theta = 0.51 by default; at E = 1e-20 the scaled radiation residual holds -dt theta src / u_E,
    # so the emissivity shows in the difference of two linearisations
    f1 = s.linearize(1.0)["f"][2]
    want = src.copy()
    for (i, j, k), r in zip(ijk, rate):
        want[i + 3 * (j + 4 * k)] += r * p.photon_energy / 1e20 ** 3
    s.set_state(one * 1e-20, one * 1e11, one * 5e-4, one * 1e-3, want)
    f2 = s.linearize(1.0)["f"][2]
    assert np.array_equal(f1, f2) and shape
    s.close()
