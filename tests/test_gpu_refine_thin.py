"""GPU: refined Poisson solves of boxes of few planes, whose residual kernels take pairs of planes alone and
groups of four in a group of boxes: the oracle's solution, and the same bits both ways."""

import numpy as np
import pytest

import oracle
from paper_2502_06296_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def chanfs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_06296_gb300 import build as libbuild
    libbuild.build()
    from paper_2502_06296_gb300 import chanfs as c
    c.lib()
    return c


@pytest.mark.parametrize("nz", [3, 4, 5, 6, 7, 8, 9, 10])
def test_boxes_of_few_planes(chanfs, nz):
    nx, ny = 36, 27
    dz = synth.tanh_dz(nz, 1.3)
    f = synth.remove_weighted_mean(synth.normal(nz, (nz, ny, nx)), dz)
    ref = oracle.poisson_solve(f, 2.0, 1.0, dz, 0)
    t = torch.from_numpy(f).cuda()
    with chanfs.Plan(nx, ny, nz, 2.0, 1.0, dz, 0, chanfs.F32_REFINED) as plan, \
            chanfs.Plan(32, 24, 16, 2.0, 1.0, np.full(16, 0.1), 0, chanfs.F32_REFINED) as beside:
        alone = plan.poisson_solve(t)
        iters, rho = plan.last_info()
        assert rho <= 1e-10 and 1 <= iters <= 4
        # the target, with the order of magnitude that the operator's condition leaves to the solution
        assert np.max(np.abs(alone.cpu().numpy() - ref)) / np.max(np.abs(ref)) < 1e-9
        other = torch.from_numpy(synth.normal(5, (16, 24, 32))).cuda()
        with chanfs.Group([beside, plan]) as g:
            assert torch.equal(g.poisson_solve([other, t])[1], alone)
