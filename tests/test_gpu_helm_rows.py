"""GPU: the Helmholtz Thomas sweeps at the edges of their groups of rows (8 in FP64, 12 in FP32, two groups in
flight), alone and in a group, with column counts that end inside a block."""

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


@pytest.mark.parametrize("nz", [4, 7, 8, 9, 12, 13, 15, 16, 17, 24, 25, 33, 40])
@pytest.mark.parametrize("loc", [0, 1])
def test_every_remainder_of_a_group_of_rows(chanfs, nz, loc):
    nx, ny, c = 24, 9, 3e-2
    dz = synth.tanh_dz(nz, 1.5)
    r = synth.normal(nz + 100 * loc, (nz, ny, nx))
    ref = oracle.helmholtz_solve(r, dz, c, loc)
    scale = np.max(np.abs(ref))
    t = torch.from_numpy(r).cuda()
    with chanfs.Plan(nx, ny, nz, 2.0, 1.0, dz) as plan:
        plan.set_option(chanfs.OPT_HELM_THOMAS, 1)
        u = plan.helmholtz_solve(c, t, loc).cpu().numpy()
        assert np.max(np.abs(u - ref)) / scale < 1e-13  # two roundings a row, 40 rows, diagonally dominant
    other = torch.from_numpy(synth.normal(7, (nz + 3, 6, 36))).cuda()
    with chanfs.Plan(nx, ny, nz, 2.0, 1.0, dz, 0, chanfs.F32_REFINED) as plan, \
            chanfs.Plan(36, 6, nz + 3, 2.0, 1.0, synth.tanh_dz(nz + 3, 1.2), 0, chanfs.F32_REFINED) as beside:
        for fp64 in (0, 1):
            for p in (plan, beside):
                p.set_option(chanfs.OPT_HELM_THOMAS32, 1)
                p.set_option(chanfs.OPT_HELM_THOMAS, 1)
                p.set_option(chanfs.OPT_HELM_FP64, fp64)
            alone = plan.helmholtz_solve(c, t, loc)
            tol = 1e-13 if fp64 else 1e-10  # (the refinement's target)
            assert np.max(np.abs(alone.cpu().numpy() - ref)) / scale < tol
            with chanfs.Group([beside, plan]) as g:
                out = g.helmholtz_solve([c, c], [other, t], [loc, loc])
                assert torch.equal(out[1], alone)
                assert torch.equal(out[0], beside.helmholtz_solve(c, other, loc))
