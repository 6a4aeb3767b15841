"""GPU: the block fixed-point FP64 transforms and the z sweeps at the edges of
their dispatch: compiled and general lengths, single and repeated first passes,
every radix, ragged tiles, lines of special values; z sweeps with one, two and
four right-hand sides per thread and every remainder of a row group."""

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


def packed(f):
    """The packed spectrum of cfs_spectral_forward by numpy."""
    nz, ny, nx = f.shape
    m = nx // 2
    x = np.fft.fft(np.fft.rfft(f, axis=2), axis=1)
    out = x[:, :, :m].copy()
    for k in range(ny):
        if (2 * k) % ny == 0:
            out[:, k, 0] = x[:, k, 0].real + 1j * x[:, k, m].real
        elif 2 * k > ny:
            out[:, k, 0] = x[:, ny - k, m]
    return out


# L2 errors: one rounding of the result (2^-53) and fixed-point noise of a few 2^-54 here; numpy's own
# FFT is within about 0.6 log2(n) 2^-53 of the exact transform: together below 16 x 2^-53
TOL = 16 * 2.0**-53

X = [16, 18, 24, 36, 54, 64, 96, 108, 162, 192, 216, 256, 384, 432, 486, 512, 768, 972, 1024, 1296, 1536, 1944,
     2048, 2916, 3456, 3888, 4096]
Y = [8, 9, 12, 16, 18, 27, 48, 54, 64, 81, 96, 128, 162, 192, 243, 256, 384, 432, 512, 576, 768, 1024, 1536, 2048, 2304]


@pytest.mark.parametrize("nx,ny", [(n, 3) for n in X] + [(20 if n % 2 else 32, n) for n in Y if n % 5] + [(54, n) for n in Y[::3]])
def test_transforms_match_numpy(chanfs, nx, ny):
    nx = 24 if nx == 20 else nx
    nz = 3
    rng = np.random.default_rng(nx * 10007 + ny)
    f = rng.standard_normal((nz, ny, nx)) * 10.0 ** rng.uniform(-3, 3, (nz, 1, 1))
    f[1] = np.cos(2 * np.pi * np.arange(nx) / nx) + 1e-9 * f[1]  # one dominant mode
    with chanfs.Plan(nx, ny, nz, 2.0, 1.0, np.full(nz, 0.5)) as plan:
        if ny > 1024:
            plan.set_option(chanfs.OPT_Y_TILE, 1)  # (the default tile of such a plan does not fit)
        t = torch.from_numpy(f).cuda()
        s = plan.spectral_forward(t)
        got = s.cpu().numpy().view(np.complex128).reshape(nz, ny, nx // 2)
        back = plan.spectral_inverse(s).cpu().numpy()
        assert plan.check() == 0
    ref = packed(f)
    for z in range(nz):
        assert np.linalg.norm(got[z] - ref[z]) < TOL * np.linalg.norm(ref[z]), z
        assert np.linalg.norm(back[z] - f[z]) < 2 * TOL * np.linalg.norm(f[z]), z


@pytest.mark.parametrize("nx,ny", [(512, 48), (108, 27), (24, 16)])
def test_special_lines(chanfs, nx, ny):
    """Zero planes give zeros, an infinity or NaN spoils its own plane's spectrum and no other, and a power of
    two as a factor of the field comes out as that factor, from the smallest to the largest exponents."""
    nz = 4
    f = np.random.default_rng(nx).standard_normal((nz, ny, nx))
    f[1] = 0.0
    with chanfs.Plan(nx, ny, nz, 2.0, 1.0, np.full(nz, 0.5)) as plan:
        base = plan.spectral_forward(torch.from_numpy(f).cuda()).cpu().numpy()
        assert not base[1].any()
        for e in (-1000, -950, -100, 100, 900):
            s = plan.spectral_forward(torch.from_numpy(np.ldexp(f, e)).cuda()).cpu().numpy()
            assert np.linalg.norm(np.ldexp(s, -e) - base) < TOL * np.linalg.norm(base), e
        for bad in (np.inf, np.nan):
            g = f.copy()
            g[2, ny // 2, 3] = bad
            s = plan.spectral_forward(torch.from_numpy(g).cuda()).cpu().numpy()
            assert not np.isfinite(s[2]).any()
            assert np.array_equal(s[[0, 1, 3]], base[[0, 1, 3]])


@pytest.mark.parametrize("nz", [3, 4, 6, 7, 13, 16])
@pytest.mark.parametrize("nx,ny,bc,ybc", [(512, 384, 0, 0), (512, 192, 0, 0), (96, 54, 1, 0), (96, 54, 0, 1), (512, 162, 1, 2)])
def test_z_sweeps_match_the_oracle(chanfs, nx, ny, nz, bc, ybc):
    dz = synth.tanh_dz(nz, 1.4)
    f = synth.normal(nx + ny + nz, (nz, ny, nx))
    if bc == 0 and ybc != 2:
        f = synth.remove_weighted_mean(f, dz)
    ref = oracle.poisson_solve_walls(f, 12.8, 6.4, dz, bc, ybc) if ybc else oracle.poisson_solve(f, 12.8, 6.4, dz, bc)
    with chanfs.Plan(nx, ny, nz, 12.8, 6.4, dz, bc, 0, ybc) as plan:
        p = plan.poisson_solve(torch.from_numpy(f).cuda()).cpu().numpy()
        assert plan.check() == 0
    assert np.max(np.abs(p - ref)) / np.max(np.abs(ref)) < 1e-12
