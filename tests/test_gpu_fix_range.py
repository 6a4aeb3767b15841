"""GPU: the block fixed-point FP64 transforms on data whose values differ widely, against transforms in
extended precision: lengths of many radix-3 passes, columns like 1/k^2 (what the inverse transforms of a
Poisson solve receive) and columns with one dominant value."""

import numpy as np
import pytest

import oracle
from paper_2502_06296_gb300 import synth

torch = pytest.importorskip("torch")
fft = pytest.importorskip("scipy.fft")
pytestmark = pytest.mark.gpu
X_FORWARD, Y_FORWARD, Y_INVERSE = 0, 1, 3  # stages of cfs_poisson_stage


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
    """The packed spectrum of cfs_spectral_forward in extended precision."""
    nz, ny, nx = f.shape
    m = nx // 2
    x = fft.fft(fft.rfft(f.astype(np.longdouble), axis=2), axis=1)
    out = x[:, :, :m].copy()
    for k in range(ny):
        if (2 * k) % ny == 0:
            out[:, k, 0] = x[:, k, 0].real + 1j * x[:, k, m].real
        elif 2 * k > ny:
            out[:, k, 0] = x[:, ny - k, m]
    return out


def field(kind, nz, ny, nx, seed):
    rng = np.random.default_rng(seed)
    f = rng.standard_normal((nz, ny, nx))
    if kind == "spectrum":
        j, i = np.ogrid[:ny, :nx]
        return f / (np.maximum(np.minimum(j, ny - j), 0.5) * np.maximum(np.minimum(i, nx - i), 0.5)) ** 2
    f *= 1e-9
    f[np.arange(nz), rng.integers(0, ny, nz), rng.integers(0, nx, nz)] += 1.0
    return f


def check(chanfs, nx, ny, kind):
    nz = 3
    f = field(kind, nz, ny, nx, nx + ny)
    ref = packed(f)
    with chanfs.Plan(nx, ny, nz, 2.0, 1.0, np.full(nz, 0.5)) as plan:
        got = plan.spectral_forward(torch.from_numpy(f).cuda()).cpu().numpy().view(np.complex128)
        s = torch.from_numpy(ref.astype(np.complex128).view(np.float64).reshape(nz, ny, nx)).cuda()
        back = plan.spectral_inverse(s).cpu().numpy()
        assert plan.check() == 0
    # each transform within 0.6 log2(n) 2^-53 of the exact one in L2, and one rounding between them
    tol = (0.6 * np.log2(nx * ny) + 1) * 2.0**-53
    for z in range(nz):
        norm = lambda a: float(np.sqrt(np.sum(np.abs(a) ** 2)))
        assert norm(got[z].reshape(ref[z].shape) - ref[z]) < tol * norm(ref[z]), z
        assert norm(back[z] - f[z].astype(np.longdouble)) < tol * norm(f[z]), z


@pytest.mark.parametrize("kind", ["spectrum", "one value"])
@pytest.mark.parametrize("nx,ny", [(162, 3), (486, 3), (972, 3), (1458, 3), (1944, 3), (2916, 3), (3888, 3), (16, 81),
                                   (24, 243), (16, 486), (36, 729)])
def test_lengths_of_many_radix_3_passes(chanfs, nx, ny, kind):
    check(chanfs, nx, ny, kind)


def same_values(a, b):
    return np.array_equal(a, b)  # (-0 and 0 alike)


@pytest.mark.parametrize("nx,ny", [(512, 3), (216, 48), (162, 27), (32, 3), (96, 243), (1536, 4), (24, 9), (64, 16)])
def test_powers_of_two_come_out_as_they_went_in(chanfs, nx, ny):
    """Every plane times its own power of two, near and far from 1: the same bits times that power, both ways.
    Planes of one power fill blocks of lines; with few lines per plane, blocks hold several powers."""
    e = np.array([0, 100, -100, 3, -300, 600, -700, 900, -950, 91, -91])
    nz = e.size
    f = np.random.default_rng(nx * ny).standard_normal((nz, ny, nx))
    f[2, :, nx // 2:] = 0.0  # (lone threads with nothing but zeros, beside a far line)
    f[3] *= 1e-40            # (a far line, as its own power leaves it)
    g = np.ldexp(f, e[:, None, None])
    with chanfs.Plan(nx, ny, nz, 2.0, 1.0, np.full(nz, 0.5)) as plan:
        base = plan.spectral_forward(torch.from_numpy(f).cuda())
        back = plan.spectral_inverse(base).cpu().numpy()
        base = base.cpu().numpy()
        s = plan.spectral_forward(torch.from_numpy(g).cuda()).cpu().numpy()
        t = plan.spectral_inverse(torch.from_numpy(np.ldexp(base, e[:, None, None])).cuda()).cpu().numpy()
        tiny = np.random.default_rng(1).integers(-9, 10, f.shape).astype(float)
        tiny[1] = 0.0
        x = lambda f: plan.poisson_stage(X_FORWARD, torch.from_numpy(f).cuda()).cpu().numpy()
        base_tiny, low = x(tiny), x(np.ldexp(tiny, -1074))
        assert plan.check() == 0
    assert same_values(s, np.ldexp(base, e[:, None, None]))
    assert same_values(t, np.ldexp(back, e[:, None, None]))
    assert not low[1].any()
    # subnormal data along x: the result rounded once to the units of the type (and once before, to 53 bits)
    assert np.max(np.abs(np.ldexp(low, 1074) - base_tiny)) <= 0.5 + 2.0**-40


@pytest.mark.parametrize("ybc", [0, 1, 2])
@pytest.mark.parametrize("nx,ny", [(64, 16), (54, 27), (36, 48), (72, 243), (48, 162), (128, 512)])
def test_columns_of_a_tile_keep_their_own_powers(chanfs, nx, ny, ybc):
    """The y transforms alone, neighbouring columns far apart in magnitude."""
    nz = 3
    rng = np.random.default_rng(nx + ny)
    e = np.repeat(rng.choice([0, 0, 120, -120, 700, -800], nx // 2), 2)
    f = rng.standard_normal((nz, ny, nx))
    with chanfs.Plan(nx, ny, nz, 2.0, 1.0, np.full(nz, 0.5), 0, 0, ybc) as plan:
        for stage in (Y_FORWARD, Y_INVERSE):
            base = plan.poisson_stage(stage, torch.from_numpy(f).cuda()).cpu().numpy()
            got = plan.poisson_stage(stage, torch.from_numpy(np.ldexp(f, e)).cuda()).cpu().numpy()
            assert same_values(got, np.ldexp(base, e)), stage
        assert plan.check() == 0


def test_far_long_columns_keep_their_bits(chanfs):
    """White noise times 2^-100 along 768 and 1024 points, which the line's sum scales."""
    for ny in (768, 1024):
        f = np.random.default_rng(ny).standard_normal((3, ny, 16))
        ref = packed(f)
        with chanfs.Plan(16, ny, 3, 2.0, 1.0, np.full(3, 0.5)) as plan:
            s = plan.spectral_forward(torch.from_numpy(np.ldexp(f, -100)).cuda()).cpu().numpy()
        got = np.ldexp(s, 100).view(np.complex128).reshape(ref.shape)
        err = float(np.sqrt(np.sum(np.abs(got - ref) ** 2) / np.sum(np.abs(ref) ** 2)))
        assert err < 3 * 2.0**-53  # (the fixed-point error of white noise is 1.5 at 4096)


@pytest.mark.parametrize("ny", [972, 1296, 1458, 1944, 2048, 2187, 2916, 3072, 3888, 4096])
def test_default_plans_transform_long_columns(chanfs, ny):
    """Every length runs on a plan as it is made: one to four columns per tile, compiled and general kernels."""
    check(chanfs, 18, ny, "spectrum")


@pytest.mark.parametrize("ybc", [1, 2])
@pytest.mark.parametrize("ny", [384, 432, 768, 1536, 2187, 4096])
def test_default_plans_solve_between_walls(chanfs, ny, ybc):
    nx, nz = 16 if ny % 2 else 4, 3  # (an odd count of rows asks for eight columns)
    dz = synth.tanh_dz(nz, 1.4)
    f = synth.normal(ny + ybc, (nz, ny, nx))
    if ybc == 1:
        f = synth.remove_weighted_mean(f, dz)
    ref = oracle.poisson_solve_walls(f, 2.0, 1.0, dz, 0, ybc)
    with chanfs.Plan(nx, ny, nz, 2.0, 1.0, dz, 0, 0, ybc) as plan:
        p = plan.poisson_solve(torch.from_numpy(f).cuda()).cpu().numpy()
        assert plan.check() == 0
    assert np.max(np.abs(p - ref)) / np.max(np.abs(ref)) < 1e-12  # (as the z sweeps' test)


@pytest.mark.parametrize("ny", [2048, 2187])
def test_a_tuned_plan_keeps_the_bits_and_the_choice(chanfs, ny):
    nx, nz = 18, 4
    f = torch.from_numpy(synth.normal(ny, (nz, ny, nx))).cuda()
    with chanfs.Plan(nx, ny, nz, 2.0, 1.0, np.full(nz, 0.5)) as plan:
        before = plan.spectral_forward(f)
        chosen = plan.autotune()
        assert torch.equal(before, plan.spectral_forward(f))
        assert plan.autotune() == chosen
        p = plan.poisson_solve(f)
        assert plan.check() == 0 and bool(torch.isfinite(p).all())
