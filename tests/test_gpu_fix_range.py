"""GPU: the block fixed-point FP64 transforms on data whose values differ widely, against transforms in
extended precision: lengths of many radix-3 passes, columns like 1/k^2 (what the inverse transforms of a
Poisson solve receive) and columns with one dominant value."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
fft = pytest.importorskip("scipy.fft")
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
@pytest.mark.parametrize("nx,ny", [(162, 3), (486, 3), (972, 3), (1458, 3), (2916, 3), (3888, 3), (16, 81),
                                   (24, 243), (16, 486), (36, 729)])
def test_lengths_of_many_radix_3_passes(chanfs, nx, ny, kind):
    check(chanfs, nx, ny, kind)
