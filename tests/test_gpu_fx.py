"""The fixed-point DFT of double plans (csrc/fx.cuh) against numpy's FFT in long double.

The bar: the row pass and the column pass each round their results to double once (2^-53
each, uniformly distributed: 2^-53/sqrt(3) in the 2-norm), and their fixed-point stages add
at most 2^-58 of a block's largest value per stage, which for N points is at most sqrt(N)
times the block's rms: below 2^-53 again for up to five stages and 2048 points.  Together
below 3 2^-53 in the relative 2-norm; the bar is 4 2^-53.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
BAR = 4 * 2.0 ** -53

KINDS = {
    "noise": lambda x, y, rng: rng.standard_normal((y.size, x.size)),
    "smooth": lambda x, y, rng: np.exp(np.sin(3 * x) + np.cos(2 * y)),
    "point": lambda x, y, rng: 1.3 * ((x == x[0, x.size // 5]) & (y == y[y.size // 3, 0])),
    "range": lambda x, y, rng: (rng.standard_normal((y.size, x.size))
                                * 10.0 ** rng.uniform(-12, 12, (y.size, x.size))),
}


def plan_of(nx, ny):
    from paper_2010_03901_gb300 import fc2d
    n = min(nx, ny)
    h = 2.0 / (0.45 * n)  # the unit disk, off the grid's centre
    return fc2d.fc2d_plan(np.array([[0, 1.0], [0, 0], [0, 0], [0, 1.0]]),
                          (-0.5 * nx * h + 0.3 * h, -0.5 * ny * h + 0.2 * h, h, nx, ny),
                          dict(B=256, k1=min(0.012, h)))


def spectrum(plan, f):
    import torch
    t = torch.tensor(f, dtype=torch.float64, device="cuda")
    out = torch.full((len(f), plan.ny, plan.nx // 2 + 1, 2), 7.0, dtype=torch.float64, device="cuda")
    plan.fc2d_coeffs(len(f), t, out)
    plan.fc2d_sync_status()
    got = out.cpu().numpy()
    return got[..., 0] + 1j * got[..., 1]


@pytest.mark.parametrize("nx,ny", [(64, 64), (128, 1024), (256, 128), (512, 256), (1024, 512),
                                   (2048, 64), (4096, 128), (128, 2048), (128, 4096), (8192, 64),
                                   # every radix of the other sizes, first and last; one, two
                                   # and many stages; one power-of-two side
                                   (60, 90), (96, 72), (100, 50), (162, 486), (250, 750), (128, 1200),
                                   (1728, 64), (2160, 80), (4374, 54), (540, 2048), (72, 3750)])
def test_against_long_double(nx, ny):
    fft = pytest.importorskip("scipy.fft")
    plan = plan_of(nx, ny)
    rng = np.random.default_rng(nx + ny)
    x, y = np.linspace(-1, 1, nx)[None, :], np.linspace(-1, 1, ny)[:, None]
    f = np.stack([fn(x, y, rng) * np.ones((ny, nx)) for fn in KINDS.values()])
    got = spectrum(plan, f)
    for k, name in enumerate(KINDS):
        ref = fft.rfft2(f[k].astype(np.longdouble)) / (nx * ny)
        err = np.sqrt(float((np.abs(got[k] - ref) ** 2).sum() / (np.abs(ref) ** 2).sum()))
        assert err < BAR, (name, err)


@pytest.mark.parametrize("nx,ny", [(64, 64), (256, 128)])
def test_edges_of_the_range(nx, ny):
    """Zero fields, powers of two far from 1 (exact scalings of the same field, down to
    subnormal results), and non-finite values, which stay within their own field."""
    plan = plan_of(nx, ny)
    rng = np.random.default_rng(5)
    a = rng.standard_normal((ny, nx))
    big, small, tiny = 2.0 ** 1000, 2.0 ** -1000, 2.0 ** -1060
    bad, inf = a.copy(), a.copy()
    bad[ny // 2, 3], inf[1, nx - 1] = np.nan, -np.inf
    got = spectrum(plan, np.stack([a, 0 * a, a * big, a * small, bad, inf, a * tiny, a]))
    assert np.array_equal(got[0], got[7]) and not got[1].any()
    assert np.array_equal(got[2], got[0] * big)
    assert np.array_equal(got[3], got[0] * small)
    assert np.isnan(got[4].real).all() and np.isnan(got[5].imag).all()
    # inputs near 2^-1060 keep 14 bits or so: two roundings to the smallest subnormal each
    assert np.abs(got[6] - got[0] * tiny).max() <= 2.0 ** -1074 * np.sqrt(nx * ny)
