"""The integer strip values of double plans (csrc/fx_strip.cu), through fc2d_extend, against
the double-precision kernels behind fc2d_blend and fc2d_interp.

Both start from the same Gram coefficients (the same FP64 operations), so they differ by the
rounding of A_r c and of the interpolation alone: the bar of the extended grid for each order
(3e-11 of max |F| for d <= 5, 1.5e-7 for d = 10, see tests/test_gpu_parity.py and
tests/test_gpu_high_order.py) covers the two kernels' summation orders with room to spare.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def make(d, M, n_r, C, n=96):
    from paper_2010_03901_gb300 import fc2d
    h = 2.0 / (0.5 * n)
    k1 = min(0.012, 0.3 / C)
    return fc2d.fc2d_plan(np.array([[0, 1.0], [0, 0], [0, 0], [0, 1.0]]),
                          (-0.5 * n * h + 0.3 * h, -0.5 * n * h + 0.2 * h, h, n, n),
                          dict(d=d, M=M, n_r=n_r, C=C, B=250, k1=k1))


def extend(plan, f, b):
    import torch
    ext = torch.zeros_like(f)
    plan.fc2d_extend(len(f), f, b, ext)
    plan.fc2d_sync_status()
    return ext.reshape(len(f), -1)[:, torch.tensor(plan.fc2d_strip_points()[0].astype(np.int64), device="cuda")]


def fields(plan, n_f):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(4)
    f = torch.randn((n_f, plan.ny, plan.nx), dtype=torch.float64, device="cuda", generator=gen)
    b = torch.randn((n_f, plan.n_bdry), dtype=torch.float64, device="cuda", generator=gen)
    return f, b


@pytest.mark.parametrize("d,M,n_r,C", [(2, 2, 6, 27), (4, 7, 6, 27), (5, 8, 6, 27), (5, 8, 16, 27),
                                       (5, 9, 8, 25), (3, 16, 5, 27), (8, 11, 6, 27), (10, 13, 6, 27)])
@pytest.mark.parametrize("bdry", [True, False])
def test_against_the_double_kernels(d, M, n_r, C, bdry):
    import torch
    plan = make(d, M, n_r, C)
    f, b = fields(plan, 2)
    b = b if bdry else None
    F = torch.zeros((2, plan.params["B"], C * n_r + 1), dtype=torch.float64, device="cuda")
    vals = torch.zeros((2, plan.n_strip), dtype=torch.float64, device="cuda")
    plan.fc2d_blend(2, f, b, F)
    plan.fc2d_interp(2, F, vals)
    got = extend(plan, f, b)
    assert float((got - vals).abs().max()) < (3e-11 if d <= 5 else 1.5e-7) * float(F.abs().max())


def test_scaling_and_non_finite_values():
    """Powers of two scale the strip exactly; a NaN or infinity stays within its function and
    reaches every strip point whose normals read it."""
    import torch
    plan = make(5, 8, 6, 27)
    f, b = fields(plan, 1)
    ref = extend(plan, f, b)
    for k in (-900, -1, 3, 900):
        s = 2.0 ** k
        assert torch.equal(extend(plan, f * s, b * s), ref * s)
    assert not extend(plan, 0 * f, 0 * b).any()
    f2, b2 = torch.cat([f, f]), torch.cat([b, b])
    b2[0, 3] = float("nan")  # the foot of normal 3
    got = extend(plan, f2, b2)
    assert torch.equal(got[1], ref[0]) and bool(torch.isnan(got[0]).any()) and not bool(torch.isnan(got[0]).all())
    theta = plan.fc2d_strip_points()[1]
    touched = np.abs((theta / (2 * np.pi) * 250 - 3 + 125) % 250 - 125) < 3  # within the 8 normals
    assert bool(torch.isnan(got[0][torch.tensor(touched, device="cuda")]).all())


@pytest.mark.parametrize("M", [7, 8, 13])
@pytest.mark.parametrize("tiny", [0.0, 2.0 ** -300])
def test_normals_that_vanish_beside_others(M, tiny):
    """Ten boundary data, 25 normals apart, all other data zero (or far below it): the normals without data add
    nothing, so strip values of the opposite datum are the opposite ones.  Every rounding is to
    nearest, symmetric but for ties; a unit lost per vanishing normal shows where the weight of
    the datum's normals is below 2^-8 and the value keeps its last bits."""
    import torch
    plan = make(5, M, 6, 27)
    f, b = (tiny * x for x in fields(plan, 1))
    b[0, ::25] = 1.2345678901234567
    got, opp = extend(plan, f, b)[0], extend(plan, -f, -b)[0]
    top = float(got.abs().max())
    small = (got != 0) & (got.abs() < 2.0 ** -9 * top) & (got.abs() > 2.0 ** -60 * top)
    assert int(small.sum()) > 20
    assert float((got + opp)[small].ne(0).double().mean()) < 0.05
