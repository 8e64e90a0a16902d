"""The fixed-point modal solutions of Fourier Forwarding (csrc/fx_wave.cu) against the same
formulas in long double, from the plan's own extensions of u and u_t.

The bar: forward transforms, time factors and inverse transforms each within 3 2^-53 (see
test_gpu_fx.py; the factors are 60-bit) of operators of norm 1 and t (for u), or w_max and
1 (for u_t): 10 2^-53 (|F| + t |G|) and 10 2^-53 (w_max |F| + |G|) in the 2-norm.  The phase
w t is exact to 2^-64 of a turn per cell travelled, so long times keep the bar.
"""
import numpy as np
import pytest

from test_gpu_fx import plan_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(512, 512), (64, 512), (1024, 512), (512, 1024), (128, 2048),
                                   (64, 4096), (90, 100), (162, 250), (360, 72), (1200, 512), (128, 720)])
@pytest.mark.parametrize("cells", [0.0, 1e-7, 0.01, 0.5, 8.0, 1000.25])
def test_modal_solutions(nx, ny, cells):
    torch = pytest.importorskip("torch")
    fft = pytest.importorskip("scipy.fft")
    plan = plan_of(nx, ny)
    n = min(nx, ny)
    h, c = 2.0 / (0.45 * n), 1.7
    t = cells * h / c
    rng = np.random.default_rng(nx + ny)
    x = (np.arange(nx) - 0.5 * nx) * h
    y = (np.arange(ny) - 0.5 * ny) * h
    xy = plan.fc2d_boundary_points().T
    fields = []
    for amp in (1.0, 1.0 / max(t, h)):
        k, s = rng.uniform(2, 8, 4), rng.uniform(0, 6, 4)
        fn = lambda X, Y: amp * sum(np.cos(kk * (X * np.cos(ss) + Y * np.sin(ss)) + ss) for kk, ss in zip(k, s))  # noqa: E731,B023
        fields.append((fn(x[None, :], y[:, None]), fn(xy[0], xy[1])))
    T = lambda a: torch.tensor(a[None], dtype=torch.float64, device="cuda")  # noqa: E731
    (u, ub), (v, vb) = [(T(a), T(b)) for a, b in fields]
    ext = []
    for a, b in ((u, ub), (v, vb)):
        e = torch.zeros_like(a)
        plan.fc2d_extend(1, a, b, e)
        ext.append(e.cpu().numpy()[0].astype(np.longdouble))
    got, got_t = torch.zeros_like(u), torch.zeros_like(u)
    plan.fc2d_wave_interior(1, c, t, u, ub, v, vb, got, got_t)
    plan.fc2d_sync_status()
    F, G = fft.rfft2(ext[0]), fft.rfft2(ext[1])
    L = np.longdouble
    l = np.arange(nx // 2 + 1, dtype=L) / nx
    m = np.abs(np.fft.fftfreq(ny) * ny).astype(L) / ny
    two_pi = 2 * L("3.14159265358979323846264338327950288")
    w = two_pi * L(c) * np.sqrt(l[None, :] ** 2 + m[:, None] ** 2) / L(h)
    wt = two_pi * ((w / two_pi * L(t)) % 1)
    sw = np.where(w > 0, np.sin(wt) / np.where(w > 0, w, 1), L(t))
    ref = fft.irfft2(F * np.cos(wt) + G * sw, s=(ny, nx))
    ref_t = fft.irfft2(G * np.cos(wt) - F * w * np.sin(wt), s=(ny, nx))
    norm = lambda a: float(np.sqrt((np.abs(a) ** 2).sum()))  # noqa: E731
    f, g = norm(ext[0]), norm(ext[1])
    # wt itself, in the reference, from the doubles h, c and t: c t/h is rounded once
    slack = float(w.max()) * t * 2.0 ** -52
    eps = 10 * 2.0 ** -53 + slack
    assert norm(got.cpu().numpy()[0] - ref) < eps * (f + t * g)
    assert norm(got_t.cpu().numpy()[0] - ref_t) < eps * (float(w.max()) * f + g)


def test_first_call_inside_a_capture():
    """A plan whose workspace an earlier call has grown takes its first wave call inside a stream
    capture, and without waiting for other streams: equal to another plan's call bit for bit."""
    torch = pytest.importorskip("torch")
    gen = torch.Generator(device="cuda").manual_seed(12)
    plans = [plan_of(256, 192) for _ in range(3)]
    rnd = lambda *s: torch.randn(s, dtype=torch.float64, device="cuda", generator=gen)  # noqa: E731
    fields = [rnd(16, p, q) for p, q in [(192, 256)] * 2]
    bdry = [rnd(16, plans[0].n_bdry) for _ in range(2)]
    spec = torch.zeros((16, 192, 129, 2), dtype=torch.float64, device="cuda")
    for p in plans:
        p.fc2d_extend_coeffs(16, fields[0], bdry[0], spec)
    outs = [(torch.zeros_like(fields[0][:1]), torch.zeros_like(fields[0][:1])) for _ in plans]

    def call(k, **kw):
        plans[k].fc2d_wave_interior(1, 1.3, 0.02, fields[0][:1], bdry[0][:1], fields[1][:1], bdry[1][:1],
                                    *outs[k], **kw)

    call(0)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(1)
    graph.replay()
    mine, other, busy = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Event()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(400_000_000)  # about 0.2 s
        busy.record()
    call(2, stream=mine)
    waited = busy.query()
    torch.cuda.synchronize()
    assert not waited
    for got in outs[1:]:
        assert torch.equal(outs[0][0], got[0]) and torch.equal(outs[0][1], got[1])


@pytest.mark.parametrize("nx,ny", [(512, 512), (90, 100), (1200, 512)])
@pytest.mark.parametrize("cells", [1e-9, 1e-5, 1e-3, 0.05, 0.2])
@pytest.mark.parametrize("amp", [(1, 0), (0, 1), (1, 1)])
def test_times_below_a_cell(nx, ny, cells, amp):
    """u and t u_t of the same size (or one of them zero) at times in which a wave crosses a small
    part of a cell.  The bars of test_modal_solutions with u_t's factor at that time: w sin(w t)
    is at most w min(1, w t)."""
    torch = pytest.importorskip("torch")
    fft = pytest.importorskip("scipy.fft")
    plan = plan_of(nx, ny)
    h, c = 2.0 / (0.45 * min(nx, ny)), 1.7
    t = cells * h / c
    x, y = (np.arange(nx) - 0.5 * nx) * h, (np.arange(ny) - 0.5 * ny) * h
    xy = plan.fc2d_boundary_points().T
    fn = lambda X, Y: np.cos(2.1 * X + 0.3) * np.cos(1.7 * Y - 0.2)  # noqa: E731
    T = lambda a: torch.tensor(a[None], dtype=torch.float64, device="cuda")  # noqa: E731
    data, ext = [], []
    for a in (amp[0], amp[1] / t):
        data += [T(a * fn(x[None, :], y[:, None])), T(a * fn(xy[0], xy[1]))]
        e = torch.zeros_like(data[0])
        plan.fc2d_extend(1, data[-2], data[-1], e)
        ext.append(e.cpu().numpy()[0].astype(np.longdouble))
    got, got_t = data[0], data[2]  # in place
    plan.fc2d_wave_interior(1, c, t, *data, got, got_t)
    plan.fc2d_sync_status()
    F, G = fft.rfft2(ext[0]), fft.rfft2(ext[1])
    L = np.longdouble
    l, m = np.arange(nx // 2 + 1, dtype=L) / nx, np.abs(np.fft.fftfreq(ny) * ny).astype(L) / ny
    w = 2 * L("3.14159265358979323846264338327950288") * L(c) * np.sqrt(l[None, :] ** 2 + m[:, None] ** 2) / L(h)
    sw = np.where(w > 0, np.sin(w * L(t)) / np.where(w > 0, w, 1), L(t))
    ref = fft.irfft2(F * np.cos(w * L(t)) + G * sw, s=(ny, nx))
    ref_t = fft.irfft2(G * np.cos(w * L(t)) - F * w * np.sin(w * L(t)), s=(ny, nx))
    norm = lambda a: float(np.sqrt((np.abs(a) ** 2).sum()))  # noqa: E731
    f, g, top = norm(ext[0]), norm(ext[1]), float(w.max())
    eps = 10 * 2.0 ** -53 + top * t * 2.0 ** -52
    e = norm(got.cpu().numpy()[0] - ref), norm(got_t.cpu().numpy()[0] - ref_t)
    bar = eps * (f + t * g), eps * (top * min(1.0, top * t) * f + g)
    print(nx, ny, cells, amp, e[0] / bar[0], e[1] / bar[1])
    assert e[0] < bar[0] and e[1] < bar[1]


def test_times_without_a_phase():
    """Time zero gives the data's extensions, times and speeds whose phase is not finite NaN."""
    import torch
    plan = plan_of(128, 96)
    gen = torch.Generator(device="cuda").manual_seed(13)
    rnd = lambda *s: torch.randn(s, dtype=torch.float64, device="cuda", generator=gen)  # noqa: E731
    u, v, ub, vb = rnd(2, 96, 128), rnd(2, 96, 128), rnd(2, plan.n_bdry), rnd(2, plan.n_bdry)
    a, b, e = torch.zeros_like(u), torch.zeros_like(u), torch.zeros_like(u)
    for c, t in ((1.0, float("inf")), (float("inf"), 1.0), (1e200, 1e200)):
        plan.fc2d_wave_interior(2, c, t, u, ub, v, vb, a, b)
        assert bool(torch.isnan(a).all()) and bool(torch.isnan(b).all()), (c, t)
    plan.fc2d_wave_interior(2, 1.0, 1e25, u, ub, v, vb, a, b)
    assert bool(torch.isfinite(a).all()) and bool(torch.isfinite(b).all())
    plan.fc2d_wave_interior(2, 1.0, 0.0, u, ub, v, vb, a, b)
    for got, f, fb in ((a, u, ub), (b, v, vb)):
        plan.fc2d_extend(2, f, fb, e)
        # each transform within 3 2^-53 in the 2-norm
        assert float((got - e).norm() / e.norm()) < 6 * 2.0 ** -53


def test_the_tallest_grid():
    """ny up to 4842 in both wave calls (4800 = 2^6 3 5^2 is the largest such size), one message
    above."""
    import torch
    from paper_2010_03901_gb300 import fc2d
    z = lambda p: torch.zeros((1, p.ny, p.nx), dtype=torch.float64, device="cuda")  # noqa: E731
    tall = plan_of(64, 4860)
    u = z(tall)
    b = torch.zeros((1, tall.n_bdry), dtype=torch.float64, device="cuda")
    for call in (lambda: tall.fc2d_wave_interior(1, 1.0, 0.1, u, b, u, b, z(tall), z(tall)),
                 lambda: tall.fc2d_forward_wave(1, 1.0, 4, 1, u, u.clone())):
        with pytest.raises(fc2d.Fc2dError, match="ny <= 4842") as e:
            call()
        assert e.value.status == 7
    plan = plan_of(64, 4800)
    u, ut = torch.ones_like(z(plan)), z(plan)
    b = torch.ones((1, plan.n_bdry), dtype=torch.float64, device="cuda")
    out, ext = [z(plan), z(plan)], z(plan)
    plan.fc2d_wave_interior(1, 1.0, 0.0, u, b, ut, 0 * b, *out)
    plan.fc2d_extend(1, u, b, ext)
    assert float((out[0] - ext).norm() / ext.norm()) < 6 * 2.0 ** -53


@pytest.mark.parametrize("nx,ny", [(512, 512), (1024, 1024), (2048, 2048), (64, 4800), (1200, 1728)])
def test_transforms_of_smooth_fields(nx, ny):
    """At time 0 the call is one forward and one inverse transform of the extension.  Four passes
    round to double once each (2^-53/sqrt(3) in the 2-norm), the fixed-point stages add less than
    2^-53 for spectra with a few large modes too: below 2.2 2^-53 together, the bar is 3 2^-53 (FP64
    transforms: 4 2^-53)."""
    torch = pytest.importorskip("torch")
    plan = plan_of(nx, ny)
    h = 2.0 / (0.45 * min(nx, ny))
    x, y = (np.arange(nx) - 0.5 * nx) * h, (np.arange(ny) - 0.5 * ny) * h
    xy = plan.fc2d_boundary_points().T
    fn = lambda X, Y: np.cos(2.1 * X + 0.3) * np.cos(1.7 * Y - 0.2)  # noqa: E731
    u, ub = (torch.tensor(a[None], dtype=torch.float64, device="cuda")
             for a in (fn(x[None, :], y[:, None]), fn(xy[0], xy[1])))
    out, ext = [torch.zeros_like(u), torch.zeros_like(u)], torch.zeros_like(u)
    plan.fc2d_wave_interior(1, 1.0, 0.0, u, ub, 0 * u, 0 * ub, *out)
    plan.fc2d_extend(1, u, ub, ext)
    err = float((out[0] - ext).norm() / ext.norm())
    print(nx, ny, err * 2.0 ** 53)
    assert err < 3 * 2.0 ** -53


@pytest.mark.parametrize("nx,ny", [(512, 512), (64, 4096), (4096, 64)])
@pytest.mark.parametrize("cells", [8.0, 200.25])
def test_phases_after_many_cells(nx, ny, cells):
    """u from u alone: c t/h and the modes' frequencies carry two doubles, so that the phases add
    nothing to the error of the two transforms (the bar of test_transforms_of_smooth_fields, 3 2^-53 of the
    2-norm) however many turns they make; rounded to one double they add w t 2^-53."""
    torch = pytest.importorskip("torch")
    fft = pytest.importorskip("scipy.fft")
    plan = plan_of(nx, ny)
    h, c = 2.0 / (0.45 * min(nx, ny)), 1.7
    t = cells * h / c
    x, y = (np.arange(nx) - 0.5 * nx) * h, (np.arange(ny) - 0.5 * ny) * h
    xy = plan.fc2d_boundary_points().T
    fn = lambda X, Y: np.cos(2.1 * X + 0.3) * np.cos(1.7 * Y - 0.2)  # noqa: E731
    u, ub = (torch.tensor(a[None], dtype=torch.float64, device="cuda")
             for a in (fn(x[None, :], y[:, None]), fn(xy[0], xy[1])))
    got, got_t, ext = torch.zeros_like(u), torch.zeros_like(u), torch.zeros_like(u)
    plan.fc2d_wave_interior(1, c, t, u, ub, 0 * u, 0 * ub, got, got_t)
    plan.fc2d_extend(1, u, ub, ext)
    L = np.longdouble
    F = fft.rfft2(ext.cpu().numpy()[0].astype(L))
    l = np.arange(nx // 2 + 1).astype(L) / nx
    m = np.minimum(np.arange(ny), ny - np.arange(ny)).astype(L) / ny
    w = 2 * L("3.14159265358979323846264338327950288") * L(c) * np.sqrt(l[None, :] ** 2 + m[:, None] ** 2) / L(h)
    ref = fft.irfft2(F * np.cos(w * L(t)), s=(ny, nx))
    norm = lambda a: float(np.sqrt((np.abs(a) ** 2).sum()))  # noqa: E731
    err = norm(got.cpu().numpy()[0] - ref) / norm(ref)
    print(nx, ny, cells, err * 2.0 ** 53)
    assert err < 3 * 2.0 ** -53
