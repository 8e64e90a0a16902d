"""Double-layer sums of the Poisson solver against long double sums of the same terms.

With f = 0 the solution is the double-layer potential alone: at the inside points away
from the curve its trapezoidal sum over the n_b nodes, nearer (but not in the innermost
band) over the 8 n_b refined ones, with the density that the call returns.  Grids and node
counts cover sums without expansions, one to many levels of boxes, more nodes than grid
lines and a grid that is not square."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

REFINE = 8


def direct(z, zn, q):
    """sum_k Im q_k / (z - z_k) and the sum of the terms' moduli, in long double"""
    v, a = np.empty(len(z), np.longdouble), np.empty(len(z), np.longdouble)
    for k in range(0, len(z), 256):
        t = q[None] / (z[k:k + 256, None] - zn[None])
        v[k:k + 256], a[k:k + 256] = t.imag.sum(1), np.abs(t).sum(1)
    return v, a


@pytest.mark.parametrize("name,nb", [("disk128", 64), ("disk128", 128), ("star200", 0),
                                     ("kite160x144", 0), ("disk64", 1024), ("star200", 2000)])
def test_double_layer_sums(name, nb):
    torch = pytest.importorskip("torch")
    from oracle import geometry as OG
    from paper_2010_03901_gb300 import fc2d
    w = W.workload(name)
    g, p = w.grid, w.params
    plan = fc2d.fc2d_plan(w.boundary.arrays(), (g.a0, g.b0, g.h, g.nx, g.ny),
                          dict(B=p.B, k1=p.k1))
    plan.fc2d_poisson_plan(nb)
    xy = plan.fc2d_poisson_nodes()
    n = len(xy)
    th = 2 * np.pi * np.arange(n) / n
    dev = torch.device("cuda:0")
    bxy = plan.fc2d_boundary_points()
    fg = torch.zeros((1, g.ny, g.nx), dtype=torch.float64, device=dev)
    fb = torch.zeros((1, len(bxy)), dtype=torch.float64, device=dev)
    gn = torch.tensor((np.cos(2 * th) + 0.3 * np.sin(3 * th) + 1.0)[None], device=dev)
    u = torch.zeros_like(fg)
    phi = torch.zeros((1, n), dtype=torch.float64, device=dev)
    plan.fc2d_poisson(1, fg, fb, gn, u, phi)
    plan.fc2d_sync_status()
    u, phi = u.cpu().numpy()[0], phi.cpu().numpy()[0]

    geo = OG.build_geometry(w)
    curve = geo.curve
    m = REFINE * n
    t = 2 * np.pi * np.arange(m) / m

    def at(t, d):
        return curve.x(t, d).astype(np.longdouble) + 1j * curve.y(t, d).astype(np.longdouble)

    h = np.fft.rfft(phi) / n
    if n % 2 == 0:
        h[-1] *= 0.5
    fine = np.fft.irfft(np.concatenate([h, np.zeros(m // 2 + 1 - len(h))]), m) * m
    zn, zr = at(th, 0), at(t, 0)
    qn = at(th, 1) * phi / n
    qr = at(t, 1) * fine / m
    s = 2 * np.pi / n * float(np.abs(at(2 * np.pi * np.arange(4096) / 4096, 1)).max())
    jj, ii = np.nonzero(geo.inside.reshape(g.ny, g.nx))
    sel = np.arange(len(ii))[:: max(1, len(ii) // 1500)]
    ii, jj = ii[sel], jj[sel]
    z = (g.a0 + g.h * ii) + 1j * (g.b0 + g.h * jj)
    dense = at(2 * np.pi * np.arange(8 * m) / (8 * m), 0).astype(complex)
    dist = np.array([np.abs(v - dense).min() for v in z])
    margin = 2 * np.pi / (8 * m) * s * n  # of the sampled distance
    far = dist > 5 * s + margin
    mid = (dist < 5 * s - margin) & (dist > 5 * s / REFINE + margin)
    assert far.any() or mid.any()
    # Near terms: double-float coordinates, products and reciprocal, 2^-44 of a term's size in
    # all; expansions: 2^-52 of it.  The refined density adds its own rounding, n/2 terms of at
    # most max|phi|, to both sides.
    for pick, zz, q, extra in ((far, zn, qn, 0.0), (mid, zr, qr, n * 2.0 ** -52)):
        if not pick.any():
            continue
        v, a = direct(z[pick].astype(np.clongdouble), zz, q)
        got = u[jj[pick], ii[pick]]
        size = float(np.abs(phi).max() / m * np.abs(at(t, 1)).max())
        near = size * m / np.maximum(dist[pick], g.h / 8)
        bound = (2.0 ** -44 + 2.0 ** -50 / dist[pick]) * a + extra * near + 2.0 ** -52 * np.abs(v)
        err = np.abs(got - v)
        print(name, nb, int(pick.sum()), float((err / bound).max()), float((err / a).max()))
        assert (err <= bound).all()


@pytest.mark.parametrize("name,nb", [("disk128", 40), ("star200", 200), ("star200", 333),
                                     ("kite160x144", 1201), ("star200", 3000)])
def test_boundary_density(name, nb):
    """The density solves the Nystrom system: node counts below, at and above one row per warp
    and block, odd ones among them."""
    torch = pytest.importorskip("torch")
    from oracle import geometry as OG
    from oracle import poisson as OP
    from paper_2010_03901_gb300 import fc2d
    w = W.workload(name)
    g, p = w.grid, w.params
    plan = fc2d.fc2d_plan(w.boundary.arrays(), (g.a0, g.b0, g.h, g.nx, g.ny),
                          dict(B=p.B, k1=p.k1))
    plan.fc2d_poisson_plan(nb)
    dev = torch.device("cuda:0")
    n = len(plan.fc2d_poisson_nodes())
    fg = torch.zeros((2, g.ny, g.nx), dtype=torch.float64, device=dev)
    fb = torch.zeros((2, len(plan.fc2d_boundary_points())), dtype=torch.float64, device=dev)
    th = 2 * np.pi * np.arange(n) / n
    gn = np.stack([np.cos(2 * th) + 0.3 * np.sin(3 * th) + 1.0, np.zeros(n)])
    u, phi = torch.zeros_like(fg), torch.ones((2, n), dtype=torch.float64, device=dev)
    plan.fc2d_poisson(2, fg, fb, torch.tensor(gn, device=dev), u, phi)
    plan.fc2d_sync_status()
    phi = phi.cpu().numpy()
    assert (phi[1] == 0).all() and float(u[1].abs().max()) == 0.0
    A = OP.bie_matrix(OG.build_geometry(w).curve, n)
    res = np.linalg.norm(A @ phi[0] - gn[0])
    # the stopping rule, and n products and sums per row in either program
    bound = 1e-14 * np.linalg.norm(gn[0]) + n * 2.0 ** -52 * np.linalg.norm(np.abs(A) @ np.abs(phi[0]))
    print(name, n, res / bound)
    assert res <= bound
