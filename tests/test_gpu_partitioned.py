"""The Poisson solve on a stream that has a part of the SMs only (a green context): GMRES, one
cooperative launch, then takes fewer blocks of more rows each."""
import ctypes as ct

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


class PartialStream:
    """A stream over at least n_sm SMs, by the driver API."""

    def __init__(self, n_sm):
        cu = self.cu = ct.CDLL("libcuda.so.1")
        self.ctx, self.cuda_stream = ct.c_void_p(), None
        dev, desc, stream, n = ct.c_int(), ct.c_void_p(), ct.c_void_p(), ct.c_uint(1)
        # CUdevResource: type, 92 bytes, then (type SM = 1) the SM count; 144 bytes in all
        every, part, rest = (ct.create_string_buffer(256) for _ in range(3))

        def call(name, *args):
            err = getattr(cu, name)(*args)
            if err:
                pytest.skip(f"{name} returned {err}")

        call("cuDeviceGet", ct.byref(dev), 0)
        call("cuDeviceGetDevResource", dev, every, 1)
        call("cuDevSmResourceSplitByCount", part, ct.byref(n), every, rest, 0, n_sm)
        self.n_sm = int.from_bytes(part.raw[96:100], "little")
        call("cuDevResourceGenerateDesc", ct.byref(desc), part, 1)
        call("cuGreenCtxCreate", ct.byref(self.ctx), desc, dev, 1)
        call("cuGreenCtxStreamCreate", ct.byref(stream), self.ctx, 1, 0)
        self.cuda_stream = stream.value

    def close(self):
        if self.cuda_stream:
            self.cu.cuStreamDestroy_v2(ct.c_void_p(self.cuda_stream))
        if self.ctx:
            self.cu.cuGreenCtxDestroy(self.ctx)


@pytest.mark.parametrize("n_sm,nb", [(8, 0), (8, 333), (40, 3000)])
def test_poisson_on_a_part_of_the_sms(n_sm, nb):
    torch = pytest.importorskip("torch")
    from oracle import geometry as OG
    from oracle import poisson as OP
    from paper_2010_03901_gb300 import fc2d
    w = W.workload("star200")
    g, p = w.grid, w.params
    plan = fc2d.fc2d_plan(w.boundary.arrays(), (g.a0, g.b0, g.h, g.nx, g.ny),
                          dict(B=p.B, k1=p.k1))
    plan.fc2d_poisson_plan(nb)
    n = len(plan.fc2d_poisson_nodes())
    fg = torch.zeros((1, g.ny, g.nx), dtype=torch.float64, device="cuda")
    fb = torch.zeros((1, len(plan.fc2d_boundary_points())), dtype=torch.float64, device="cuda")
    th = 2 * np.pi * np.arange(n) / n
    gn = np.cos(2 * th) + 0.3 * np.sin(3 * th) + 1.0
    gd = torch.tensor(gn[None], device="cuda")
    out = [(torch.zeros_like(fg), torch.zeros((1, n), dtype=torch.float64, device="cuda"))
           for _ in range(2)]
    torch.cuda.synchronize()
    part = PartialStream(n_sm)
    try:
        assert part.n_sm < torch.cuda.get_device_properties(0).multi_processor_count
        plan.fc2d_poisson(1, fg, fb, gd, *out[0], stream=part)
        torch.cuda.synchronize()
    finally:
        part.close()
    plan.fc2d_poisson(1, fg, fb, gd, *out[1])
    torch.cuda.synchronize()
    A = OP.bie_matrix(OG.build_geometry(w).curve, n)
    # the stopping rule, and n products and sums per row in either program
    for u, phi in out:
        f = phi.cpu().numpy()[0]
        bound = 1e-14 * np.linalg.norm(gn) + n * 2.0 ** -52 * np.linalg.norm(np.abs(A) @ np.abs(f))
        assert np.linalg.norm(A @ f - gn) <= bound
