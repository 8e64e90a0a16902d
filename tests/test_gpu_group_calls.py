"""Plan-group calls with changing arguments: direct launches, the capture of a repeated
call, replays of an older graph's arguments, changed function counts and boundary data, in
both forms, equal to separate calls bit for bit."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("form", ["branches", "persistent"])
def test_calls_in_any_order(form, precision):
    torch = pytest.importorskip("torch")
    from paper_2010_03901_gb300 import fc2d
    prec = fc2d.FC2D_FP64 if precision == "fp64" else fc2d.FC2D_MIXED
    out_t = torch.float64 if precision == "fp64" else torch.float32
    names = ["disk64", "star200", "kite160x144"]
    plans = []
    for name in names * 3:  # nine records: more than one launch of the persistent form's
        w = W.workload(name)
        g, p = w.grid, w.params
        plans.append(fc2d.fc2d_plan(w.boundary.arrays(), (g.a0, g.b0, g.h, g.nx, g.ny),
                                    dict(B=p.B, k1=p.k1), precision=prec))
    gen = torch.Generator(device="cuda").manual_seed(3)

    def fields(n_f):
        rnd = lambda *s: torch.randn(s, dtype=torch.float64, device="cuda", generator=gen)  # noqa: E731
        return (n_f, [rnd(n, p.ny, p.nx) for n, p in zip(n_f, plans)],
                [rnd(n, p.n_bdry) for n, p in zip(n_f, plans)])

    sets = [fields([1] * 9), fields([1] * 9), fields([1, 2, 3] * 3)]
    outs = [[torch.zeros((n, p.ny, p.nx // 2 + 1, 2), dtype=out_t, device="cuda")
             for n, p in zip(s[0], plans)] for s in sets]
    grp = fc2d.fc2d_group_create(plans)
    grp.fc2d_group_tuning_set(form, 256)
    for k, bdry in [(0, True), (1, True), (0, True), (0, True), (0, True), (1, True), (0, True),
                    (2, True), (2, False), (2, False), (0, True), (0, True)]:
        n_f, f, b = sets[k]
        b = b if bdry else None
        for o in outs[k]:
            o.fill_(7.0)
        grp.fc2d_group_extend_coeffs(n_f, f, b, outs[k])
        for i, p in enumerate(plans):
            ref = torch.zeros_like(outs[k][i])
            p.fc2d_extend_coeffs(n_f[i], f[i], b[i] if bdry else None, ref)
            assert torch.equal(ref, outs[k][i]), (k, bdry, i)
    grp.fc2d_group_destroy()


def mixed_plans(fc2d):
    plans = []
    for name in ["disk64", "star200", "kite160x144"]:
        w = W.workload(name)
        g, p = w.grid, w.params
        plans.append(fc2d.fc2d_plan(w.boundary.arrays(), (g.a0, g.b0, g.h, g.nx, g.ny),
                                    dict(B=p.B, k1=p.k1), precision=fc2d.FC2D_MIXED))
    return plans


def call_set(torch, plans, n_f, gen):
    rnd = lambda *s: torch.randn(s, dtype=torch.float64, device="cuda", generator=gen)  # noqa: E731
    f = [rnd(n, p.ny, p.nx) for n, p in zip(n_f, plans)]
    b = [rnd(n, p.n_bdry) for n, p in zip(n_f, plans)]
    out = [torch.zeros((n, p.ny, p.nx // 2 + 1, 2), dtype=torch.float32, device="cuda")
           for n, p in zip(n_f, plans)]
    return list(n_f), f, b, out


@pytest.mark.parametrize("form", ["branches", "persistent"])
@pytest.mark.parametrize("counts,grown", [(([3, 2, 3], [1, 1, 1]), False),
                                          (([1, 1, 1], [3, 2, 3]), True),
                                          (([2, 1, 3], [3, 1, 2]), True)])
def test_return_to_captured_arguments(form, counts, grown):
    """A call is repeated until it runs as a graph, calls with other function counts (fewer;
    more, with the workspaces already large enough; exchanged) replace the work items, then
    the first call's arguments come back: equal to separate calls bit for bit every time."""
    torch = pytest.importorskip("torch")
    from paper_2010_03901_gb300 import fc2d
    plans = mixed_plans(fc2d)
    gen = torch.Generator(device="cuda").manual_seed(9)
    sets = [call_set(torch, plans, n_f, gen) for n_f in counts]
    refs = []
    for n_f, f, b, out in sets if grown else sets[:1]:
        for i, p in enumerate(plans):  # the workspaces take their final size
            p.fc2d_extend_coeffs(n_f[i], f[i], b[i], out[i])
    for n_f, f, b, out in sets:
        refs.append([torch.zeros_like(o) for o in out])
        for i, p in enumerate(plans):
            p.fc2d_extend_coeffs(n_f[i], f[i], b[i], refs[-1][i])
    grp = fc2d.fc2d_group_create(plans)
    grp.fc2d_group_tuning_set(form, 256)
    for k in (0, 0, 0, 1, 0, 0, 0, 1, 1, 1, 0, 1):
        n_f, f, b, out = sets[k]
        for o in out:
            o.fill_(7.0)
        grp.fc2d_group_extend_coeffs(n_f, f, b, out)
        for i in range(len(plans)):
            assert torch.equal(refs[k][i], out[i]), (k, i)
    grp.fc2d_group_destroy()


@pytest.mark.parametrize("form", ["branches", "persistent"])
def test_alternating_calls_do_not_wait_for_the_device(form):
    """Only a call with the arguments of the call just before it is captured, which waits for
    the device: after A has been captured, calls that alternate between two sets of buffers
    return while an unrelated stream is still busy."""
    torch = pytest.importorskip("torch")
    from paper_2010_03901_gb300 import fc2d
    plans = mixed_plans(fc2d)
    gen = torch.Generator(device="cuda").manual_seed(10)
    sets = [call_set(torch, plans, [1, 2, 1], gen) for _ in range(2)]
    refs = []
    for n_f, f, b, out in sets:
        refs.append([torch.zeros_like(o) for o in out])
        for i, p in enumerate(plans):
            p.fc2d_extend_coeffs(n_f[i], f[i], b[i], refs[-1][i])
    grp = fc2d.fc2d_group_create(plans)
    grp.fc2d_group_tuning_set(form, 256)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    call = lambda k: grp.fc2d_group_extend_coeffs(*sets[k], stream=mine.cuda_stream)  # noqa: E731
    call(0)
    call(0)  # captured
    waited = []
    for k in (1, 0, 1, 0, 1, 0):
        torch.cuda.synchronize()
        for o in sets[k][3]:
            o.fill_(7.0)
        torch.cuda.synchronize()
        busy = torch.cuda.Event()
        with torch.cuda.stream(other):
            torch.cuda._sleep(200_000_000)  # about 0.1 s
            busy.record()
        call(k)
        waited.append(busy.query())
        torch.cuda.synchronize()
        for i in range(len(plans)):
            assert torch.equal(refs[k][i], sets[k][3][i]), (k, i)
    assert not any(waited), waited
    grp.fc2d_group_destroy()


@pytest.mark.parametrize("form", ["branches", "persistent"])
@pytest.mark.parametrize("seen", [0, 1, 3])
def test_inside_a_capture_of_the_caller(form, seen):
    """A caller's graph that holds a group call (whose arguments were never passed before, once,
    or run as the group's own graph) keeps its work items when calls with fewer and with more
    functions follow; function counts that were not called before are refused, and the capture
    goes on."""
    torch = pytest.importorskip("torch")
    from paper_2010_03901_gb300 import fc2d
    plans = mixed_plans(fc2d)
    gen = torch.Generator(device="cuda").manual_seed(11)
    sets = [call_set(torch, plans, n_f, gen) for n_f in ([2, 1, 2], [2, 1, 2], [1, 1, 1], [3, 2, 3])]
    refs = []
    for n_f, f, b, out in reversed(sets):  # the largest counts first: no workspace grows later
        refs.insert(0, [torch.zeros_like(o) for o in out])
        for i, p in enumerate(plans):
            p.fc2d_extend_coeffs(n_f[i], f[i], b[i], refs[0][i])
    grp = fc2d.fc2d_group_create(plans)
    grp.fc2d_group_tuning_set(form, 256)

    def check(k, run):
        for o in sets[k][3]:
            o.fill_(7.0)
        run()
        torch.cuda.synchronize()
        for i in range(len(plans)):
            assert torch.equal(refs[k][i], sets[k][3][i]), (k, i)

    call = lambda k: grp.fc2d_group_extend_coeffs(*sets[k])  # noqa: E731
    call(1)
    for _ in range(seen):
        call(0)
    torch.cuda.synchronize()
    graph, mark = torch.cuda.CUDAGraph(), torch.zeros(1, device="cuda")
    with torch.cuda.graph(graph):
        call(0)
        with pytest.raises(fc2d.Fc2dError, match="stream capture"):
            call(2)
        mark.add_(1.0)
    check(0, graph.replay)
    for k in (2, 2, 2, 3, 0, 0, 0, 1):
        check(k, lambda: call(k))  # noqa: B023
        check(0, graph.replay)
    assert float(mark) == 9.0
    grp.fc2d_group_destroy()
