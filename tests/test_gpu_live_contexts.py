"""Contexts that share a kernel and differ in size, alive at the same time: the
dynamic shared memory a kernel may use is a property of the function, so it
must not follow the context created last.  The larger context, created first,
gives what it gives alone -- stepped in turn with the smaller one, after a
kin_step_noalloc of the smaller problem, and in one batch with it."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kin():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_11010_gb300 import build
    build.build()
    import paper_2212_11010_gb300 as kin
    kin.load_library()
    return kin


def line(n, degree, prec):
    return workloads.advection1d(seed=n, n=n, tiles=4, degree=degree, dt=2.4 / n, precision=prec), {}


def plane(n, tiles, degree, block, prec="f32"):
    w = workloads.vortex2d(seed=n, n=n, degree=degree, tiles=tiles, dt_mult=4.0)
    return workloads.with_(w, precision=prec), dict(block=block) if block else {}


# (larger, smaller): several steps per launch in 1D, one block or eight; the
# generic kernel with tiles of 50 to 220 KB
PAIRS = {
    "1d-f32": (line(8192, 3, "f32"), line(256, 3, "f32")),
    "1d-f64": (line(4096, 1, "f64"), line(64, 1, "f64")),
    "2d-p1": (plane(116, 4, 1, (29, 29)), plane(68, 4, 1, (17, 17))),
    "2d-p2": (plane(39, 3, 2, (13, 13)), plane(33, 3, 2, (11, 11))),
    "2d-p3-f64": (plane(28, 4, 3, (7, 7), "f64"), plane(20, 4, 3, (5, 5), "f64")),
}


def run(ctx, w, steps=5):
    ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
    for _ in range(steps):
        ctx.step(1)
    return ctx.get_kinetic()


@pytest.mark.parametrize("name", list(PAIRS))
def test_larger_context_survives_a_smaller_one(kin, name):
    import torch
    (big, kb), (small, ks) = PAIRS[name]
    alone = []
    for w, k in PAIRS[name]:
        with kin.Context.from_workload(w, **k) as ctx:
            alone.append(run(ctx, w))
    with kin.Context.from_workload(big, **kb) as a, kin.Context.from_workload(small, **ks) as b:
        assert np.array_equal(run(a, big), alone[0])
        assert np.array_equal(run(b, small), alone[1])
        for ctx, w in ((a, big), (b, small)):
            ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        for _ in range(5):
            a.step(1)
            b.step(1)
        assert np.array_equal(a.get_kinetic(), alone[0])
        assert np.array_equal(b.get_kinetic(), alone[1])
        mesh, model, opts = kin.make_args(small.dim, small.n, small.lo, small.hi, small.system, small.lam,
                                          omega=small.omega, gamma=small.gamma, adv=small.adv, tiles=small.tiles,
                                          iters=small.iters,
                                          precision=kin.KIN_FP32 if small.precision == "f32" else kin.KIN_FP64, **ks)
        f = torch.from_numpy(alone[1].copy()).cuda()
        kin.kin_step_noalloc(mesh, model, small.degree, small.dt, opts, f, 1)
        assert np.array_equal(run(a, big), alone[0])
        for ctx, w in ((a, big), (b, small)):
            ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        with kin.Batch([a, b]) as batch:
            batch.step(5)
            batch.sync()
        assert np.array_equal(a.get_kinetic(), alone[0])
        assert np.array_equal(b.get_kinetic(), alone[1])


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dim", [2, 3])
def test_wavefront_sweeps_of_two_sizes(kin, dim, prec):
    # one kernel instance for up to 256 columns per subdomain (3D: degree 2)
    if dim == 2:
        ws = [workloads.vortex2d(seed=n, n=n, degree=2, tiles=1, dt_mult=4.0, velset=1) for n in (200, 12)]
        if prec == "f32":           # without room for its records: the sweep in one kernel
            with kin.Context.from_workload(ws[0]) as ctx:
                need = ctx.info.device_bytes - 256
    else:
        ws = [workloads.densitywave3d(seed=n, n=n, degree=2, tiles=1, dt_mult=4.0, velset=1) for n in (12, 4)]
    ws = [workloads.with_(w, precision=prec) for w in ws]
    kw = [{}, {}]
    if dim == 2 and prec == "f32":
        kw[0] = dict(mem_budget=need)
    alone = []
    for w, k in zip(ws, kw):
        with kin.Context.from_workload(w, **k) as ctx:
            alone.append(run(ctx, w, 2))
    with kin.Context.from_workload(ws[0], **kw[0]) as a, kin.Context.from_workload(ws[1], **kw[1]) as b:
        assert np.array_equal(run(b, ws[1], 2), alone[1])
        assert np.array_equal(run(a, ws[0], 2), alone[0])


def test_a_block_beyond_shared_memory_is_refused(kin):
    # a tile of 230,400 bytes fits 227 KB, its inflow traces beside it do not
    w, k = plane(30, 1, 1, (30, 30))
    with pytest.raises(kin.KinError) as e:
        kin.Context.from_workload(w, **k)
    assert e.value.status == kin.KIN_ECUDA
