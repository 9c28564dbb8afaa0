"""The split D2Q3 sweep (FP32: local part, chain over the outflow nodes, full
solve with the relaxation) against the FP64 oracle, 1e-5 of the largest value
(the FP32 parity bound): unequal subdomains below, at and above a warp of columns
and above two, cells that do not fill the groups of 32, every degree, K = 1..3,
omega below 2, scalar advection; a constant state is kept exactly; without
room for the records the one-kernel sweep gives the same to rounding."""
import numpy as np
import pytest

import oracle
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


def problem(L, tiles, degree, K, omega=2.0, system="euler"):
    n = tuple(a * b for a, b in zip(L, tiles))
    w = workloads.vortex2d(seed=2, n=n[0], degree=degree, tiles=1, dt_mult=4.0, velset=1)
    xy = workloads.node_coords(2, n, (0.0, 0.0), (10.0, 10.0), degree)
    rho, vel, pr = workloads._vortex_fields(xy[:, 0], xy[:, 1], 4.0, 5.0, 3.5, 1.4, 10.0, 1.0, 1.0)
    W0 = workloads._euler_conserved(rho, vel, pr, 1.4)
    w = workloads.with_(w, n=n, tiles=tiles, iters=K, omega=omega, W0=W0, dt=w.dt * min(1.0, n[0] / n[1]))
    if system == "advection":
        w = workloads.with_(w, system=workloads.ADVECTION, adv=(1.0, 0.5, 0.0), W0=np.ascontiguousarray(W0[:1]))
    return w


CASES = [((8, 8), (2, 2), 1, 3), ((5, 7), (3, 2), 2, 3), ((7, 5), (2, 3), 3, 2), ((32, 32), (2, 1), 2, 3),
         ((40, 33), (1, 2), 1, 3), ((70, 9), (1, 2), 2, 2), ((3, 1), (5, 9), 3, 3), ((16, 24), (2, 2), 2, 1),
         ((1, 1), (6, 5), 1, 3), ((9, 80), (2, 1), 3, 1)]


@pytest.mark.parametrize("omega,system", [(2.0, "euler"), (1.7, "euler"), (1.9, "advection")])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_matches_oracle(kin, case, omega, system):
    w = problem(*CASES[case], omega=omega, system=system)
    P = oracle.Problem(**w.oracle_kwargs())
    fo = oracle.init(P, w.W0)
    oracle.step(P, fo, 3)
    got = []
    for tight in (False, True):
        need = 0
        if tight:                       # a budget without room for the records
            with kin.Context.from_workload(w) as ctx:
                need = ctx.info.device_bytes - 256
        with kin.Context.from_workload(w, mem_budget=need) as ctx:
            ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
            ctx.step(3)
            got.append(ctx.get_kinetic())
    for f in got:
        err = np.abs(f - fo.reshape(-1)).max() / np.abs(fo).max()
        assert err < 1e-5, err


@pytest.mark.parametrize("degree", [1, 2, 3])
def test_constant_state_is_kept(kin, degree):
    w = problem((6, 9), (2, 2), degree, 3, omega=1.5)
    W0 = np.empty_like(w.W0)
    W0[:] = np.array([1.25, 0.5, -0.25, 2.5])[:, None]
    with kin.Context.from_workload(workloads.with_(w, W0=W0)) as ctx:
        ctx.set_state(W0.reshape(-1))
        ctx.step(1)
        f = ctx.get_kinetic().reshape(12, -1)
    assert (f == f[:, :1]).all()        # the transport leaves every node of a population alike


def test_records_follow_the_state(kin):
    # the records a step leaves for the next one are those of f however the
    # steps are split, and a new f (synchronous or not) replaces them
    import torch
    w = problem((12, 10), (2, 3), 2, 3)
    other = problem((12, 10), (2, 3), 2, 3, omega=1.7)
    with kin.Context.from_workload(w) as ctx:
        ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        ctx.step(4)
        want = ctx.get_kinetic()
        ctx.set_state(np.ascontiguousarray(other.W0.reshape(-1)[::-1].copy()))
        ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        ctx.step(1)
        ctx.step(3)
        assert np.array_equal(ctx.get_kinetic(), want)
        ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        ctx.step(2)
        mid = ctx.get_kinetic()
        ctx.step(3)
        ctx.set_kinetic(mid)
        ctx.step(2)
        assert np.array_equal(ctx.get_kinetic(), want)
        h = torch.from_numpy(mid).pin_memory()
        ctx.step(1)
        ctx.sync()
        kin.kin_set_kinetic_async(ctx.ctx, h)
        ctx.step(2)
        assert np.array_equal(ctx.get_kinetic(), want)


def test_captured_step_can_be_replayed(kin):
    # a step captured into a graph advances the state on every replay, between
    # and after steps that were not captured
    import torch
    w = problem((12, 10), (2, 3), 2, 3)
    st = torch.cuda.Stream()
    with kin.Context.from_workload(w, stream=st.cuda_stream) as ctx:
        ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        ctx.step(6)
        want = ctx.get_kinetic()
        ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        ctx.step(1)
        ctx.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            ctx.step(1)
        with torch.cuda.stream(st):
            g.replay()
            g.replay()
        ctx.step(1)
        with torch.cuda.stream(st):
            g.replay()
        ctx.step(1)
        assert np.array_equal(ctx.get_kinetic(), want)
