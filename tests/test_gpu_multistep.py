"""1D problems whose steps of a call run in one launch: against the FP64
oracle (1e-12 FP64, 1e-5 FP32 of the largest value), the same result however
the steps are split over calls or run in a batch, and the state left for what
follows (diagnostics, single steps of a larger problem's path)."""
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


def problem(n, tiles, degree, system, prec, **kw):
    w = workloads.advection1d(seed=1, n=n, tiles=tiles, degree=degree, dt=0.6 / n * 4, precision=prec)
    if system == "euler":
        rho = np.abs(w.W0) + 0.5
        w = workloads.with_(w, system=workloads.EULER, lam=6.0, dt=1.0 / n,
                            W0=np.concatenate([rho, 0.4 * rho, 2.0 + 0.08 * rho]))
    return workloads.with_(w, **kw)


CASES = [
    (256, 4, 1, "advection", {}),
    (256, 1, 1, "advection", dict(dt=0.02)),        # one subdomain that wraps onto itself
    (24, 3, 2, "advection", dict(iters=2, omega=1.7)),   # fewer cell blocks than thread blocks
    (5, 1, 1, "advection", {}), (1, 1, 2, "advection", {}),
    (130, 13, 3, "euler", {}),                       # blocks do not divide evenly
    (60, 4, 1, "euler", dict(inflow=(1, 0, 0), Wb=np.tile([1.0, 0.4, 2.0], (3, 2, 1)))),
    (2048, 8, 3, "advection", {}),                   # the FP64 limit (16384 values)
    (2049, 3, 3, "advection", {}),                   # just above it
    (8192, 8, 3, "advection", {}),                   # the FP32 limit (65536 values)
]


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_matches_oracle_and_splits(kin, case, prec):
    n, tiles, degree, system, kw = CASES[case]
    w = problem(n, tiles, degree, system, prec, **kw)
    P = oracle.Problem(**w.oracle_kwargs())
    fo = oracle.init(P, w.W0)
    oracle.step(P, fo, 5)
    out, resid = [], []
    for split in ([5], [2, 3], [1, 1, 1, 2], "batch"):
        with kin.Context.from_workload(w) as ctx:
            ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
            if split == "batch":
                with kin.Batch([ctx]) as b:
                    b.step(3)
                    b.step(2)
                    b.sync()
            else:
                for s in split:
                    ctx.step(s)
            out.append(ctx.get_kinetic())
            assert ctx.info.dim == 1 and kin.kin_query(ctx.ctx).steps_done == 5
            if not any(w.inflow):
                resid.append(ctx.diag()[1:])
    err = np.abs(out[0] - fo.reshape(-1)).max() / np.abs(fo).max()
    assert err < (1e-12 if prec == "f64" else 1e-5), err
    for f in out[1:]:
        assert np.array_equal(out[0], f)
    for r in resid[1:]:                               # the summaries are those of the same state
        assert np.array_equal(resid[0][0], r[0]) and resid[0][1] == r[1]
