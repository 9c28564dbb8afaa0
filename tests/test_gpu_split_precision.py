"""The split D2Q3 sweep is no further from the FP64 oracle than the one-kernel
sweep (a context whose budget has no room for the records): the errors of
six problems per degree, summed."""
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


def run(kin, w, steps, **kw):
    with kin.Context.from_workload(w, **kw) as ctx:
        ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        ctx.step(steps)
        return ctx.get_kinetic(), ctx.info.device_bytes


@pytest.mark.parametrize("degree", [1, 2, 3])
def test_no_further_off_than_one_kernel(kin, degree):
    total = np.zeros(2)
    for seed, (L, tiles, K, omega, mult) in enumerate([(8, 4, 3, 2.0, 4.0), (16, 3, 3, 1.8, 7.0), (32, 2, 3, 2.0, 3.0),
                                                       (25, 2, 3, 2.0, 5.0), (40, 2, 2, 1.8, 4.0), (12, 5, 3, 2.0, 8.0)]):
        w = workloads.vortex2d(seed=seed, n=L * tiles, degree=degree, tiles=tiles, dt_mult=mult, velset=1, iters=K,
                               omega=omega)
        P = oracle.Problem(**w.oracle_kwargs())
        fo = oracle.init(P, w.W0)
        oracle.step(P, fo, 10)
        split, held = run(kin, w, 10)
        one, _ = run(kin, w, 10, mem_budget=held - 256)
        assert not np.array_equal(split, one)
        fo = fo.reshape(-1)
        total += [np.linalg.norm(f - fo) / np.linalg.norm(fo) for f in (split, one)]
    assert total[0] <= total[1], total
