"""FP32 tetrahedra: the error against the FP64 oracle grows by less than one ulp
(2^-23 of the 2-norm) per step.  The solve, the extrapolation and the relaxation
round a value by half an ulp each, with signs that vary from cell to cell and
step to step; on a mesh of congruent cells the rounding of the coefficients is
the same everywhere and always, and adds up.
"""
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


@pytest.mark.parametrize("n,tiles", [(4, 1), (5, 1), (6, 2)])
@pytest.mark.parametrize("velset", [0, 1])
@pytest.mark.parametrize("system", ["maxwell", "euler"])
def test_one_ulp_per_step(kin, system, velset, n, tiles):
    steps = 8
    if system == "maxwell":
        w = workloads.tet_maxwell(seed=1, n=n, tiles=tiles, velset=velset, dt_mult=5.0, sigma=1.0)
    else:
        w = workloads.tet_densitywave(seed=1, n=n, tiles=tiles, velset=velset, dt_mult=5.0)
    P, T = oracle.tet_problem(w), oracle.TetMesh.from_workload(w)
    fo = oracle.tet_init(P, T, w.W0)
    oracle.tet_step(P, T, fo, steps)
    with kin.TetContext.from_workload(w, precision=kin.KIN_FP32) as ctx:
        ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        ctx.step(steps)
        f = ctx.get_kinetic()
    fo = fo.reshape(-1)
    err = np.linalg.norm(f - fo) / np.linalg.norm(fo)
    assert err < steps * 2.0 ** -23, err
