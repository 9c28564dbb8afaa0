"""Tetrahedral sweeps against the FP64 oracle where the sweep changes shape:
all variables of a cell in one block (many subdomains), split over blocks
(few), levels wider than a chunk, chunks cut by their interface cells, one
iterate only, and a mesh whose levels are too wide for shared memory (the
iterate in global memory).

FP64 tolerance 1e-12, FP32 1e-5 of the largest value, those of the
tetrahedral parity tests.
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


CASES = {
    "together": lambda: workloads.tet_densitywave(seed=1, n=8, tiles=4, velset=1, dt_mult=8.0),
    "together-d3q6": lambda: workloads.tet_maxwell(seed=2, n=9, tiles=3, velset=0, dt_mult=6.0, sigma=1.0),
    "split": lambda: workloads.tet_densitywave(seed=3, n=10, tiles=2, velset=1, dt_mult=5.0, iters=2),
    "wide": lambda: workloads.tet_densitywave(seed=4, n=12, tiles=1, velset=1, dt_mult=5.0),
    "one-iterate": lambda: workloads.tet_densitywave(seed=5, n=8, tiles=4, velset=1, dt_mult=5.0, iters=1),
    "four-iterates": lambda: workloads.tet_advection(seed=6, n=6, tiles=3, velset=1, iters=4),
    "global": lambda: workloads.tet_densitywave(seed=7, n=24, tiles=1, velset=1, dt_mult=5.0),
}


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("name", list(CASES))
def test_matches_oracle(kin, name, prec):
    w = CASES[name]()
    steps = 2 if name == "global" else 3
    P = oracle.tet_problem(w)
    T = oracle.TetMesh.from_workload(w)
    fo = oracle.tet_init(P, T, w.W0)
    oracle.tet_step(P, T, fo, steps)
    with kin.TetContext.from_workload(w, precision=kin.KIN_FP64 if prec == "f64" else kin.KIN_FP32) as ctx:
        ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        ctx.step(steps)
        f = ctx.get_kinetic()
        if name == "global" and prec == "f64":
            assert ctx.info.smem_bytes == 0
    fo = fo.reshape(w.npop, -1)
    err = np.abs(f.reshape(w.npop, -1) - fo).max(1) / np.abs(fo).max()
    assert err.max() < (1e-12 if prec == "f64" else 1e-5)
