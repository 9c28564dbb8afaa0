"""The fixed-shape kernels of 3D degrees 2 and 3 and of FP64, and the generic
kernel on rows that are not whole 16-byte words, against the FP64 oracle:
periodic and inflow axes, omega below 2, K = 2.  Tolerances as in the parity
tests (1e-12 FP64, 1e-5 FP32, relative to the largest value)."""
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


# (dim, degree, precision, system, block (None: the default choice), cells per subdomain)
SHAPES = [
    (2, 1, "f32", "euler", (8, 8, 1), 8), (2, 1, "f64", "euler", (8, 8, 1), 8), (2, 3, "f64", "euler", (8, 4, 1), 8),
    (3, 2, "f32", "euler", (4, 2, 2), 4), (3, 3, "f32", "euler", (2, 2, 2), 4),
    (3, 2, "f32", "maxwell", (4, 2, 2), 4), (3, 3, "f32", "maxwell", (2, 2, 2), 2),
    (3, 1, "f64", "euler", (4, 4, 2), 4), (3, 2, "f64", "euler", (2, 2, 2), 4), (3, 3, "f64", "euler", (2, 2, 1), 2),
    (3, 1, "f64", "maxwell", (4, 4, 2), 4), (3, 2, "f64", "maxwell", (2, 2, 2), 2),
    (3, 3, "f64", "maxwell", (2, 2, 1), 2),
    # generic: odd extents, rows of 4- and 8-byte multiples
    (2, 2, "f32", "euler", None, 5), (2, 2, "f64", "euler", None, 7), (2, 2, "f32", "euler", None, 1),
    (3, 2, "f32", "euler", None, 3), (3, 2, "f32", "maxwell", None, 3), (2, 1, "f32", "euler", None, 9),
]


@pytest.mark.parametrize("inflow", [0, 1])
@pytest.mark.parametrize("shape", SHAPES, ids=[str(s) for s in SHAPES])
def test_matches_oracle(kin, shape, inflow):
    dim, degree, prec, system, block, L = shape
    tiles = (3, 2, 1)[:dim]
    n = tuple(L * t for t in tiles)
    if system == "maxwell":
        w = workloads.maxwell3d(seed=3, n=6, degree=degree, tiles=1, dt_mult=20.0, sigma=2.0, omega=1.8, precision=prec)
    elif dim == 2:
        w = workloads.vortex2d(seed=3, n=6, degree=degree, tiles=1, dt_mult=20.0, precision=prec)
    else:
        w = workloads.densitywave3d(seed=3, n=6, degree=degree, tiles=1, dt_mult=20.0, iters=2, precision=prec)
    nodes = int(np.prod(n)) * (degree + 1) ** dim
    idx = np.arange(nodes) % (w.W0.size // w.m)              # a field of the same values on the odd mesh
    w = workloads.with_(w, n=n, tiles=tiles, W0=np.ascontiguousarray(w.W0.reshape(w.m, -1)[:, idx]))
    if inflow:
        Wb = np.zeros((3, 2, w.m))
        if system == "euler":
            Wb[...] = [1.0] + [0.5] * dim + [2.5 + 0.125 * dim]
        w = workloads.with_(w, inflow=tuple([1] * dim + [0] * (3 - dim)), Wb=Wb)
    P = oracle.Problem(**w.oracle_kwargs())
    fo = oracle.init(P, w.W0)
    oracle.step(P, fo, 3)
    with kin.Context.from_workload(w, **({"block": block} if block else {})) as ctx:
        ctx.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        ctx.step(3)
        f = ctx.get_kinetic()
        if block:
            assert ctx.info.specialised == 1 and tuple(ctx.info.block) == block
        else:
            assert ctx.info.specialised == 0
    err = np.abs(f - fo.reshape(-1)).max() / np.abs(fo).max()
    assert err < (1e-12 if prec == "f64" else 1e-5), err
