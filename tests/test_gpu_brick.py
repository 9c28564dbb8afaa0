"""The D3Q4 sweep on bricks of 2 x 2 x 2 cells (FP32, degree 1, even
subdomains) against the FP64 oracle, 1e-5 of the largest value: streams of
several widths per warp, one and several subdomains, unequal extents, more and
fewer problems than warps, K = 1, 2, 3 (and the
neighbouring shapes that keep the one-cell sweep); and a periodic field, whose
copies must come out bit for bit alike wherever they were swept.
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


# (cells per subdomain, subdomains, K)
SHAPES = [((8, 8, 8), (2, 2, 2), 3), ((2, 2, 2), (3, 2, 4), 3), ((4, 4, 4), (3, 1, 2), 2), ((6, 6, 6), (1, 2, 1), 3),
          ((10, 10, 2), (2, 1, 1), 3), ((4, 8, 6), (2, 2, 3), 1), ((8, 4, 12), (1, 3, 2), 3), ((16, 8, 4), (1, 1, 1), 2),
          ((2, 10, 4), (5, 1, 2), 3), ((12, 12, 4), (1, 1, 2), 3), ((6, 4, 3), (2, 3, 2), 3), ((4, 4, 2), (12, 10, 9), 3)]


@pytest.mark.parametrize("omega", [2.0, 1.8])
@pytest.mark.parametrize("shape", SHAPES, ids=[str(s) for s in SHAPES])
def test_matches_oracle(kin, shape, omega):
    L, tiles, K = shape
    n = tuple(a * b for a, b in zip(L, tiles))
    w = workloads.densitywave3d(seed=4, n=8, degree=1, tiles=1, dt_mult=8.0, iters=K, omega=omega, velset=1)
    rng = np.random.default_rng(1)
    nodes = int(np.prod(n)) * 8
    W0 = np.ascontiguousarray(w.W0.reshape(5, -1)[:, rng.integers(0, w.W0.size // 5, nodes)])
    w = workloads.with_(w, n=n, tiles=tiles, W0=W0)
    P = oracle.Problem(**w.oracle_kwargs())
    fo = oracle.init(P, w.W0)
    oracle.step(P, fo, 2)
    with kin.Context.from_workload(w) as ctx:
        ctx.set_state(W0.reshape(-1))
        ctx.step(2)
        f = ctx.get_kinetic()
        bricks = all(a % 2 == 0 for a in L) and L[0] * L[1] <= 128
        assert (ctx.info.threads == 32) == (bricks or L[0] * L[1] <= 32)
    err = np.abs(f - fo.reshape(-1)).max() / np.abs(fo).max()
    assert err < 1e-5, err


def test_periodic_copies_of_one_field_agree(kin):
    # 6-cell subdomains of a field that repeats every 6 cells: every
    # subdomain gives the same state, whichever stream and warp swept it
    w = workloads.densitywave3d(seed=5, n=6, degree=1, tiles=1, dt_mult=6.0, velset=1)
    W1 = w.W0.reshape(5, 6, 6, 6, 8)
    big = np.ascontiguousarray(np.tile(W1, (1, 2, 3, 4, 1)))
    with kin.Context.from_workload(w) as one, \
            kin.Context.from_workload(workloads.with_(w, n=(24, 18, 12), hi=(4.0, 3.0, 2.0), tiles=(4, 3, 2))) as many:
        one.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        many.set_state(big.reshape(-1))
        one.step(3)
        many.step(3)
        a = one.get_kinetic().reshape(20, 6, 6, 6, 8)
        b = many.get_kinetic().reshape(20, 12, 18, 24, 8)
    assert np.array_equal(np.tile(a, (1, 2, 3, 4, 1)), b)
