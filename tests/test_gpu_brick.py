"""The D3Q4 sweep on bricks of 2 x 2 x 2 cells (FP32, degree 1, even
subdomains) against the FP64 oracle, 1e-5 of the largest value: streams of
several widths per warp, unequal extents, K = 2, 3 (and the neighbouring shapes
that keep the one-cell sweep); and, for K = 1, 2, 3, a periodic field, whose
copies must come out bit for bit like the one-cell sweep of one period.
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


# (cells per subdomain, subdomains, K, bricks): 32 / ((L0/2)(L1/2)) streams per
# warp, and 16 warps' work per SM before bricks are taken
SHAPES = [((8, 8, 8), (7, 6, 6), 3, 1), ((2, 2, 2), (16, 16, 16), 3, 1), ((4, 4, 4), (10, 10, 10), 2, 1),
          ((6, 6, 6), (8, 8, 6), 3, 1), ((10, 10, 2), (5, 5, 5), 3, 1),
          ((16, 8, 4), (5, 5, 5), 2, 1), ((2, 10, 4), (9, 9, 10), 3, 1),
          ((8, 8, 8), (2, 2, 2), 3, 0), ((12, 12, 4), (5, 5, 5), 3, 0), ((6, 4, 3), (9, 9, 9), 2, 0)]


@pytest.mark.parametrize("omega", [2.0, 1.8])
@pytest.mark.parametrize("shape", SHAPES, ids=[str(s) for s in SHAPES])
def test_matches_oracle(kin, shape, omega):
    L, tiles, K, bricks = shape
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
        bx, by = L[0] // 2, L[1] // 2
        smem = 4 * (32 * 68 + (32 + 32 // (bx * by) * (bx + by)) * 20)
        assert (ctx.info.threads == 32 and ctx.info.smem_bytes == smem) == bool(bricks)
    err = np.abs(f - fo.reshape(-1)).max() / np.abs(fo).max()
    assert err < 1e-5, err


@pytest.mark.parametrize("K", [1, 2, 3])
def test_periodic_copies_of_one_field_agree(kin, K):
    # 6-cell subdomains of a field that repeats every 6 cells: every subdomain
    # gives the same state, whichever stream and warp swept it, and the same as
    # one subdomain alone, which is too little work for bricks
    w = workloads.densitywave3d(seed=5, n=6, degree=1, tiles=1, dt_mult=6.0, iters=K, velset=1)
    W1 = w.W0.reshape(5, 6, 6, 6, 8)
    big = np.ascontiguousarray(np.tile(W1, (1, 6, 8, 8, 1)))
    with kin.Context.from_workload(w) as one, \
            kin.Context.from_workload(workloads.with_(w, n=(48, 48, 36), hi=(8.0, 8.0, 6.0), tiles=(8, 8, 6))) as many:
        one.set_state(np.ascontiguousarray(w.W0.reshape(-1)))
        many.set_state(big.reshape(-1))
        one.step(3)
        many.step(3)
        a = one.get_kinetic().reshape(20, 6, 6, 6, 8)
        b = many.get_kinetic().reshape(20, 36, 48, 48, 8)
    assert np.array_equal(np.tile(a, (1, 6, 8, 8, 1)), b)
