"""Tetrahedra read across a subdomain boundary by a cell that they do not
border in turn: what a subdomain hands to the others is decided by the readers.
The mesh has one cell more than the box, a copy of an interior cell in a subdomain
of its own: it reads the neighbours of the cell it copies, and no cell reads it."""
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


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("velset", [0, 1])
def test_one_sided_neighbour(kin, velset, prec):
    w = workloads.tet_densitywave(seed=2, n=6, tiles=2, velset=velset, dt_mult=5.0)
    m, sub = w.mesh, w.subdomains()
    nbr = np.asarray(m.nbr).reshape(-1, 4)
    inner = np.nonzero((sub[nbr] == sub[:, None]).all(1) & (np.asarray(m.wrap).reshape(-1, 4) == 0).all(1))[0]
    y = int(inner[len(inner) // 2])
    more = lambda a, k: np.concatenate([np.asarray(a).reshape(-1, *k), np.asarray(a).reshape(-1, *k)[y:y + 1]])
    xyz, vid, nbr, wrap = more(m.xyz, (4, 3)), more(m.vid, (4,)), more(nbr, (4,)), more(m.wrap, (4,))
    sub = np.concatenate([sub, [sub.max() + 1]]).astype(np.int32)
    W0 = np.asarray(w.W0).reshape(5, -1, 4)
    W0 = np.ascontiguousarray(np.concatenate([W0, W0[:, y:y + 1]], axis=1))
    P = oracle.tet_problem(w)
    T = oracle.TetMesh(xyz, vid, nbr, sub, wrap)
    fo = oracle.tet_init(P, T, W0.reshape(5, -1))
    oracle.tet_step(P, T, fo, 3)
    with kin.TetContext(xyz, vid, nbr, sub, wrap, w.system, kin.KIN_D3Q4 if velset else kin.KIN_D3Q6, w.lam, w.dt,
                        omega=w.omega, gamma=w.gamma, iters=3,
                        precision=kin.KIN_FP64 if prec == "f64" else kin.KIN_FP32) as ctx:
        ctx.set_state(W0.reshape(-1))
        ctx.step(3)
        f = ctx.get_kinetic()
    fo = fo.reshape(-1)
    err = np.abs(f - fo).max() / np.abs(fo).max()
    assert err < (1e-12 if prec == "f64" else 1e-5), err
