"""f = M(W): the FP32 state (evaluated on FP32 pairs where the values allow it)
against the FP64 state of the same field rounded to FP32.

Tolerance, derived: the pairs carry 47 bits, and a Maxwellian is a dozen
operations, so before the last rounding a value is off by less than 2^-40 of
the largest value of its node; the rounding to FP32 adds half an ulp,
2^-24 of the value (2^-150 when it is subnormal).
"""
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


SETS = {"advection1d": ("advection", 1, None), "euler1d": ("euler", 1, None), "advection2d": ("advection", 2, None),
        "euler2d": ("euler", 2, None), "euler3d": ("euler", 3, None), "maxwell3d": ("maxwell", 3, None),
        "d2q3": ("euler", 2, "simplex"), "d3q4": ("euler", 3, "simplex"), "tet-d3q4": ("euler", 3, "tet1"),
        "tet-d3q6": ("maxwell", 3, "tet0"), "tet-adv": ("advection", 3, "tet1")}


def field(system, dim, nodes, scale, rng):
    if system == "euler":
        rho = rng.uniform(0.5, 1.5, nodes)
        u = rng.normal(size=(dim, nodes)) * rng.choice([0.0, 1e-9, 1.0], size=(dim, nodes))
        E = rng.uniform(1.0, 3.0, nodes) + 0.5 * rho * (u ** 2).sum(0)
        W = np.concatenate([rho[None], rho * u, E[None]])
    else:
        W = rng.normal(size=(1 if system == "advection" else 6, nodes))
        W[:, ::5] = 0.0
    return W * scale


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 20, 2.0 ** 30, 2.0 ** -20, 2.0 ** -74, 2.0 ** 110])
@pytest.mark.parametrize("name", sorted(SETS))
def test_fp32_state_is_the_rounded_fp64_state(kin, name, scale):
    system, dim, kind = SETS[name]
    sysid = {"advection": kin.KIN_ADVECTION, "euler": kin.KIN_EULER, "maxwell": kin.KIN_MAXWELL}[system]
    out = {}
    for prec in (kin.KIN_FP64, kin.KIN_FP32):
        if kind and kind.startswith("tet"):
            m = workloads.tet_box(3)
            ctx = kin.TetContext(m.xyz, m.vid, m.nbr, m.subdomains(1), m.wrap, sysid,
                                 kin.KIN_D3Q4 if kind == "tet1" else kin.KIN_D3Q6, 5.0, 1e-3, precision=prec)
        else:
            vs = None if kind is None else {2: kin.KIN_D2Q3, 3: kin.KIN_D3Q4}[dim]
            ctx = kin.Context(dim, (5, 3, 2)[:dim], (0.0,) * dim, (1.0,) * dim, 2, sysid, 5.0, 1e-3, adv=(1.0, 0.5, 0.0),
                              precision=prec, velset=vs)
        with ctx:
            W = field(system, dim, ctx.info.nodes, scale, np.random.default_rng(7))
            if scale == 1.0:
                W[-1, 3], W[-1, 4] = np.nan, np.inf      # end up where the FP64 evaluation puts them
            ctx.set_state(np.ascontiguousarray(W.reshape(-1)))
            out[prec] = ctx.get_kinetic().reshape(ctx.info.npop, -1)
    f64, f32 = out[kin.KIN_FP64], out[kin.KIN_FP32].astype(np.float64)
    with np.errstate(over="ignore"):
        fine = np.isfinite(f64.astype(np.float32))
        assert np.array_equal(fine, np.isfinite(f32))
    top = np.where(np.isfinite(f64), np.abs(f64), 0.0).max(0)
    tol = 2.0 ** -24 * np.abs(f64) + 2.0 ** -40 * top + 2.0 ** -150
    assert (np.abs(f32[fine] - f64[fine]) <= tol[fine]).all()
