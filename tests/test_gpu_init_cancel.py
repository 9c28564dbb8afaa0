"""f = M(W) of FP32 contexts where values cancel: pressures that are a small part of
the energy, and equilibria that change sign, against the FP64 state of the
same field.

Tolerance, derived: the pairs leave each value right to 2^-32 of itself or give
the node to the FP64 evaluation; the rounding to FP32 adds 2^-24 of the value,
and the two FP64 evaluations (a dozen operations each, contracted differently
perhaps) differ by less than 2^-49 of the node's largest value.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

LAM, GAMMA = 5.0, 1.4


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


SETS = {"euler1d": ("euler", 1, None), "euler2d": ("euler", 2, None), "euler3d": ("euler", 3, None),
        "maxwell3d": ("maxwell", 3, None), "d2q3": ("euler", 2, "simplex"), "d3q4": ("euler", 3, "simplex"),
        "tet-d3q4": ("euler", 3, "tet1"), "tet-d3q6": ("maxwell", 3, "tet0"), "tet-euler-d3q6": ("euler", 3, "tet0")}


def field(system, dim, nodes, bits, rng):
    near = 1.0 + rng.uniform(-1.0, 1.0, nodes) * 2.0 ** -bits
    if system == "maxwell":
        W = rng.normal(size=(6, nodes))
        W[4] = W[2] * (2 * LAM / 6.0) * near              # E_z / 6 against H_y / (2 lambda)
        W[5] = W[1] * (2 * LAM / 6.0) * near
        return W
    rho, u = rng.uniform(0.5, 1.5, nodes), rng.normal(size=(dim, nodes))
    third = nodes // 3
    u[:, :third] *= 30.0                                    # E / p up to 2^bits
    u[0, :third:2] = 0.0
    ke = 0.5 * rho * (u ** 2).sum(0)
    E = rng.uniform(1.0, 3.0, nodes) + ke
    E[:third] = (ke * (1.0 + 2.0 ** -bits * rng.uniform(0.5, 2.0, nodes)))[:third]
    # rho / (2d) against rho u / (2 lambda)
    u[0, third:2 * third] = (LAM / dim * near)[third:2 * third]
    E[third:2 * third] = (1.0 + 0.5 * rho * (u ** 2).sum(0))[third:2 * third]
    # momentum: m / (2d) against (m u + p) / (2 lambda) at rest pressure
    a = LAM / dim
    u[0, 2 * third:] = 0.5 * (a - np.sqrt(a * a - 1.6)) * near[2 * third:] if dim < 3 else u[0, 2 * third:]
    u[1:, 2 * third:] = 0.0
    E[2 * third:] = (0.4 * rho / (GAMMA - 1.0) + 0.5 * rho * (u ** 2).sum(0))[2 * third:]
    return np.concatenate([rho[None], rho * u, E[None]])


@pytest.mark.parametrize("bits", [3, 8, 14, 24, 40])
@pytest.mark.parametrize("name", sorted(SETS))
def test_cancelling_values_keep_their_bits(kin, name, bits):
    system, dim, kind = SETS[name]
    sysid = {"euler": kin.KIN_EULER, "maxwell": kin.KIN_MAXWELL}[system]
    out = {}
    for prec in (kin.KIN_FP64, kin.KIN_FP32):
        if kind and kind.startswith("tet"):
            m = workloads.tet_box(4)
            ctx = kin.TetContext(m.xyz, m.vid, m.nbr, m.subdomains(1), m.wrap, sysid,
                                 kin.KIN_D3Q4 if kind == "tet1" else kin.KIN_D3Q6, LAM, 1e-3, precision=prec)
        else:
            vs = None if kind is None else {2: kin.KIN_D2Q3, 3: kin.KIN_D3Q4}[dim]
            ctx = kin.Context(dim, (16, 9, 8)[:dim], (0.0,) * dim, (1.0,) * dim, 2, sysid, LAM, 1e-3, gamma=GAMMA,
                              precision=prec, velset=vs)
        with ctx:
            W = field(system, dim, ctx.info.nodes, bits, np.random.default_rng(7))
            ctx.set_state(np.ascontiguousarray(W.reshape(-1)))
            out[prec] = ctx.get_kinetic().reshape(ctx.info.npop, -1).astype(np.float64)
    f64, f32 = out[kin.KIN_FP64], out[kin.KIN_FP32]
    tol = 2.0 ** -24 * (1.0 + 2.0 ** -7) * np.abs(f64) + 2.0 ** -49 * np.abs(f64).max(0) + 2.0 ** -149
    off = np.abs(f32 - f64) - tol
    assert (off <= 0).all(), (int((off > 0).sum()), off.max())
