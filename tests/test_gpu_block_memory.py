"""Default cell blocks of 2D problems whose subdomains take 8 x 8 blocks but
not 16 x 8: the block summaries stay within what the thickest block of
about 48 KB needs, so that budgets and the static scratch of
kin_step_noalloc (16 MiB) keep taking the problems they can hold."""
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


@pytest.mark.parametrize("n,tiles,thick", [((648, 648), 27, (12, 12)), ((696, 696), 29, (12, 12)),
                                           ((320, 320), 8, (10, 10)), ((192, 320), 8, (12, 10))])
def test_budget_of_the_thick_block_is_enough(kin, n, tiles, thick):
    import torch
    w = workloads.vortex2d(seed=1, n=n[0], degree=1, tiles=tiles, dt_mult=4.0)
    w = workloads.with_(w, n=n, tiles=(tiles, tiles))
    with kin.Context.from_workload(w, block=thick) as ctx:
        need = ctx.info.device_bytes
    with kin.Context.from_workload(w, mem_budget=need) as ctx:
        assert ctx.info.device_bytes <= need
    mesh, model, opts = kin.make_args(2, w.n, w.lo, w.hi, w.system, w.lam, tiles=w.tiles, precision=kin.KIN_FP32)
    f = torch.ones(w.npop * n[0] * n[1] * 4, device="cuda")
    kin.kin_step_noalloc(mesh, model, 1, w.dt, opts, f, 0)       # accepted: the summaries fit its scratch
