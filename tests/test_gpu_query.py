"""kin_query names the launch that runs: the cluster that takes all steps of a 1D
call, and the chain of the split D2Q3 sweep."""
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


@pytest.mark.parametrize("n,blocks", [(256, 1), (4096, 8)])
def test_steps_of_a_1d_call(kin, n, blocks):
    w = workloads.advection1d(seed=0, n=n, tiles=4, degree=1, precision="f32")
    with kin.Context.from_workload(w) as ctx:
        i = ctx.info
        assert (i.grid, i.threads) == (blocks, 512)
        # f and the summaries (two parities, two values) of the blocks of one thread block
        per = -(-(n // i.block[0]) // blocks)
        assert i.smem_bytes == 4 * 2 * per * (4 + 2 * i.block[0])
    with kin.Context.from_workload(w, threads=128) as ctx:
        assert ctx.info.threads == 128


def test_chain_of_the_split_sweep(kin):
    w = workloads.vortex2d(seed=0, n=128, degree=2, tiles=4, velset=1)
    with kin.Context.from_workload(w) as ctx:
        split = ctx.info
    with kin.Context.from_workload(w, mem_budget=split.device_bytes - 256) as ctx:
        one = ctx.info
    assert split.threads == one.threads == 32
    assert split.grid == 3 * 64                       # one problem per block: 4 variables, 16 subdomains
    # two parities of 8 + 4 record and 3 face values per lane, 32 cells' inflow and outflow faces
    assert split.smem_bytes == 4 * (2 * 32 * (12 + 3) + 2 * 32 * 3)
    assert split.smem_bytes != one.smem_bytes


@pytest.mark.parametrize("prec,L,tiles,clustered", [("f64", 83, 4, False), ("f64", 64, 4, True), ("f64", 25, 4, True),
                                                    ("f64", 67, 1, False), ("f32", 331, 4, False), ("f32", 83, 2, True),
                                                    ("f64", 121, 8, True)])
def test_long_lookbacks_take_one_launch_per_step(kin, prec, L, tiles, clustered):
    # (blocks of one cell where the subdomain is a prime: 60 folds in FP32, 120 in FP64)
    n = L * tiles
    w = workloads.advection1d(seed=0, n=n, tiles=tiles, degree=3 if L == 121 else 1, dt=2.4 / n, precision=prec)
    with kin.Context.from_workload(w) as ctx:
        assert (ctx.info.threads == 512) == clustered
