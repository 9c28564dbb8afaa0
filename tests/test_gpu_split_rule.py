"""Where the D2Q3 sweep is split (the context holds its records): few columns per
SM, several iterates or a high degree; elsewhere the sweep runs in one kernel
and nothing more is held."""
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


@pytest.mark.parametrize("degree,K,L,tiles,split", [
    (1, 1, 8, 4, False), (1, 1, 16, 4, True), (1, 1, 16, 8, False), (1, 1, 128, 2, False), (1, 2, 8, 12, True),
    (1, 2, 16, 4, True), (1, 2, 16, 8, False), (1, 3, 16, 12, True), (1, 3, 32, 4, True), (1, 3, 128, 4, False), (1, 3, 16, 32, False),
    (1, 4, 64, 4, True), (2, 1, 16, 8, True), (2, 1, 16, 12, False), (2, 2, 32, 12, True), (3, 1, 40, 8, False),
    (3, 1, 32, 6, True), (3, 1, 64, 4, True), (3, 2, 32, 8, True), (3, 2, 32, 12, False), (3, 2, 64, 6, True),
    (3, 3, 32, 12, True)])
def test_split_where_it_pays(kin, degree, K, L, tiles, split):
    w = workloads.vortex2d(seed=0, n=L * tiles, degree=degree, tiles=tiles, velset=1, iters=K)
    cells, slots = (L * tiles) ** 2, {1: 4, 2: 8, 3: 8}[degree]
    with kin.Context.from_workload(w) as ctx:
        rest = ctx.info.device_bytes - 4 * ctx.info.kinetic_values - 8 * ctx.info.state_values
        assert (rest >= 2 * 4 * 12 * cells * slots) == split
