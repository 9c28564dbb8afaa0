"""A state set by a captured call: a graph that sets the state of a D2Q3 context
(FP32) may be replayed at any time, and the steps after it start from that
state, whether they were captured or not."""
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


@pytest.mark.parametrize("setter", ["state", "kinetic", "kinetic_async"])
def test_replayed_setter(kin, setter):
    import torch
    w = workloads.vortex2d(seed=3, n=24, degree=2, tiles=2, dt_mult=4.0, velset=1)
    st, own = torch.cuda.Stream(), torch.cuda.Stream()
    W = torch.from_numpy(np.ascontiguousarray(w.W0.reshape(-1))).cuda()
    torch.cuda.synchronize()
    # (an asynchronous copy may go to another stream than the context's)
    with kin.Context.from_workload(w, stream=(own if setter == "kinetic_async" else st).cuda_stream) as ctx:
        ctx.set_state(W)
        f0 = ctx.get_kinetic()
        ctx.step(3)
        want = ctx.get_kinetic()
        fd, fh = torch.from_numpy(f0).cuda(), torch.from_numpy(f0).pin_memory()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            if setter == "state":
                ctx.set_state(W)
            elif setter == "kinetic":
                ctx.set_kinetic(fd)
            else:
                kin.kin_set_kinetic_async(ctx.ctx, fh, st.cuda_stream)
        for steps in (1, 2):
            ctx.step(steps)                # the records of the next step are those of this state
            ctx.sync()
            with torch.cuda.stream(st):
                g.replay()
            torch.cuda.synchronize()
            ctx.step(3)
            assert np.array_equal(ctx.get_kinetic(), want)
