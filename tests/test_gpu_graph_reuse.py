"""A step graph captured by one call serves the next ones, whatever the number
of steps: the profiler's record of the second and later calls has graph
launches and no instantiation."""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402


@pytest.mark.parametrize("n", [1000, 8192, 8193, 20011])
@pytest.mark.parametrize("steps", [3, 4, 5, 6])
def test_no_capture_after_the_first_calls(n, steps):
    from torch.profiler import ProfilerActivity, profile

    p = ics.plummer(n, 96)
    dev = lambda t: torch.from_numpy(np.ascontiguousarray(t)).cuda()  # noqa: E731
    X = [dev(p[k].astype(np.float64)) for k in ("x", "y", "z")]
    V = [dev(p[k]) for k in ("vx", "vy", "vz")]
    A, M = [torch.zeros(n, device="cuda") for _ in range(3)], dev(p["m"])
    ctx = nb.nbody_create(nb.nbody_config_default(eps=1 / 64, use_graph=1))
    try:
        # the first call has no order to start its first sort from: a sort of
        # its own, after which the buffers lie as they then stay from call to call
        for _ in range(2):
            nb.nbody_step(ctx, *X, *V, M, *A, 1 / 256, steps)
        with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]):
            torch.cuda.synchronize()  # a process's first record may be empty
        with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as prof:
            for _ in range(3):
                nb.nbody_step(ctx, *X, *V, M, *A, 1 / 256, steps)
            torch.cuda.synchronize()
    finally:
        nb.nbody_destroy(ctx)
    names = [e.name for e in prof.events()]
    launches = sum("GraphLaunch" in k for k in names)
    if not launches:
        pytest.skip("the profiler records no graph launches here")
    assert launches >= 3 * ((steps - 1) // 2)
    assert not [k for k in names if "GraphInstantiate" in k or "BeginCapture" in k]
