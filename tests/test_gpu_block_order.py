"""Block steps sum in one fixed order (walk_ordered.cuh).

With steps of dt = 1/8 the FP32 rounding of the accelerations reaches the FP64
positions, so a run followed with block steps has to end where it always ended:
the positions after two calls are compared, bit by bit, with those recorded
from the library when every walk was one warp per group in this order.  The
state is made of FP32 products of random integers, exact on every machine, so
that only the library's own arithmetic is recorded.
"""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402


def state(n, seed):
    """A cluster with a dense middle: uniform in a cube, drawn inwards by |u|^2."""
    g = np.random.Generator(np.random.PCG64(seed))
    ints = lambda: g.integers(-2 ** 20, 2 ** 20, (3, n)).astype(np.float32) / np.float32(2 ** 20)  # noqa: E731
    u, w = ints(), ints()
    r2 = (u * u).max(axis=0)
    x = u * r2 * np.float32(4)
    return x.astype(np.float64), w * np.float32(0.5), -u * r2


def positions(n, seed, calls=2, **config):
    x, v, a = state(n, seed)
    dev = lambda t: [torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in t]  # noqa: E731
    X, V, A = dev(x), dev(v), dev(a)
    M = torch.full((n,), 1.0 / n, device="cuda", dtype=torch.float32)
    ctx = nb.nbody_create(nb.nbody_config_default(eps=1.0 / 64, block_levels=6, **config))
    try:
        for _ in range(calls):
            nb.nbody_step(ctx, *X, *V, M, *A, 1.0 / 8, 1)
    finally:
        nb.nbody_destroy(ctx)
    return np.stack([t.cpu().numpy() for t in X])


CASES = [
    (1500, 1, {}, "c1af56381c1b7efb"),
    (3001, 2, dict(rebuild_interval=4), "85599f2e61debd5a"),
    (8193, 3, dict(rebuild_interval=4, compensated=1), "08098f0faa2554ae"),
    (20011, 4, dict(quadrupole=1), "033900f2e2d55c90"),
    (140001, 5, dict(group_size=32), "08894d3732786748"),
]


@pytest.mark.parametrize("n,seed,config,recorded", CASES)
def test_positions_after_two_calls(n, seed, config, recorded):
    assert hashlib.sha256(positions(n, seed, **config).tobytes()).hexdigest()[:16] == recorded


def run_from_first_forces(n, seed, **config):
    """Forces and potential without |a_old|, then one call of block steps."""
    x, v, _ = state(n, seed)
    dev = lambda t: [torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in t]  # noqa: E731
    X, V = dev(x), dev(v)
    M = torch.full((n,), 1.0 / n, device="cuda", dtype=torch.float32)
    A = [torch.empty(n, device="cuda", dtype=torch.float32) for _ in range(4)]
    ctx = nb.nbody_create(nb.nbody_config_default(eps=1.0 / 64, block_levels=6, want_potential=1, **config))
    try:
        nb.nbody_build(ctx, *[t.float() for t in X], M)
        nb.nbody_walk(ctx, None, *A)
        first = torch.stack(A).cpu().numpy()
        nb.nbody_step(ctx, *X, *V, M, *A[:3], 1.0 / 8, 1)
    finally:
        nb.nbody_destroy(ctx)
    return np.concatenate([first.ravel().view(np.uint8), np.stack([t.cpu().numpy() for t in X]).ravel().view(np.uint8)])


FIRST = [
    (2000, 6, {}, "3bb0e24b4aa66e39"),
    (9001, 7, dict(compensated=1, rebuild_interval=4), "45c6109f2b555608"),
    (30011, 8, dict(quadrupole=1), "8b9f14fab04d2c16"),
    (150001, 9, dict(group_size=48), "89ff0105e60c8085"),
]


@pytest.mark.parametrize("n,seed,config,recorded", FIRST)
def test_run_from_its_first_forces(n, seed, config, recorded):
    got = run_from_first_forces(n, seed, **config)
    assert hashlib.sha256(got.tobytes()).hexdigest()[:16] == recorded
