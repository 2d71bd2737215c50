"""Cubes where 32 particles hold one, few or many systems (empty ones among
them): the extents are merged per system or per particle, and both give the
oracle's cube, twice on one context."""
import numpy as np
import pytest

import ics
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402


@pytest.mark.parametrize("lo,hi", [(1, 2), (0, 3), (6, 10), (8, 9), (7, 8), (20, 40), (0, 300)])
@pytest.mark.parametrize("nsys", [70, 2100])
def test_cubes(lo, hi, nsys):
    sizes = ics.rng(97).integers(lo, hi, nsys)
    sizes[-1] = 1
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    ctx = nb.nbody_create(nb.nbody_config_default())
    try:
        for seed in (98, 99):
            g = ics.rng(seed)
            p = [g.normal(size=n).astype(np.float32) for _ in range(3)]
            nb.nbody_build_batched(ctx, off, None, *[torch.from_numpy(c).cuda() for c in p],
                                   torch.ones(n, device="cuda"))
            box = nb.nbody_export(ctx, nb.nbody.EXPORT_SYS_BOX)
            for s in range(nsys):
                sl = slice(off[s], off[s + 1])
                want = oracle.cube(*[c[sl] for c in p]) if sizes[s] else np.array([0, 0, 0, 1], np.float32)
                assert np.array_equal(box[s], want)
    finally:
        nb.nbody_destroy(ctx)
