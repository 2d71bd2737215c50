"""The build's routes for small inputs: keys up to 8192 are sorted by counting
(in any order, ties by index), the groups of up to 65536 particles are compacted
by one block, and the cubes of up to 2048 systems come out of the extent pass.
Checked at the edges against the oracle's cube, keys and stable sort, and
against the group partition's own invariants, twice on one context so that the
buffers that every build has to leave clean are seen used.
"""
import numpy as np
import pytest

import ics
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402

E = nb.nbody


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def ties(n, seed):
    """Plummer particles of which many share one of a few positions."""
    p = ics.plummer(n, seed)
    k = ics.rng(seed, 9).integers(0, 5, n)
    for c in ("x", "y", "z"):
        p[c] = np.where(ics.rng(seed, 8).uniform(size=n) < 0.4, p[c][np.minimum(k, n - 1)], p[c]).astype(np.float32)
    return p


def check_groups(ctx, n, G):
    first, count = nb.nbody_export(ctx, E.EXPORT_GROUP_FIRST), nb.nbody_export(ctx, E.EXPORT_GROUP_COUNT)
    assert first[0] == 0 and count.min() >= 1 and count.max() <= G
    assert np.array_equal(first[1:], np.cumsum(count)[:-1]) and count.sum() == n


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 255, 257, 4095, 8191, 8192, 8193, 16384, 16385, 65535, 65536, 65537])
def test_one_system(n):
    ctx = nb.nbody_create(nb.nbody_config_default())
    try:
        for seed, make in ((51, ics.plummer), (52, ties), (53, ics.hernquist)):
            p = make(n, seed)
            nb.nbody_build(ctx, *[dev(p[k]) for k in ("x", "y", "z", "m")])
            k, cube = oracle.keys(p["x"], p["y"], p["z"], 21)
            order = oracle.sort_order(k)
            assert np.array_equal(nb.nbody_export(ctx, E.EXPORT_SYS_BOX)[0], cube)
            assert np.array_equal(nb.nbody_export(ctx, E.EXPORT_PERM), order.astype(np.int32))
            assert np.array_equal(nb.nbody_export(ctx, E.EXPORT_KEYS), k[order])
            check_groups(ctx, n, 64)
    finally:
        nb.nbody_destroy(ctx)


@pytest.mark.parametrize("nsys", [3, 2048, 2049, 5000])
def test_many_systems(nsys):
    """Systems of 0 to 5 particles: boxes, the order and the roots' ranges."""
    sizes = ics.rng(61).integers(0, 6, nsys)
    sizes[-1] = 3
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    ctx = nb.nbody_create(nb.nbody_config_default())
    try:
        for seed in (62, 63):
            g = ics.rng(seed)
            p = [g.normal(size=n).astype(np.float32) for _ in range(3)]
            m = np.full(n, 1.0, np.float32)
            nb.nbody_build_batched(ctx, off, None, *[dev(c) for c in p], dev(m))
            box = nb.nbody_export(ctx, E.EXPORT_SYS_BOX)
            perm = nb.nbody_export(ctx, E.EXPORT_PERM)
            assert np.array_equal(np.sort(perm), np.arange(n))
            assert np.array_equal(np.searchsorted(off, perm, side="right"),
                                  np.searchsorted(off, np.arange(n), side="right"))
            for s in range(nsys):
                sl = slice(off[s], off[s + 1])
                want = oracle.cube(*[c[sl] for c in p]) if sizes[s] else np.array([0, 0, 0, 1], np.float32)
                assert np.array_equal(box[s], want)
            out = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(3)]
            nb.nbody_walk(ctx, None, *out)  # every system finds its root
            alone = np.repeat(sizes == 1, sizes)
            a = np.sqrt(sum(o.cpu().numpy().astype(np.float64) ** 2 for o in out))
            assert np.all(a[alone] == 0) and np.all(a[~alone] > 0)
    finally:
        nb.nbody_destroy(ctx)
