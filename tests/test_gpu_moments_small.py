"""Node moments at the edges of the two passes: trees of up to 8192 particles
with leaves of at most 16 are done by one block (records in shared memory up to
4096 nodes, through L2 above), the rest by the climbing pass.  Checked against
FP64 sums over each node's own members: mass and centre of mass within FP32
rounding of the node's size, b_J covering every member, and the pass repeated
over the same positions (a refit) leaving mass and centre unchanged bit for bit.
"""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402

E = nb.nbody


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# leaf_cap 1 gives more than 4096 nodes from about 3000 particles on
@pytest.mark.parametrize("n,cap", [(1, 16), (17, 16), (2500, 1), (5000, 1), (8192, 1), (8192, 16), (8193, 16),
                                   (8192, 17), (20000, 8)])
def test_moments_of_every_node(n, cap):
    p = ics.plummer(n, 71)
    p["m"] = (ics.rng(72).uniform(0.5, 1.5, n) / n).astype(np.float32)
    ctx = nb.nbody_create(nb.nbody_config_default(leaf_cap=cap, group_size=max(32, cap)))
    try:
        X = [dev(p[k]) for k in ("x", "y", "z", "m")]
        nb.nbody_build(ctx, *X)
        perm = nb.nbody_export(ctx, E.EXPORT_PERM)
        start, count = nb.nbody_export(ctx, E.EXPORT_NODE_START), nb.nbody_export(ctx, E.EXPORT_NODE_COUNT)
        A, B = nb.nbody_export(ctx, E.EXPORT_NODE_A), nb.nbody_export(ctx, E.EXPORT_NODE_B)
        nb.nbody_refit(ctx, *X)
        A2 = nb.nbody_export(ctx, E.EXPORT_NODE_A)
    finally:
        nb.nbody_destroy(ctx)
    assert np.array_equal(A, A2)
    x = np.stack([p[k][perm].astype(np.float64) for k in ("x", "y", "z")], 1)
    m = p["m"][perm].astype(np.float64)
    for j in range(start.size):
        s = slice(start[j], start[j] + count[j])
        M = m[s].sum()
        com = (m[s, None] * x[s]).sum(0) / M
        far = np.sqrt(((x[s] - A[j, :3].astype(np.float64)) ** 2).sum(1)).max()
        # FP32 sums of offsets inside the node: a few ulps of its size, and the
        # rounding of the position itself
        tol = 16 * 2.0 ** -24 * (B[j, 0] + np.abs(com).max())
        assert abs(A[j, 3] - M) <= 2.0 ** -22 * M
        assert np.abs(A[j, :3] - com).max() <= tol
        assert B[j, 0] >= far * (1 - 1e-12)
