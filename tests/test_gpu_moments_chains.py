"""Node moments where the nodes have few children: chains of single children
below coincident points, pairs on a line, up to four on a plane, beside ordinary
nodes.  Mass, centre and b_J of every node against FP64 sums over its members,
after a build and after a refit, and the quadrupoles of a few levels."""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402

E = nb.nbody


def points(kind, n):
    g = ics.rng(95)
    x = g.normal(size=(3, n)).astype(np.float32)
    if kind == "points":
        x = x[:, g.integers(0, max(n // 40, 1), n)]
    elif kind == "line":
        x[1:] = 0
    elif kind == "plane":
        x[2] = 0
    elif kind == "mixed":
        x[:, n // 2:] = x[:, g.integers(0, max(n // 40, 1), n - n // 2)]
    return np.ascontiguousarray(x), (g.uniform(0.5, 1.5, n) / n).astype(np.float32)


def check(ctx, x, m):
    perm = nb.nbody_export(ctx, E.EXPORT_PERM)
    start, count = nb.nbody_export(ctx, E.EXPORT_NODE_START), nb.nbody_export(ctx, E.EXPORT_NODE_COUNT)
    A, B = nb.nbody_export(ctx, E.EXPORT_NODE_A), nb.nbody_export(ctx, E.EXPORT_NODE_B)
    Q = nb.nbody_export(ctx, E.EXPORT_NODE_Q)
    xs, ms = x[:, perm].T.astype(np.float64), m[perm].astype(np.float64)
    for j in range(start.size):
        s = slice(start[j], start[j] + count[j])
        M = ms[s].sum()
        com = (ms[s, None] * xs[s]).sum(0) / M
        d = xs[s] - A[j, :3].astype(np.float64)
        r2 = (d ** 2).sum(1)
        # FP32 sums of offsets inside the node, as many as its levels below
        tol = 16 * 2.0 ** -24 * (B[j, 0] + np.abs(com).max())
        assert abs(A[j, 3] - M) <= 2.0 ** -22 * M
        assert np.abs(A[j, :3] - com).max() <= tol
        assert B[j, 0] >= np.sqrt(r2.max()) * (1 - 1e-12)
        if j % 7 == 0:  # Q_ab = sum m (3 d_a d_b - r^2 delta_ab)
            q = [(ms[s] * (3 * d[:, a] * d[:, b] - (r2 if a == b else 0))).sum()
                 for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
            # FP32 sums over the levels below: a few ulps of m b^2 each, and the
            # centres' own rounding against the distances
            assert np.abs(Q[j, :6] - q).max() <= M * B[j, 0] * (2.0 ** -18 * B[j, 0] + 64 * tol)


@pytest.mark.parametrize("kind", ["points", "line", "plane", "mixed"])
@pytest.mark.parametrize("n,cap", [(257, 1), (2191, 16), (2193, 16), (5000, 1), (12001, 16)])
def test_every_node(kind, n, cap):
    x, m = points(kind, n)
    X = [torch.from_numpy(c).cuda() for c in x] + [torch.from_numpy(m).cuda()]
    ctx = nb.nbody_create(nb.nbody_config_default(leaf_cap=cap, quadrupole=1))
    try:
        nb.nbody_build(ctx, *X)
        check(ctx, x, m)
        nb.nbody_refit(ctx, *X)
        check(ctx, x, m)
    finally:
        nb.nbody_destroy(ctx)
