"""The cooperative walk and the groups cut at the quota.

A group whose members have |a_old| = 0 accepts no node that holds more than
one point (Eq. 2 with a right side of 0), so its list must hold every particle
of its system exactly once -- whichever kernels walked it, however often it was
cut and into however many parts -- and its members' forces must be the direct
sum.  The sizes take the routes in turn: one group of several parts; parts of
one CTA; parts cut and walked again; the last size walked cooperatively and
the first walked by one warp per group, whose long groups are cut there.
"""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402

EPS = 1 / 128


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def opened_groups(p, quad, comp, phi, zero_at):
    """Costs of the groups holding the particles zero_at (|a_old| = 0 there),
    and the walk's accelerations (and potential) at those particles."""
    n = p["x"].size
    X = [dev(p[k]) for k in ("x", "y", "z", "m")]
    ctx = nb.nbody_create(nb.nbody_config_default(eps=EPS, quadrupole=quad, compensated=comp,
                                                  want_potential=phi))
    try:
        out = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(3 + phi)]
        nb.nbody_build(ctx, *X)
        nb.nbody_walk(ctx, None, *out)
        aold = torch.sqrt(out[0] ** 2 + out[1] ** 2 + out[2] ** 2)
        aold[torch.from_numpy(zero_at).cuda()] = 0.0
        st = nb.nbody_walk(ctx, aold, *out)
        first = nb.nbody_export(ctx, nb.nbody.EXPORT_GROUP_FIRST)
        count = nb.nbody_export(ctx, nb.nbody.EXPORT_GROUP_COUNT)
        perm = nb.nbody_export(ctx, nb.nbody.EXPORT_PERM)
        cost = np.empty(first.size, np.int32)
        nb.nbody_get_group_costs(ctx, cost)
        rank = np.empty(n, np.int64)
        rank[perm] = np.arange(n)
        g = np.searchsorted(first, rank[zero_at], side="right") - 1
        assert st.interactions == int((cost.astype(np.int64) * count).sum())
        assert st.list_entries == int(cost.astype(np.int64).sum())
        return cost[g], [o.cpu().numpy()[zero_at].astype(np.float64) for o in out]
    finally:
        nb.nbody_destroy(ctx)


@pytest.mark.parametrize("n", [300, 5003, 20011, 60013, 131072, 131073, 200003])
@pytest.mark.parametrize("quad,comp,phi", [(0, 0, 0), (0, 1, 1), (1, 0, 1)])
def test_fully_opened_groups_are_the_direct_sum(n, quad, comp, phi):
    p = ics.plummer(n, 31)
    X = [dev(p[k]) for k in ("x", "y", "z", "m")]
    ref = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(4)]
    nb.nbody_direct(*X, 1.0, EPS, 1, *ref)
    ref = [r.cpu().numpy().astype(np.float64) for r in ref]
    amag = np.sqrt(sum(r ** 2 for r in ref[:3]))
    # particles where the forces hardly cancel, spread over three groups at most
    zero_at = np.argsort(amag)[[int(0.97 * n), int(0.98 * n), int(0.99 * n)]]
    cost, got = opened_groups(p, quad, comp, phi, zero_at)
    assert np.all(cost == n), cost
    # FP32 sums of n terms of one sign mostly: compensated to a few ulps of the
    # terms (2^-22 each), plain within n 2^-24 / 32 of a lane's chain
    tol = 2e-5 if comp else 1e-4
    for c in range(3):
        assert np.max(np.abs(got[c] - ref[c][zero_at]) / amag[zero_at]) <= tol
    if phi:
        assert np.max(np.abs(got[3] / ref[3][zero_at] - 1.0)) <= tol


def test_cut_groups_do_not_depend_on_the_queue_order():
    """Bitwise equal forces in Morton and in last-cost order, with groups cut
    by both kernels (the records of cut groups are taken in any order)."""
    for n in (60013, 200003):
        p = ics.plummer(n, 32)
        X = [dev(p[k]) for k in ("x", "y", "z", "m")]
        ctx = nb.nbody_create(nb.nbody_config_default(eps=EPS))
        try:
            out = [torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(3)]
            nb.nbody_build(ctx, *X)
            nb.nbody_walk(ctx, None, *out)
            aold = torch.sqrt(out[0] ** 2 + out[1] ** 2 + out[2] ** 2)
            aold[::4001] = 0.0
            res = []
            for sched in (nb.SCHED_MORTON, nb.SCHED_LASTCOST, nb.SCHED_MORTON):
                cfg = nb.nbody_get_config(ctx)
                cfg.schedule = sched
                nb.nbody_set_config(ctx, cfg)
                nb.nbody_walk(ctx, aold, *out)
                res.append([o.cpu().numpy().copy() for o in out])
        finally:
            nb.nbody_destroy(ctx)
        for r in res[1:]:
            for a, b in zip(res[0], r):
                assert np.array_equal(a, b)
