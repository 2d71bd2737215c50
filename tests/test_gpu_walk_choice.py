"""Which walk takes a call: one warp per group or the cooperative walk, and
whether groups may be cut, depend on the sizes of the systems and the groups.

With |a_old| = 0 no node of more than one point is accepted, so every list holds
its whole system and the forces are each system's direct sum, whichever walk
ran.  How many kernels a walk launched tells which: beside the order of |a_old|,
alpha and the costs (three), one without groups that may be cut, two
cooperatively with parts that may be cut, three for one warp per group, cut.
"""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def forest(sizes, seed):
    parts = [ics.plummer(int(k), seed + i % 7) for i, k in enumerate(sizes)]
    p = [np.concatenate([q[c] for q in parts]) for c in ("x", "y", "z", "m")]
    return [dev(c) for c in p], np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def check(X, off, config):
    n = int(off[-1])
    ctx = nb.nbody_create(nb.nbody_config_default(eps=1 / 64, **config))
    try:
        a = [torch.empty(n, device="cuda") for _ in range(3)]
        if off.size == 2:
            nb.nbody_build(ctx, *X)
        else:
            nb.nbody_build_batched(ctx, off, None, *X)
        st = nb.nbody_walk(ctx, torch.zeros(n, device="cuda"), *a)
    finally:
        nb.nbody_destroy(ctx)
    k = np.argsort(np.diff(off))[-1]  # the largest system, and a few others
    for s in {int(k), 0, off.size // 2 - 1, off.size - 2}:
        sl = slice(int(off[s]), int(off[s + 1]))
        r = [torch.empty(sl.stop - sl.start, device="cuda") for _ in range(3)]
        nb.nbody_direct(*[t[sl].contiguous() for t in X], 1.0, 1 / 64, 1, *r)
        got = torch.stack([t[sl] for t in a]).double()
        want = torch.stack(r).double()
        # FP32 sums of up to 25000 terms: n 2^-24 / 32 of a lane's chain, 1e-4
        assert float((got - want).norm()) <= 1e-4 * float(want.norm()) + 1e-12
    return st.kernels - 3


@pytest.mark.parametrize("sizes,config,walks", [
    ([4000], {}, 1),                                    # cooperative, nothing to cut
    ([4096], {}, 1),
    ([4097], {}, 2),
    ([20000], {}, 2),
    ([60], {}, 1),                                      # one warp per group, nothing to cut
    ([256], dict(compensated=1), 1),
    ([10] * 1200, {}, 1),
    ([40] * 2500, {}, 1),
    ([300] * 300, dict(group_size=16), 1),
    ([25000] + [10] * 9000, dict(group_size=24), 3),    # one warp per group, groups cut
])
def test_forces_and_kernels(sizes, config, walks):
    X, off = forest(sizes, 101)
    assert check(X, off, config) == walks


def test_step_graph_follows_the_sizes():
    """Two forests of equal particles and systems: the graph captured for one,
    where no group can be cut, must not serve the other."""
    n = 26000
    even, odd = [10] * (n // 10), [23401] + [1] * (n // 10 - 1)
    assert sum(odd) == n
    res = []
    for first in (even, None):
        X, off = forest(odd, 102)
        ctx = nb.nbody_create(nb.nbody_config_default(eps=1 / 64, delta_acc=2.0 ** -9, use_graph=1, group_size=24))
        try:
            for sizes in ([first] if first else []) + [odd]:
                Y, off = forest(sizes, 102)
                x = [t.double() for t in Y[:3]]
                v = [torch.zeros(n, device="cuda") for _ in range(3)]
                a = [torch.zeros(n, device="cuda") for _ in range(3)]
                st = nb.nbody_step_batched(ctx, off, None, *x, *v, Y[3], *a, 1 / 256, 5)
            res.append(torch.stack(a).cpu())
        finally:
            nb.nbody_destroy(ctx)
    assert torch.equal(res[0], res[1])
