"""Node records are complete when their parent reads them.

The climbing moments pass hands records from lane to lane and from SM to SM.
Builds of two particle sets alternate on one context, over the same memory, so
a parent formed from a record that was not there yet would hold the other set's
numbers: every record has to repeat bit for bit.
"""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402

E = nb.nbody
RECORDS = (E.EXPORT_NODE_COUNT, E.EXPORT_NODE_A, E.EXPORT_NODE_B, E.EXPORT_NODE_Q)


@pytest.mark.parametrize("n,cap", [(8193, 16), (20011, 1), (150001, 8)])
def test_records_repeat(n, cap):
    sets = [[torch.from_numpy(np.ascontiguousarray(p[k])).cuda() for k in ("x", "y", "z", "m")]
            for p in (ics.plummer(n, 81), ics.hernquist(n, 82))]
    ctx = nb.nbody_create(nb.nbody_config_default(leaf_cap=cap, quadrupole=1))
    try:
        want = [None, None]
        for k in range(12):
            nb.nbody_build(ctx, *sets[k % 2])
            got = [nb.nbody_export(ctx, r) for r in RECORDS]
            want[k % 2] = want[k % 2] or got
            assert all(np.array_equal(a, b) for a, b in zip(got, want[k % 2]))
    finally:
        nb.nbody_destroy(ctx)
