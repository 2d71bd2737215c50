"""Sizes around which the counting sort's keys and its own shared memory pass
the 48 KB that a kernel may use without asking: each in a process of its own,
since a larger build before it leaves the kernel's limit raised."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

RUN = """
import sys
import numpy as np, torch
import ics, oracle, paper_1811_02761_gb300 as nb
n = int(sys.argv[1])
p = ics.plummer(n, 91)
c = nb.nbody_create(nb.nbody_config_default())
nb.nbody_build(c, *[torch.from_numpy(p[k]).cuda() for k in ("x", "y", "z", "m")])
perm = nb.nbody_export(c, nb.nbody.EXPORT_PERM)
k, _ = oracle.keys(p["x"], p["y"], p["z"], 21)
assert np.array_equal(perm, oracle.sort_order(k))
nb.nbody_destroy(c)
"""


@pytest.mark.parametrize("n", [6016, 6017, 6144, 6145])
def test_first_build_of_a_process(n):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RUN, str(n)], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
