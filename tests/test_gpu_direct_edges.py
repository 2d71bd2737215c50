"""The direct sum at the edges of its target blocks, source chunks and tiles.

One target block is 96 targets, a tile 512 sources, and below 8192 blocks
eight CTAs share the sources in chunks of a multiple of 16.  Reference: the
same sum in FP64 with torch.  Tolerances: compensated 1e-5 relative to the
largest |a| (as the other tests of this kernel), plain n 2^-24 / 16 for a
lane's chain on top of it.
"""
import pytest

import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402


def reference(X, m, eps):
    d = [c[None, :] - c[:, None] for c in X]
    r2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2 + eps * eps
    w = torch.where(r2 > 0, r2, torch.ones_like(r2)) ** -0.5
    w.fill_diagonal_(0.0)
    return [((w ** 3 * c) @ m) for c in d] + [-(w @ m)]


@pytest.mark.parametrize("n", [1, 2, 95, 96, 97, 127, 129, 511, 512, 513, 4095, 4097, 8193])
@pytest.mark.parametrize("eps", [1.0 / 64, 0.0])
@pytest.mark.parametrize("comp", [0, 1])
def test_direct_sum_at_block_and_tile_edges(n, eps, comp):
    p = ics.plummer(n, 41)
    X = [torch.from_numpy(p[k]).cuda() for k in ("x", "y", "z", "m")]
    ref = reference([t.double() for t in X[:3]], X[3].double(), eps)
    out = [torch.full((n,), float("nan"), device="cuda") for _ in range(4)]
    nb.nbody_direct(*X, 1.0, eps, comp, *out)
    three = [torch.full((n,), float("nan"), device="cuda") for _ in range(3)]
    nb.nbody_direct(*X, 1.0, eps, comp, *three)
    tol = 1e-5 + (0.0 if comp else n * 2.0 ** -24 / 16)
    for group in (range(3), [3]):
        scale = max(float(ref[c].abs().max()) for c in group) + 1e-30
        for c in group:
            assert float((out[c].double() - ref[c]).abs().max()) <= tol * scale
    for c in range(3):
        assert float((three[c].double() - out[c].double()).abs().max()) <= \
            tol * (max(float(ref[k].abs().max()) for k in range(3)) + 1e-30)
