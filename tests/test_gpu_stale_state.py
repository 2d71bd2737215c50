"""What a context keeps between calls does not outlive the groups it belongs to:
the cost model's features after a step call, then after a build of more
particles, and a step graph captured before the context saw more systems."""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def state(p):
    X = [dev(p[k].astype(np.float64)) for k in ("x", "y", "z")]
    V = [dev(p[k]) for k in ("vx", "vy", "vz")]
    return X, V, dev(p["m"])


def test_features_after_a_step_and_after_a_larger_build():
    ctx = nb.nbody_create(nb.nbody_config_default(eps=1 / 64))
    try:
        nb.nbody_mlp_set_params(ctx, ics.mlp_init(3))
        p = ics.plummer(3000, 91)
        X, V, m = state(p)
        A = [torch.zeros(3000, device="cuda") for _ in range(3)]
        nb.nbody_build(ctx, *[x.float() for x in X], m)
        nb.nbody_walk(ctx, None, *A)
        nb.nbody_step(ctx, *X, *V, m, *A, 1.0 / 256, 2)
        _, f = nb.nbody_mlp_predict(ctx, want_features=True)
        assert np.all(np.isfinite(f)) and f.shape[0] > 10
        assert nb.nbody_mlp_train(ctx, 1, 1e-3, 512) > 0
        q = ics.plummer(200000, 92)
        nb.nbody_build(ctx, *[dev(q[k]) for k in ("x", "y", "z", "m")])
        out = [torch.empty(200000, device="cuda") for _ in range(3)]
        nb.nbody_walk(ctx, None, *out)
        pred, f = nb.nbody_mlp_predict(ctx, want_features=True)
        assert np.all(np.isfinite(f)) and f.shape[0] > 1000
    finally:
        nb.nbody_destroy(ctx)


def test_graph_after_a_forest_of_more_systems():
    def run(between):
        ctx = nb.nbody_create(nb.nbody_config_default(eps=1 / 64, use_graph=1))
        try:
            p = ics.plummer(20000, 93)
            X, V, m = state(p)
            A = [torch.zeros(20000, device="cuda") for _ in range(3)]
            nb.nbody_step(ctx, *X, *V, m, *A, 1.0 / 256, 5)
            if between:  # an eager call that grows the systems' buffers
                b = ics.batched(50, 94, sizes=[100] * 50)
                Y, W, mm = state(b)
                B = [torch.zeros(5000, device="cuda") for _ in range(3)]
                nb.nbody_step_batched(ctx, b["offsets"], b["eps"], *Y, *W, mm, *B, 1.0 / 256, 1)
            nb.nbody_step(ctx, *X, *V, m, *A, 1.0 / 256, 5)
            return [t.cpu().numpy() for t in X + V + A]
        finally:
            nb.nbody_destroy(ctx)

    for a, b in zip(run(False), run(True)):
        assert np.array_equal(a, b)
