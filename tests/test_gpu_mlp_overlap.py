"""nbody_mlp_eval with arrays that share memory gives what it gives with arrays
of their own: every input is read as it was before the call."""
import ctypes as C

import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402

P = nb.MLP_PARAMS


def evaluate(n, feat, target, w, norm, pred, grad, loss):
    lib = nb.nbody.load()
    ptr = lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
    torch.cuda.synchronize()
    st = lib.nbody_mlp_eval(C.c_int64(n), ptr(feat), ptr(target), ptr(w), ptr(norm), ptr(pred), ptr(grad),
                            ptr(loss), None)
    assert st == 0


@pytest.mark.parametrize("n", [1, 65, 20011])
@pytest.mark.parametrize("shared", ["pred=targets", "pred in features", "grad=params", "loss in norm",
                                    "loss in targets", "pred in params"])
def test_shared_memory(n, shared):
    if shared == "pred in params" and n > P:
        pytest.skip("pred is larger than params")
    g = ics.rng(93)
    host = [g.normal(1.0, 2.0, 8 * n), g.normal(0.0, 1.0, n), g.uniform(-0.4, 0.4, P), np.full(16, 2.0)]
    make = lambda: ([torch.from_numpy(h.astype(np.float32)).cuda() for h in host] +  # noqa: E731
                    [torch.zeros(k, device="cuda") for k in (n, P, 1)])
    want = make()
    evaluate(n, *want)
    got = make()
    feat, target, w, norm = got[:4]
    if shared == "pred=targets":
        got[4] = target
    elif shared == "pred in features":
        got[4] = feat[7 * n // 2:7 * n // 2 + n]
    elif shared == "grad=params":
        got[5] = w
    elif shared == "loss in norm":
        got[6] = norm[9:10]
    elif shared == "loss in targets":
        got[6] = target[n - 1:]
    else:
        got[4] = w[P - n:]
    evaluate(n, *got)
    for a, b in zip(got[4:], want[4:]):
        assert torch.equal(a, b)


def test_outputs_that_share_memory():
    """pred, then grad, then loss are written: the last one is whole."""
    n, g = 1000, ics.rng(94)
    ins = [torch.from_numpy(h.astype(np.float32)).cuda() for h in
           (g.normal(1.0, 2.0, 8 * n), g.normal(0.0, 1.0, n), g.uniform(-0.4, 0.4, P), np.full(16, 2.0))]
    own = [torch.zeros(k, device="cuda") for k in (n, P, 1)]
    evaluate(n, *ins, *own)
    buf = torch.zeros(2000, device="cuda")
    evaluate(n, *ins, buf[:n], buf[500:500 + P], buf[600:601])
    assert torch.equal(buf[:500], own[0][:500])
    assert torch.equal(buf[500:600], own[1][:100]) and torch.equal(buf[601:500 + P], own[1][101:])
    assert torch.equal(buf[600:601], own[2])
