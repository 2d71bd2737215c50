"""The cost model's stateless pass at the edges of its blocks of 64 samples, with
host and device arrays in every role, against the FP64 oracle (weights rounded
to BF16 as the kernels use them), and from several threads and streams at once."""
import threading

import numpy as np
import pytest

import ics
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1811_02761_gb300 as nb  # noqa: E402


def inputs(n, seed):
    g = ics.rng(seed)
    feat = g.normal(1.0, 2.0, (n, 8)).astype(np.float32)
    target = g.normal(0.0, 1.0, n).astype(np.float32)
    w = g.uniform(-0.4, 0.4, nb.MLP_PARAMS).astype(np.float32)
    norm = np.concatenate([np.full(8, 1.0), np.full(8, 2.0)]).astype(np.float32)
    return feat, target, w, norm


def reference(feat, target, w, norm):
    wr = torch.from_numpy(w).to(torch.bfloat16).float().numpy().astype(np.float64)
    return oracle.mlp_eval(feat.astype(np.float64), target.astype(np.float64), wr,
                           None if norm is None else norm.astype(np.float64))


def check(got, want):
    # FP32 sums of up to 32 products per layer and of the block's samples
    for g, r in zip(got, want):
        r = np.asarray(r)
        assert np.max(np.abs(np.asarray(g) - r)) <= 2e-5 * max(np.abs(r).max(), 1e-3)


@pytest.mark.parametrize("n", [1, 2, 31, 63, 64, 65, 127, 129, 4097])
@pytest.mark.parametrize("where", ["host", "device", "mixed"])
def test_eval_at_block_edges(n, where):
    feat, target, w, norm = inputs(n, 81)
    want = reference(feat, target, w, norm)
    a = [feat, target, w, norm]
    if where == "device":
        a = [torch.from_numpy(v).cuda() for v in a]
    elif where == "mixed":
        a = [torch.from_numpy(feat).cuda(), target, torch.from_numpy(w).cuda(), norm]
    pred, grad, loss = nb.nbody_mlp_eval(*a)
    check((pred, grad, loss), want)


def test_unaligned_device_features():
    feat, target, w, _ = inputs(100, 82)
    buf = torch.zeros(801, device="cuda")
    buf[1:] = torch.from_numpy(feat.ravel()).cuda()
    pred, grad, loss = nb.nbody_mlp_eval(buf[1:], target, w)
    check((pred, grad, loss), reference(feat, target, w, None))


def test_eval_from_threads_on_streams():
    cases = [inputs(n, 90 + n) for n in (500, 3000, 64, 20000)]
    want = [reference(*c) for c in cases]
    bad = []

    def work(k):
        stream = torch.cuda.Stream()
        for _ in range(10):
            try:
                check(nb.nbody_mlp_eval(*cases[k], stream=stream), want[k])
            except Exception as e:  # noqa: BLE001
                bad.append((k, repr(e)))
                return

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(cases))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
