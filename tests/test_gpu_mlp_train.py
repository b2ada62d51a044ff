"""The training launch (every optimiser step in one cooperative kernel)
against the gradient and Adam entry points called step by step, and the
normalisation's sums, at the edges of the kernels' sample groups (32) and
batches."""
import numpy as np
import pytest

from tests._common import mlp_random_features, mlp_random_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_0705_4371_gb300 import lbm
    lbm.load()
    assert torch.cuda.is_available()
    return torch, lbm


def _data(torch, seed, n):
    from paper_0705_4371_gb300 import inputs
    feat = torch.from_numpy(mlp_random_features(seed, n).astype(np.float32)).cuda()
    dmu = torch.from_numpy((0.05 * inputs.uniform(seed + 7, (n, 4))).astype(np.float32)).cuda()
    return feat, dmu


@pytest.mark.parametrize("n, batch, epochs", [(1, 4, 2), (31, 31, 1), (33, 32, 2), (70, 33, 2), (300, 1000, 2),
                                              (5000, 2048, 1), (9001, 4864, 1), (12000, 6001, 2)])
def test_train_equals_gradient_and_adam_steps(env, n, batch, epochs):
    # the two paths add the same FP32 products in different orders: gradients
    # agree to about 1e-6 of their norm, so every Adam update (at most ~lr per
    # entry) agrees to 1e-3 lr in the root mean square, all but gradients
    # cancelled to a thousandth of their typical size following their sign
    torch, lbm = env
    feat, dmu = _data(torch, 500 + n, n)
    p0 = torch.from_numpy(mlp_random_params(91).astype(np.float32)).cuda()
    lr0, lr1 = 2e-3, 5e-4
    a = p0.clone()
    losses = torch.full((epochs,), -1.0, dtype=torch.float32, device="cuda")
    lbm.mlp_train(a.data_ptr(), feat.data_ptr(), dmu.data_ptr(), n, batch, epochs, lr0, lr1, losses.data_ptr())
    b, g = p0.clone(), torch.zeros_like(p0)
    m, v = torch.zeros_like(p0), torch.zeros_like(p0)
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    nb = -(-n // batch)
    t, want = 0, []
    for _ in range(epochs):
        mean = 0.0
        for k in range(nb):
            i0, nn = k * batch, min(batch, n - k * batch)
            lr = lr0 * (lr1 / lr0) ** (t / (nb * epochs - 1) if nb * epochs > 1 else 0.0)
            t += 1
            lbm.mlp_grad(b.data_ptr(), feat[i0:].data_ptr(), dmu[i0:].data_ptr(), nn, g.data_ptr(), loss.data_ptr())
            lbm.mlp_adam(b.data_ptr(), g.data_ptr(), m.data_ptr(), v.data_ptr(), t, lr)
            mean += float(loss.item()) / nb
        want.append(mean)
    torch.cuda.synchronize()
    d = (a - b).double()
    assert torch.isfinite(a).all()
    assert float(d.square().mean().sqrt()) <= 1e-3 * lr0 * t
    assert not d[-12:].any()                      # the normalisation entries are not trained
    assert np.allclose(losses.cpu().numpy(), want, rtol=1e-4)


@pytest.mark.parametrize("n", [1, 255, 257, 100_003, 400_000])
def test_normalise_matches_fp64_sums(env, n):
    torch, lbm = env
    feat, dmu = _data(torch, 900 + n, n)
    p = torch.zeros(lbm.mlp_param_count(), dtype=torch.float32, device="cuda")
    lbm.mlp_normalise(p.data_ptr(), feat.data_ptr(), dmu.data_ptr(), n)
    torch.cuda.synchronize()
    f, d = feat.double(), dmu.double()
    mean = f.mean(0)
    var = (f * f).mean(0) - mean * mean
    istd = torch.where(var > 0, 1 / var.clamp_min(1e-300).sqrt(), torch.ones_like(var))
    want = torch.cat([mean, istd, (d * d).mean(0).sqrt()]).cpu().numpy()
    got = p[-12:].cpu().numpy().astype(np.float64)
    # FP64 sums of n terms in another order, then one FP32 rounding; the
    # variance is a difference of two sums (about 1e3 times smaller here)
    if n > 1:
        assert np.allclose(got, want, rtol=1.5e-7)
    else:
        assert np.allclose(got[[0, 1, 2, 3, 8, 9, 10, 11]], want[[0, 1, 2, 3, 8, 9, 10, 11]], rtol=1.5e-7)


def test_two_threads_train_at_once(env):
    # batches of one and of many sample groups need different amounts of shared
    # memory of one kernel; neither thread may disturb the other's launches
    import threading
    torch, lbm = env
    n, calls = 256, 400
    feat, dmu = _data(torch, 77, n)
    p0 = torch.from_numpy(mlp_random_params(91).astype(np.float32)).cuda()

    def train(batch):
        p = p0.clone()
        lbm.mlp_train(p.data_ptr(), feat.data_ptr(), dmu.data_ptr(), n, batch, 1, 1e-3, 1e-3, None, st[batch].cuda_stream)
        return p

    st = {b: torch.cuda.Stream() for b in (32, 256)}
    torch.cuda.synchronize()
    want = {}
    for b in st:
        with torch.cuda.stream(st[b]):
            want[b] = train(b)
    torch.cuda.synchronize()
    failed = []

    def work(batch):
        try:
            with torch.cuda.stream(st[batch]):
                for _ in range(calls):
                    p = train(batch)
                st[batch].synchronize()
                assert torch.equal(p, want[batch])
        except Exception as e:
            failed.append((batch, e))

    threads = [threading.Thread(target=work, args=(b,)) for b in st]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


def test_a_wait_that_gives_up_is_reported(env):
    # no polls: the first grid barrier gives up in every block, without a wait;
    # the later launches of the call (more than 65 536 steps) end at once
    torch, lbm = env
    feat, dmu = _data(torch, 31, 96)
    p0 = torch.from_numpy(mlp_random_params(91).astype(np.float32)).cuda()
    st = torch.cuda.current_stream().cuda_stream
    for epochs in (1, 30_000):
        p = p0.clone()
        lbm.mlp_train_bounded(p.data_ptr(), feat.data_ptr(), dmu.data_ptr(), 96, 32, epochs, 1e-3, 1e-3, 0, stream=st)
        with pytest.raises(lbm.LBError) as e:
            lbm.mlp_train_status(p.data_ptr(), st)
        assert e.value.code == lbm.LB_ERR_TIMEOUT
        assert torch.isnan(p[-12:]).all()
    # the context, the kernel and the same buffer go on as before
    a, b = p0.clone(), p
    b.copy_(p0)
    for q in (a, b):
        lbm.mlp_train(q.data_ptr(), feat.data_ptr(), dmu.data_ptr(), 96, 32, 2, 1e-3, 1e-3, None, st)
        lbm.mlp_train_status(q.data_ptr(), st)
    assert torch.isfinite(a).all() and torch.equal(a, b)
    with pytest.raises(lbm.LBError):
        lbm.mlp_train_bounded(a.data_ptr(), feat.data_ptr(), dmu.data_ptr(), 96, 32, 1, 1e-3, 1e-3, -1)


def test_more_steps_than_a_launch(env):
    # launches of 65 536 steps: the next one goes on from the moments, the step
    # count and the epoch of the one before.  The tolerance of the test above
    # (1e-3 lr a step in the root mean square) and its losses
    torch, lbm = env
    n, batch, epochs, lr = 64, 32, 33_500, 1e-6
    feat, dmu = _data(torch, 41, n)
    p0 = torch.from_numpy(mlp_random_params(91).astype(np.float32)).cuda()
    a = p0.clone()
    losses = torch.zeros(epochs, dtype=torch.float32, device="cuda")
    lbm.mlp_train(a.data_ptr(), feat.data_ptr(), dmu.data_ptr(), n, batch, epochs, lr, lr, losses.data_ptr())
    b, g = p0.clone(), torch.zeros_like(p0)
    m, v = torch.zeros_like(p0), torch.zeros_like(p0)
    loss = torch.zeros(2, dtype=torch.float32, device="cuda")
    last = []
    for t in range(2 * epochs):
        i0 = batch * (t % 2)
        lbm.mlp_grad(b.data_ptr(), feat[i0:].data_ptr(), dmu[i0:].data_ptr(), batch, g.data_ptr(),
                     loss[t % 2:].data_ptr())
        lbm.mlp_adam(b.data_ptr(), g.data_ptr(), m.data_ptr(), v.data_ptr(), t + 1, lr)
        if t % 2 and t > 2 * epochs - 20:
            last.append(float(loss.mean()))
    torch.cuda.synchronize()
    moved = (b - p0).double().square().mean().sqrt()
    assert float((a - b).double().square().mean().sqrt()) <= 1e-3 * lr * 2 * epochs
    assert float(moved) > 1e-2 * lr * 2 * epochs       # (the bound is well below what the steps do)
    assert np.allclose(losses.cpu().numpy()[-len(last):], last, rtol=1e-4)
    # what the first launch alone gives is another result
    c = p0.clone()
    lbm.mlp_train(c.data_ptr(), feat.data_ptr(), dmu.data_ptr(), n, batch, 32_768, lr, lr, None)
    lbm.mlp_train_status(c.data_ptr())
    assert torch.isfinite(c).all() and not torch.equal(a, c)
