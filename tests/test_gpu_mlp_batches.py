"""The selector network's batch kernels at the sizes where their tiles of
eight samples begin and end, and training inside one cluster (batches of up to
512 samples, sixteen ranks of 16 at a time) or as launches per step, against the
float64 oracle with the same sample order."""
import numpy as np
import pytest

from oracle import mlp as M

zf = pytest.importorskip("paper_2602_08190_gb300")
pytestmark = pytest.mark.gpu


def _batch(seed, B):
    rng = np.random.default_rng(seed)
    X = rng.normal(size=(B, M.IN)).astype(np.float32)
    y = rng.integers(0, M.OUT, B).astype(np.int32)
    mask = rng.random((B, M.OUT)) < 0.7
    mask[np.arange(B), y] = True
    return X, y, mask


# FP32 sums of at most 64 products (forward) and of B samples' terms of size
# |g| (gradient): 64 * 2^-24 and B * 2^-24 relative to the largest value, here
# at most 3e-5 for B = 513; 1e-4 as in the repository's other test of them
@pytest.mark.parametrize("B", [1, 7, 8, 9, 16, 255, 513])
def test_forward_and_gradient(B):
    import torch
    net = zf.zf_mlp_create(0, 3)
    try:
        p = zf.zf_mlp_get_params(net).astype(np.float64)
        X, y, mask = _batch(B, B)
        dx, dy = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
        dm = torch.from_numpy(mask.astype(np.uint8)).cuda()
        dz = torch.full((B + 1, M.OUT), 7.0, dtype=torch.float32, device="cuda")
        dg = torch.full((M.NPARAMS + 1,), 7.0, dtype=torch.float32, device="cuda")
        dl = torch.full((2,), 7.0, dtype=torch.float32, device="cuda")
        zf.zf_mlp_forward(net, dx.data_ptr(), B, dz.data_ptr())
        zf.zf_mlp_grad(net, dx.data_ptr(), dy.data_ptr(), dm.data_ptr(), B, dg.data_ptr(), dl.data_ptr())
        torch.cuda.synchronize()
        z_ref, _ = M.forward(p, X.astype(np.float64))
        loss_ref, g_ref = M.loss_grad(p, X.astype(np.float64), y, mask)
        z, g = dz.cpu().numpy(), dg.cpu().numpy()
        assert np.max(np.abs(z[:B] - z_ref)) <= 1e-4 * max(1.0, np.max(np.abs(z_ref)))
        assert np.max(np.abs(g[:-1] - g_ref)) <= 1e-4 * np.max(np.abs(g_ref))
        assert abs(dl[0].item() - loss_ref) <= 1e-5 + 1e-4 * abs(loss_ref)
        assert (z[B] == 7).all() and g[-1] == 7 and dl[1].item() == 7
        assert np.array_equal(zf.zf_mlp_predict(net, X, mask), np.where(mask, z[:B], -np.inf).argmax(1))
    finally:
        zf.zf_mlp_destroy(net)


def _splitmix(x):
    m = (1 << 64) - 1
    x = (x + 0x9E3779B97F4A7C15) & m
    x = ((x ^ (x >> 30)) * 0xBF58476D1CE4E5B9) & m
    x = ((x ^ (x >> 27)) * 0x94D049BB133111EB) & m
    return x ^ (x >> 31)


def _order(n, seed):
    o = np.arange(n)
    for i in range(n, 1, -1):
        j = min(int(((_splitmix(seed ^ _splitmix(i)) >> 11) + 0.5) / 9007199254740992.0 * i), i - 1)
        o[i - 1], o[j] = o[j], o[i - 1]
    return o


@pytest.mark.parametrize("count,batch,epochs", [(5, 8, 3), (100, 33, 2), (300, 256, 2), (257, 257, 2), (512, 512, 2), (1100, 512, 2), (516, 257, 2), (700, 300, 2), (1100, 513, 2), (600, 4000, 3)])
def test_training_matches_float64(count, batch, epochs):
    X, y, mask = _batch(count, count)
    net = zf.zf_mlp_create(0, 21)
    try:
        p = zf.zf_mlp_get_params(net).astype(np.float64)
        losses = zf.zf_mlp_train(net, X, y, mask.astype(np.uint8), epochs, batch, 1e-3, seed=9)
        mean, sd = zf.zf_mlp_get_scaling(net)
        xs = ((X - mean) / sd).astype(np.float64)
        m, v, t = np.zeros_like(p), np.zeros_like(p), 0
        for e in range(epochs):
            order, ls = _order(count, 9 + e), []
            for b0 in range(0, count, batch):
                i = order[b0:b0 + batch]
                loss, g = M.loss_grad(p, xs[i], y[i], mask[i])
                t += 1
                p, m, v = M.adam(p, g, m, v, t, 1e-3)
                ls.append(loss)
            assert abs(losses[e] - np.mean(ls)) <= 1e-4 * abs(np.mean(ls))
        # a gradient below FP32 rounding may move its weight the other way in a step of size lr: at most
        # 2 lr for each of a few steps (6e-3), on average the 4e-5 such flips were seen to leave
        d = np.abs(zf.zf_mlp_get_params(net) - p)
        assert d.max() <= 6e-3 and d.mean() <= 4e-5
    finally:
        zf.zf_mlp_destroy(net)


# The epochs of a call are shuffled and uploaded in groups of 1, 2, 4, ... and
# each group runs in one launch (batches above 512: an epoch per upload); one
# epoch at a time nothing is uploaded twice and no launch holds two epochs.
# The arithmetic is the same, so the bits are.
@pytest.mark.parametrize("count,batch,epochs", [(300, 256, 8), (64, 64, 70), (700, 300, 9), (1100, 512, 8), (516, 257, 5), (1100, 600, 7),
                                                (20_000, 500, 12), (20_000, 700, 6)])
def test_a_call_trains_as_its_epochs_one_by_one(count, batch, epochs):
    X, y, mask = _batch(count + 1, count)
    mask = mask.astype(np.uint8)
    a, b = zf.zf_mlp_create(0, 4), zf.zf_mlp_create(0, 4)
    try:
        together = zf.zf_mlp_train(a, X, y, mask, epochs, batch, 1e-3, seed=17)
        single = [zf.zf_mlp_train(b, X, y, mask, 1, batch, 1e-3, seed=17 + e)[0] for e in range(epochs)]
        assert np.array_equal(together, np.array(single, together.dtype))
        assert np.array_equal(zf.zf_mlp_get_params(a), zf.zf_mlp_get_params(b))
    finally:
        zf.zf_mlp_destroy(a)
        zf.zf_mlp_destroy(b)
