"""The training kernel (a cluster of CTAs shares every Adam step) against the
fp64 oracle over its edges: batches smaller than the cluster, around the 32
samples a CTA takes at a time, larger than the data, a ragged last batch.

Tolerance: a gradient element is a sum of at most K = 84 x batch products, so
its relative error is about K * 2^-24 times its condition number; Adam divides
it by its own magnitude, so a step (of length at most lr) is off by at most
lr * 1e-2 except for elements that nearly cancel (condition above 1e3), which
can be off by the whole step. Hence: all but 0.5% of the parameters within
1e-2 * lr * steps, and every one within 2 * lr * steps."""
import numpy as np
import pytest

from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1311_0378_gb300 as rc  # noqa: E402

M64 = (1 << 64) - 1


def mix(z):
    z = (z + 0x9E3779B97F4A7C15) & M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return z ^ (z >> 31)


def order(n, seed, epoch):
    perm, st = list(range(n)), mix(seed ^ mix(epoch + 1))
    for i in range(n - 1, 0, -1):
        st = mix(st)
        perm[i], perm[st % (i + 1)] = perm[st % (i + 1)], perm[i]
    return perm


@pytest.mark.parametrize("n,batch,epochs", [(1, 1, 2), (9, 1, 1), (40, 7, 2), (64, 8, 1), (300, 31, 1), (520, 256, 2),
                                            (777, 264, 2), (600, 599, 2), (250, 1000, 3)])
def test_epochs_match_oracle(n, batch, epochs):
    import paper_1311_0378_gb300.build as b
    b.build()
    rng = np.random.default_rng(n * 7 + batch)
    X = rng.uniform(0, 1, size=(n, 20)).astype(np.float32)
    T = np.stack([X[:, :5].sum(1) - 2.5, 2 * X[:, 5] - X[:, 6]], axis=1).astype(np.float32)
    lr, seed = 1e-3, 11
    theta = mlp.init(3).astype(np.float32)
    dth, dX, dT = (torch.from_numpy(a).cuda() for a in (theta.copy(), X, T))
    torch.cuda.synchronize()
    ctx = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    try:
        st, losses = rc.recon_mlp_train(ctx, dth.data_ptr(), dX.data_ptr(), dT.data_ptr(), n, epochs, batch, lr, seed)
    finally:
        rc.recon_free(ctx)
    rc.check(st, "recon_mlp_train")
    want, X, T = theta.astype(np.float64), X.astype(np.float64), T.astype(np.float64)
    m, v, t, sums = np.zeros_like(want), np.zeros_like(want), 0, []
    for e in range(epochs):
        perm, total, k = order(n, seed, e), 0.0, 0
        for s in range(0, n, batch):
            idx = perm[s:s + batch]
            Y, cache = mlp.forward(want, X[idx])
            total, k, t = total + mlp.loss(Y, T[idx]), k + 1, t + 1
            want, m, v = mlp.adam_step(want, mlp.backward(want, cache, Y, T[idx]), m, v, t, lr=lr)
        sums.append(total / k)
    off = np.abs(dth.cpu().numpy() - want)
    assert (off > 1e-2 * lr * t).mean() <= 5e-3 and off.max() <= 2 * lr * t
    np.testing.assert_allclose(losses, sums, rtol=1e-3)
