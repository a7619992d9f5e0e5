"""The ranker's gradient and training kernels at the edges of their tiles (16 rows per tile,
128 per CTA of a single gradient, ragged last batches), against the ranker oracle."""
import numpy as np
import pytest

from oracle import ranker as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2111_12478_gb300 import gwcp

    return torch, gwcp


def rows(seed, n):
    rng = np.random.default_rng(seed)
    x = np.abs(rng.normal(0, 1.5, (n, R.N_FEAT))).astype(np.float32)
    y = (rng.random(n) < 0.3).astype(np.float32)
    th = rng.normal(0, 0.25, R.N_PARAMS).astype(np.float32)
    return th, x, y


# a float sum of n terms is off by at most n * 2^-24 of the terms' sizes (40,000 * 6e-8 =
# 2.4e-3 of the largest entry), far less on average; one flipped bfloat16 rounding of a hidden
# unit moves one sample's share by 2^-8 of itself, 4e-3 / n of the sum
@pytest.mark.parametrize("n", [1, 15, 16, 17, 127, 128, 129, 4863, 4864, 4865, 40013])
def test_gradient_sizes(env, n):
    torch, gwcp = env
    th, x, y = rows(n, n)
    g, loss = gwcp.rank_grad(torch.from_numpy(th).cuda(), torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), 3.0)
    want = R.grad(th, x, y, 3.0)
    g = g.cpu().numpy().astype(np.float64)
    tol = 2.4e-3 if n > 16 else 4e-3
    assert np.linalg.norm(g - want) <= tol * np.linalg.norm(want)
    assert abs(loss - R.loss(th, x, y, 3.0)) < 1e-4 * (1 + abs(loss))


@pytest.mark.parametrize("n,batch", [(1, 8), (40, 16), (100, 33), (257, 256), (1000, 4096)])
def test_training_with_ragged_batches(env, n, batch):
    torch, gwcp = env
    th, x, y = rows(3 * n + batch, n)
    t = torch.from_numpy(th.copy()).cuda()
    tx, ty = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    losses = gwcp.rank_train(t, tx, ty, epochs=2, batch=batch, lr=1e-3, pos_weight=3.0)
    again = torch.from_numpy(th.copy()).cuda()
    gwcp.rank_train(again, tx, ty, epochs=2, batch=batch, lr=1e-3, pos_weight=3.0)
    assert torch.equal(t, again)  # sums in a fixed order
    want, m, v, step, means = th.astype(np.float64), np.zeros(R.N_PARAMS), np.zeros(R.N_PARAMS), 0, []
    nb = -(-n // batch)
    for _ in range(2):
        total = 0.0
        for q in range(nb):
            part = slice(q * batch, (q + 1) * batch)
            total += R.loss(want, x[part], y[part], 3.0) / nb
            step += 1
            want, m, v = R.adam_step(want, m, v, R.grad(want, x[part], y[part], 3.0) / nb, step, 1e-3)
        means.append(total)
    # a step moves a parameter by about lr whatever the gradient's size: an entry whose gradient
    # is lost in rounding may go either way at each step, the others follow
    assert np.abs(t.cpu().numpy() - want).max() <= 2.1e-3 * step
    assert np.linalg.norm(t.cpu().numpy() - want) <= 2e-3 * np.linalg.norm(want)
    np.testing.assert_allclose(losses, means, rtol=2e-3)
