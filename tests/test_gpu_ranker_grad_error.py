"""The ranker's gradient held to the error of 32-bit sums over unrounded 32-bit products: a
kernel with the products of the backward pass in bfloat16 is off by 2^-9 / sqrt(n) and more."""
import numpy as np
import pytest

from oracle import ranker as R

pytestmark = pytest.mark.gpu


# 32-bit sums: 1e-7 to 4e-7 of the norm. A rounding of a hidden unit to bfloat16 that falls on
# the other side in 64 bits moves one unit of 64 (an eighth of the norm) of one sample's share
# by 2^-8, up to five times that where samples cancel: 2.5e-3 / n for one. A unit so close to
# zero that its mask falls on the other side comes about once in 100,000 rows, an eighth of a
# share: 1.6e-5 with the same factor at 40,000 rows.
@pytest.mark.parametrize("n", [1, 16, 17, 128, 129, 500, 4864, 4865, 40013])
def test_gradient_error(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2111_12478_gb300 import gwcp

    rng = np.random.default_rng(n)
    x = np.abs(rng.normal(0, 1.5, (n, R.N_FEAT))).astype(np.float32)
    y = (rng.random(n) < 0.3).astype(np.float32)
    th = rng.normal(0, 0.25, R.N_PARAMS).astype(np.float32)
    g, _ = gwcp.rank_grad(torch.from_numpy(th).cuda(), torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), 3.0)
    want = R.grad(th, x, y, 3.0)
    off = np.linalg.norm(g.cpu().numpy().astype(np.float64) - want)
    assert off <= (2e-5 + 2.5e-3 / n) * np.linalg.norm(want)
