"""The split damped solve at the edges of its blocks (64 columns) and strips (256)."""
import numpy as np
import pytest
import torch

from paper_2509_14185_gb300 import inputs as I
from tests.gpu_cases import gpu_problem

pytestmark = pytest.mark.gpu


# P' = 62, 65, 128, 131, 194, 257 (a strip and a column), 320, 323, 482, 512 + 2, 1154
@pytest.mark.parametrize("hidden", [[20], [21], [42], [43], [64], [85], [106], [107], [20, 20], [170, 1], [32, 32]])
@pytest.mark.parametrize("slices", [6, 4])
def test_split_damped_solve(hidden, slices):
    p = gpu_problem(I.small_case(I.BURGERS, [1] + hidden + [1], 8), precision=2, n_slices=slices)
    n = p.P + 1
    rng = np.random.default_rng(n)
    J = torch.from_numpy(rng.standard_normal((300, n)) * 10.0 ** (-2 * rng.random(n))).cuda()
    G, g = J.T @ J / 300, torch.from_numpy(rng.standard_normal(n)).cuda()
    x = p.new_vec(n)
    rc, gam, retries = p.gn_damped_solve(G, g, 1e-1, x)
    assert rc == 0 and retries == 0 and gam == 1e-1
    A = G + gam * torch.eye(n, dtype=torch.float64, device="cuda")
    back = (A @ x - g).abs().max() / (A.abs().sum(1).max() * x.abs().max())
    # double-float blocks (2^-47 a product) and the slices' truncation, 2^(1 - 8 S), over n terms
    assert float(back) <= n * (2.0 ** -47 + 2.0 ** (1 - 8 * slices))
    y = x.clone()
    p.gn_damped_solve(G, g, 1e-1, x)
    assert torch.equal(x, y)
    # an indefinite matrix is refused after its escalations, whichever block fails
    H = G.clone()
    H[n // 2, n // 2] = -1e9
    assert p.gn_damped_solve(H, g, 1e-6, x)[0] == -5
