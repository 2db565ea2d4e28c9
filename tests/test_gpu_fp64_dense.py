"""The FP64 Gram and damped solve at the edges of their tile rules, against torch in FP64.

The Gram's tiles are 64, 32 or 16 wide by the number of tiles, with the contraction split over
the groups of a block when it is long; the solve's panels take 8 or 32 rows per CTA and its
trailing updates run beside the next diagonal block."""
import numpy as np
import pytest
import torch

from paper_2509_14185_gb300 import inputs as I
from tests.gpu_cases import gpu_problem

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _problem(hidden):
    return gpu_problem(I.small_case(I.BURGERS, [1] + hidden + [1], 8))


# P' = 65, 98, 482, 1154 (703 tiles of 32), 4050 (2080 tiles of 64)
@pytest.mark.parametrize("hidden", [[21], [8, 8], [20, 20], [32, 32], [44, 44, 44]])
@pytest.mark.parametrize("rows", [1, 63, 255, 256, 300])
def test_fp64_gram(hidden, rows):
    p = _problem(hidden)
    n = p.P + 1
    J = torch.from_numpy(np.random.default_rng(rows).standard_normal((rows, n + 3))).cuda()
    G = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    p.gn_gram(J, rows, None, G, None, precision=0)
    p.gn_gram(J, rows, None, G, None, precision=0, accumulate=True)
    A = J[:, :n]
    # two sums of `rows` products in any order, one addition, and torch's own product
    bound = (4 * rows + 2) * U * (A.abs().T @ A.abs())
    assert bool((torch.tril(G - 2 * (A.T @ A)).abs() <= bound).all())


@pytest.mark.parametrize("hidden", [[20], [21], [8, 8], [32, 32], [44, 44, 44]])   # P' = 62, 65, 98, 1154, 4050
def test_fp64_damped_solve(hidden):
    p = _problem(hidden)
    n = p.P + 1
    rng = np.random.default_rng(n)
    J = torch.from_numpy(rng.standard_normal((200, n))).cuda()
    G, g = J.T @ J / 200, torch.from_numpy(rng.standard_normal(n)).cuda()
    x = p.new_vec(n)
    rc, gam, retries = p.gn_damped_solve(G, g, 1e-1, x)
    assert rc == 0 and retries == 0 and gam == 1e-1
    A = G + gam * torch.eye(n, dtype=torch.float64, device="cuda")
    # Cholesky and two triangular solves: 3 n u |A| |x| to first order, twice that for the inverted blocks
    back = (A @ x - g).abs().max() / (A.abs().sum(1).max() * x.abs().max())
    assert float(back) <= 6 * n * U
