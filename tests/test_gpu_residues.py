"""The six-slice Gram by residues: exact on integers, and only the 48-bit operands' rounding otherwise."""
import numpy as np
import pytest
import torch

from paper_2509_14185_gb300 import inputs as I
from tests.gpu_cases import gpu_problem

pytestmark = pytest.mark.gpu


def _problem(hidden):
    p = gpu_problem(I.small_case(I.BURGERS, [1] + hidden + [1], 8), precision=1, n_slices=6)
    return p, p.P + 1


def _gram(p, J, rows, accumulate=False, G=None):
    n = p.P + 1
    G = torch.full((n, n), 3.0, dtype=torch.float64, device="cuda") if G is None else G
    p.gn_gram(J, rows, None, G, None, precision=1, accumulate=accumulate)
    return G


# P' = 65 and 254: one tile; 257 and 482: three; 1154: 15; 9044: 666 tiles (two batches).
# Contractions inside one chunk of 384 rows, at its edges, and over several.
@pytest.mark.parametrize("hidden,rows", [
    ([21], 17), ([21], 63), ([21], 384), ([84], 385), ([85], 383), ([85], 800), ([20, 20], 1000), ([32, 32], 3001),
    ([66, 66, 66], 2261)])
def test_bit_exact_on_integers(hidden, rows):
    p, n = _problem(hidden)
    g = torch.Generator(device="cuda").manual_seed(rows)
    J = torch.randint(-2 ** 20, 2 ** 20 + 1, (rows, n + 3), generator=g, device="cuda").double()
    J[:, 3] = 0.0
    J[:, 7] *= 2.0 ** -30
    J[0, 5] = 2.0 ** 20
    A = J[:, :n]
    ref = A.T @ A                                  # exact: every partial sum is below 2^53 units
    G = _gram(p, J, rows)
    assert torch.equal(torch.tril(G), torch.tril(ref))
    assert bool((torch.triu(G, 1) == torch.triu(torch.full_like(G, 3.0), 1)).all())   # left untouched
    G = _gram(p, J, rows, accumulate=True, G=G)
    assert torch.equal(torch.tril(G), torch.tril(2.0 * ref))


def test_largest_digits_do_not_overflow():
    """Columns of one repeated value: every residue product has the same sign."""
    p, n = _problem([30])
    v = torch.from_numpy(np.random.default_rng(0).integers(1, 2 ** 22, n) * 2.0 - 2 ** 22).cuda()
    rows = 2000
    J = v.repeat(rows, 1).contiguous()
    assert torch.equal(torch.tril(_gram(p, J, rows)), torch.tril(rows * torch.outer(v, v)))


@pytest.mark.parametrize("hidden,rows", [([20, 20], 2114), ([32, 32], 777)])
def test_error_is_the_operands_rounding(hidden, rows):
    p, n = _problem(hidden)
    rng = np.random.default_rng(rows)
    J = rng.standard_normal((rows, n)) * 2.0 ** rng.integers(-40, 40, n) * 10.0 ** (-6 * rng.random((rows, n)))
    Jt = torch.from_numpy(J).cuda()
    G = _gram(p, Jt, rows)
    a = Jt.abs()
    d = torch.ldexp(torch.ones(n, dtype=torch.float64, device="cuda"), torch.frexp(a.amax(0))[1] - 49)
    s = a.sum(0)
    # both operands' roundings, their product, and the rounding of G and of torch's FP64 reference
    bound = torch.outer(d, s) + torch.outer(s, d) + rows * torch.outer(d, d) + (rows + 2) * 2.0 ** -53 * (a.T @ a)
    assert bool((torch.tril(G - Jt.T @ Jt).abs() <= torch.tril(bound) + 1e-300).all())


def test_more_rows_than_one_product_takes():
    """32768 rows go into one product at most; further products are added to the first."""
    p, n = _problem([21])
    rows = 2 ** 16 + 56
    J = torch.randint(-2 ** 15, 2 ** 15, (rows, n), generator=torch.Generator(device="cuda").manual_seed(1),
                      device="cuda").double()
    assert torch.equal(torch.tril(_gram(p, J, rows)), torch.tril(J.T @ J))


def test_forced_tiles_keep_the_slice_products():
    p, n = _problem([20, 20])
    J = torch.from_numpy(np.random.default_rng(4).standard_normal((500, n))).cuda()
    ref = torch.tril(J.T @ J)
    G6 = torch.tril(_gram(p, J, 500))
    p.gn_set_gram_tile(64)
    G64 = torch.tril(_gram(p, J, 500))
    assert p.gn_gram_tile_choice(500) == 64
    assert float((G6 - ref).norm()) <= float((G64 - ref).norm())


def test_residues_leave_the_table_of_tuned_slices_alone():
    """544 rows of 2114 columns go by residues, 520 (as many chunks of the contraction) by slices: what
    one reports or records does not reach the other."""
    p, n = _problem([44, 44])
    assert n == 2114
    p.gn_set_precision(1, 6)
    J = torch.randn(544, n, generator=torch.Generator(device="cuda").manual_seed(2), dtype=torch.float64, device="cuda")
    assert (p.gn_gram_split_choice(544), p.gn_gram_tile_choice(544)) == (1, 128)
    _gram(p, J, 544)
    assert (p.gn_gram_split_choice(520), p.gn_gram_tile_choice(520)) == (0, 0)      # not tuned yet
    _gram(p, J[:520], 520)
    assert p.gn_gram_split_choice(520) >= 1 and p.gn_gram_tile_choice(520) in (64, 128)
    assert (p.gn_gram_split_choice(544), p.gn_gram_tile_choice(544)) == (1, 128)
