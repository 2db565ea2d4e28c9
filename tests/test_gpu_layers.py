"""The layered passes (many points, hidden layers as split products on the tensor cores) against the
one-warp-per-point kernel, which takes the same points when there are few of them.

A row depends on its own point (and, for CCF, on the Hilbert nodes, the same in both problems), so
the rows of a large problem at some of its points equal those of a problem of these points alone,
up to the factor sqrt(N_small / N_large) of the row weights."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2509_14185_gb300 import inputs as I
from tests.gpu_cases import TOL, col_rel, dev, gpu_problem, host, rel

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

EQS = {"burgers": (I.BURGERS, 1), "ccf": (I.CCF, 1), "ipm": (I.IPM, 2), "boussinesq": (I.BOUSSINESQ, 3)}


def _pair(name, hidden, n, n_bnd=40, seed=3, **kw):
    eq, nf = EQS[name]
    big = I.weighted(I.small_case(eq, [I.EQUATION_DIM[eq]] + hidden + [nf], n, n_bnd=n_bnd if nf > 1 else 0, seed=seed))
    pick = np.unique(np.concatenate([[0, 1, n // 2, n - 2, n - 1], np.arange(0, n, 37)]))
    few = dataclasses.replace(big, y=np.ascontiguousarray(big.y[:, pick]), rho=big.rho[pick])
    return big, few, pick, gpu_problem(big, **kw), gpu_problem(few, **kw)


def _rows(pick, ne):
    return (pick[:, None] * ne + np.arange(ne)).reshape(-1)


# tiles of 128 rows hold 64, 42, 21 or 14 items; widths with one or two 32-wide stages, ragged ones
@pytest.mark.parametrize("name,hidden,n", [
    ("burgers", [24, 24], 4096), ("burgers", [32, 64, 33], 4111), ("ccf", [64, 64, 64], 4097), ("ccf", [31, 25], 4099),
    ("ipm", [64, 64, 64, 64], 2049), ("ipm", [40, 27, 64], 2200), ("boussinesq", [48, 48, 48], 2048),
    ("boussinesq", [33, 64], 2061), ("boussinesq", [64, 56, 60], 2053), ("ipm", [44, 64], 2051),
    ("ipm", [45, 44, 63], 2048)])
def test_rows_and_jacobian_equal_the_pointwise_kernel(name, hidden, n):
    big, few, pick, pb, pf = _pair(name, hidden, n)
    ne = EQS[name][1]
    sel = torch.from_numpy(_rows(pick, ne)).cuda()
    scale = np.sqrt(len(pick) / n)
    th = dev(big.theta)
    m = len(pick) * ne
    r_b, r_f = pb.residual(th, big.lam)[0], pf.residual(th, big.lam)[0]
    assert rel(host(r_b[sel]), scale * host(r_f[:m])) <= TOL
    J_b = pb.jacobian(th, big.lam)
    J_f = scale * host(pf.jacobian(th, big.lam)[:m])
    J_s = host(J_b[sel])
    assert rel(J_s, J_f) <= TOL
    assert col_rel(J_s, J_f, floor=1e-300) <= TOL
    # a block that starts and ends inside a point equals the same rows of the whole
    lo, cnt = n // 3 * ne + 1, n // 2 * ne
    assert torch.equal(pb.jacobian(th, big.lam, row0=lo, nrows=cnt, ld=pb.P + 9), J_b[lo:lo + cnt])


@pytest.mark.parametrize("name,hidden,n,n_bnd", [
    ("burgers", [24, 24], 4096, 0), ("ccf", [64, 33, 64], 4100, 0), ("ipm", [64, 27, 64, 40], 2049, 2055),
    ("boussinesq", [48, 48, 48], 2100, 40)])
@pytest.mark.parametrize("frozen", [False, True])
def test_gradient_equals_the_rows(name, hidden, n, n_bnd, frozen):
    """J^T seed by the adjoint against the same product with the Jacobian's rows: both are FP64 sums of
    n_rows products, each off by at most n_rows u times the sum of the magnitudes."""
    big, _, _, pb, _ = _pair(name, hidden, n, n_bnd)
    pb.gn_set_lambda_trainable(not frozen)
    th = dev(big.theta)
    J = pb.jacobian(th, big.lam)
    seed = dev(np.random.default_rng(2).standard_normal(pb.n_rows))
    bound = 2.0 ** -53 * 2 * pb.n_rows * (J.abs().T @ seed.abs()) + TOL * (J.abs().T @ seed.abs())
    assert bool(((pb.gradient(th, big.lam, seed) - J.T @ seed).abs() <= bound).all())
    r = pb.residual(th, big.lam)[0]
    g = pb.gradient(th, big.lam)
    bound = 2.0 ** -53 * 2 * pb.n_rows * (J.abs().T @ r.abs()) + TOL * (J.abs().T @ r.abs())
    assert bool(((g - J.T @ r).abs() <= bound).all())
    assert torch.equal(g, pb.gradient(th, big.lam))      # a fixed order of additions


def test_many_wall_points_equal_few():
    """2050 wall points take the layered path, 900 of them the pointwise one."""
    big, _, _, pb, _ = _pair("ipm", [32, 32, 32], 300, n_bnd=2050)
    pf = gpu_problem(dataclasses.replace(big, y_bnd=np.ascontiguousarray(big.y_bnd[:, :900])))
    th = dev(big.theta)
    s = np.sqrt(900 / 2050)
    r_b, r_f = pb.residual(th, big.lam)[0], pf.residual(th, big.lam)[0]
    assert torch.equal(r_b[:600], r_f[:600]) and torch.equal(r_b[-1:], r_f[-1:])
    assert rel(host(r_b[600:1500]), s * host(r_f[600:1500])) <= TOL
    J_b, J_f = host(pb.jacobian(th, big.lam, 600, 900)), s * host(pf.jacobian(th, big.lam, 600, 900))
    assert rel(J_b, J_f) <= TOL


@pytest.mark.parametrize("name,hidden", [("burgers", [24, 24]), ("ipm", [30, 30, 30])])
def test_second_stage(name, hidden):
    n = 4100 if name == "burgers" else 2300
    big, few, pick, pb, pf = _pair(name, hidden, n)
    ne = EQS[name][1]
    w1 = [I.EQUATION_DIM[big.equation], 9, EQS[name][1]]
    for p in (pb, pf):
        p.gn_set_stage1(w1, dev(I.xavier_init(w1, 5)), big.lam, 1e-3)
    th = dev(big.theta)
    sel = torch.from_numpy(_rows(pick, ne)).cuda()
    J_s, J_f = host(pb.jacobian(th, big.lam)[sel]), host(pf.jacobian(th, big.lam)[:len(pick) * ne])
    assert rel(J_s, np.sqrt(len(pick) / n) * J_f) <= TOL


@pytest.mark.parametrize("name", ["burgers", "boussinesq"])
def test_extreme_and_non_finite_values(name):
    """Saturated and tiny weights reach the digits' limits; a NaN weight or point reaches its rows."""
    big, few, pick, pb, pf = _pair(name, [40, 40, 40], 4200)
    ne = EQS[name][1]
    sel = torch.from_numpy(_rows(pick, ne)).cuda()
    theta = big.theta.copy()
    theta[::7] *= 40.0
    theta[3::11] *= 1e-200
    th = dev(theta)
    m = len(pick) * ne
    r_s, r_f = host(pb.residual(th, big.lam)[0][sel]), host(pf.residual(th, big.lam)[0][:m])
    assert np.all(np.isfinite(r_f))
    assert rel(r_s, np.sqrt(len(pick) / 4200) * r_f) <= TOL
    theta[300] = np.nan
    assert pb.gn_residual(dev(theta), big.lam)[0] == -4
    y = big.y.copy()
    y[0, 1234] = np.nan
    pn = gpu_problem(dataclasses.replace(big, y=y))
    r = pn.new_vec(pn.n_rows)
    assert pn.gn_residual(dev(big.theta), big.lam, r)[0] == -4
    bad = np.flatnonzero(~np.isfinite(host(r)))
    assert bad.size and set(bad) <= set(range(1234 * ne, 1234 * ne + ne))


def test_jacobian_of_extreme_weights():
    """Hidden weights' entries as products (2D, wide layers): components of very different sizes."""
    big, few, pick, pb, pf = _pair("ipm", [48, 64, 48], 2100)
    sel = torch.from_numpy(_rows(pick, 2)).cuda()
    theta = big.theta.copy()
    theta[::7] *= 40.0
    theta[3::11] *= 1e-200
    J_b, J_f = pb.jacobian(dev(theta), big.lam), pf.jacobian(dev(theta), big.lam)
    assert rel(host(J_b[sel]), np.sqrt(len(pick) / 2100) * host(J_f[:2 * len(pick)])) <= TOL


def test_step_graph_equals_step():
    big, _, _, pb, _ = _pair("ccf", [32, 32], 4300, precision=2, n_slices=6)
    pg = gpu_problem(big, precision=2, n_slices=6)
    ta, tb = dev(big.theta), dev(big.theta)
    a, b = pb.gn_step(ta, big.lam, 1e-2), pg.gn_step_graph(tb, big.lam, 1e-2)
    assert a[:3] == b[:3] and torch.equal(ta, tb)


@pytest.mark.parametrize("name,hidden,n", [("burgers", [24, 24, 24], 300007), ("ipm", [32, 24, 30], 40001)])
def test_tiles_keep_their_own_exponents(name, hidden, n):
    """Many tiles per SM, outputs so narrow that half of the warps have no columns to combine, and
    neighbouring tiles whose rows differ by orders of magnitude: a row scaled by another tile's
    exponent would be off by a power of two."""
    big, few, pick, _, _ = _pair(name, hidden, n)
    # the near half of the points and the far half in turn, in stretches of one tile's points
    order = np.argsort(np.abs(big.y).sum(0))
    stretch = np.arange(n) // (64 if name == "burgers" else 21)
    big.y[:] = big.y[:, order[np.argsort(stretch % 2, kind="stable").argsort()]]
    few = dataclasses.replace(big, y=np.ascontiguousarray(big.y[:, pick]), rho=big.rho[pick])
    pb, pf = gpu_problem(big), gpu_problem(few)
    ne = EQS[name][1]
    sel = torch.from_numpy(_rows(pick, ne)).cuda()
    th = dev(big.theta)
    m = len(pick) * ne
    scale = np.sqrt(len(pick) / n)
    ref = scale * host(pf.residual(th, big.lam)[0][:m])
    first = pb.residual(th, big.lam)[0].clone()
    assert rel(host(first[sel]), ref) <= TOL
    for _ in range(5):
        assert torch.equal(pb.residual(th, big.lam)[0], first)


def _neuron(theta, widths, layer, k, s):
    """Incoming weights of a hidden neuron divided by s, outgoing ones multiplied."""
    off = 0
    for l, (i, o) in enumerate(zip(widths[:-1], widths[1:])):
        W = theta[off:off + i * o].reshape(o, i)
        if l == layer - 1:
            W[k] /= s
        elif l == layer:
            W[:, k] *= s
        off += i * o + o


def _wild(theta, widths, rng):
    """Hidden-to-hidden weights spread over five decades, which no scaling of neurons evens out."""
    off = 0
    for l, (i, o) in enumerate(zip(widths[:-1], widths[1:])):
        if 0 < l < len(widths) - 2:
            theta[off:off + i * o] *= 10.0 ** rng.uniform(-4.5, 0.5, i * o)
        off += i * o + o


@pytest.mark.parametrize("name,hidden", [("ipm", [64, 64, 64, 64]), ("burgers", [40, 40, 40]), ("boussinesq", [56, 60, 64])])
@pytest.mark.parametrize("scales", [1e2, 1e4, 1e6, 1e-5, "wild"])
def test_weights_of_different_scale(name, hidden, scales):
    """Rows and Jacobian columns as accurate as FP64 sums when a network's weights differ in scale.  An
    FP64 sum of n <= 64 products is the exact sum of operands off by at most n 2^-53 each, so what
    such changes of theta move bounds what two FP64 evaluations may differ by (times 4, for
    the layers' changes that do not point the same way)."""
    n = 4200
    big, few, pick, pb, pf = _pair(name, hidden, n)
    ne = EQS[name][1]
    rng = np.random.default_rng(8)
    theta = big.theta.copy()
    if scales == "wild":
        _wild(theta, big.widths, rng)
    else:
        for layer in range(1, len(hidden)):
            _neuron(theta, big.widths, layer, 5 + layer, scales)
    m = len(pick) * ne
    sel = torch.from_numpy(_rows(pick, ne)).cuda()
    s = np.sqrt(len(pick) / n)

    def few_at(th):
        return s * host(pf.residual(dev(th), big.lam)[0][:m]), s * host(pf.jacobian(dev(th), big.lam)[:m])

    r0, J0 = few_at(theta)
    tr, tJ = 0.0, np.zeros(J0.shape[1])
    for _ in range(4):
        r, J = few_at(theta * (1.0 + 64 * 2.0 ** -53 * rng.uniform(-1, 1, theta.size)))
        tr = max(tr, np.max(np.abs(r - r0)))
        tJ = np.maximum(tJ, np.max(np.abs(J - J0), axis=0))
    th = dev(theta)
    assert np.max(np.abs(host(pb.residual(th, big.lam)[0][sel]) - r0)) <= 4 * tr
    dJ = np.max(np.abs(host(pb.jacobian(th, big.lam)[sel]) - J0), axis=0)
    assert np.all(dJ <= 4 * tJ + 2.0 ** -48 * np.max(np.abs(J0), axis=0))


@pytest.mark.parametrize("name,hidden", [("ipm", [48, 64, 48, 45]), ("boussinesq", [56, 64, 60])])
def test_entries_of_a_constant_neuron(name, hidden):
    """A hidden neuron without incoming weights is h = tanh(b): its outgoing weight's entry is h times the
    entry of the bias behind it, in every row, however small beside the row's other entries.
    Of the FP64 sum's six terms one is not 0: off by 6 u at most, tanh by 2 ulp (4 u) on
    either side, the product here by u."""
    eq, nf = EQS[name]
    n = 8000
    w = I.weighted(I.small_case(eq, [2] + hidden + [nf], n, n_bnd=0, seed=5))
    theta, offs, off = w.theta.copy(), [], 0
    for i, o in zip(w.widths[:-1], w.widths[1:]):
        offs.append((off, i, o))
        off += i * o + o
    b = 0.7
    for off, i, o in offs[:-2]:
        theta[off + 3 * i:off + 4 * i] = 0.0
        theta[off + i * o + 3] = b
    pb = gpu_problem(w)
    J = pb.jacobian(dev(theta), w.lam)[:n * EQS[name][1]]
    for off, i, o in offs[1:-1]:
        entry, bias = J[:, off + 3:off + i * o:i], J[:, off + i * o:off + i * o + o]
        ref = bias * np.tanh(b)
        assert bool((ref != 0).any())
        assert bool(((entry - ref).abs() <= 15 * 2.0 ** -53 * ref.abs()).all())


@pytest.mark.parametrize("name,hidden,n,call,layered", [
    ("burgers", [24] * 4, 4999, "residual", False), ("burgers", [24] * 4, 5000, "residual", True),
    ("burgers", [32, 40], 4095, "residual", False), ("burgers", [32, 40], 4096, "residual", True),
    ("burgers", [64, 31], 9000, "jacobian", False), ("burgers", [39, 64], 4999, "jacobian", False),
    ("burgers", [32, 64], 5000, "jacobian", True), ("burgers", [40, 64], 4096, "jacobian", True),
    ("burgers", [27, 64], 9000, "gradient", False), ("burgers", [28, 64], 4096, "gradient", True),
    ("ipm", [24, 24], 2047, "residual", False), ("ipm", [24, 24], 2048, "residual", True),
    ("ipm", [64, 31], 3000, "jacobian", False), ("ipm", [64, 32], 2048, "jacobian", True),
    ("ipm", [64, 24], 2048, "gradient", True), ("ipm", [64, 23], 3000, "gradient", False)])
def test_route_by_width_and_points(name, hidden, n, call, layered):
    """Narrow networks and few points stay with the one-warp-per-point kernel where it is the faster one:
    the weights' transposition, the interior and the normalisation point (and a gradient's sum)."""
    from paper_2509_14185_gb300 import gn
    eq, nf = EQS[name]
    w = I.small_case(eq, [I.EQUATION_DIM[eq]] + hidden + [nf], n, n_bnd=0)
    p = gpu_problem(w)
    th = dev(w.theta)
    out = {"residual": lambda: p.gn_residual(th, w.lam, r, want_loss=False), "jacobian": lambda: p.jacobian(th, w.lam),
           "gradient": lambda: p.gradient(th, w.lam)}
    r = p.new_vec(p.n_rows)
    k = gn.lib().gn_kernel_launches()
    out[call]()
    k = gn.lib().gn_kernel_launches() - k
    torch.cuda.synchronize()
    assert (k > 5) == layered, k
