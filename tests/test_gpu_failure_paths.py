"""Failure paths of the C ABI, exercised without any GPU fault.

GN_ERR_NONFINITE: a NaN in theta or in a collocation point (host data) reaches the jet
kernel, which flags the non-finite residual row; gn_residual, gn_step and gn_step_graph
must return the code with theta and lambda untouched and without damping escalations.

GN_ERR_TIMEOUT: every mbarrier wait of the split-precision tensor-core kernels is bounded.
gn_test_bounded_waits shortens the bound to 20 ms and makes the kernels' producer issue no
copies, so no copy or MMA is ever in flight and the consumers' waits simply run out; the
kernel releases its tensor memory and returns, gn_gram / gn_damped_solve / gn_step return
GN_ERR_TIMEOUT, and after the hook is reset the same calls succeed on the same context with
the results of an undisturbed run.
"""
import ctypes

import numpy as np
import pytest
import torch

from tests.gpu_cases import dev, gpu_problem, host, small

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

GN_ERR_NONFINITE, GN_ERR_TIMEOUT = -4, -6


@pytest.mark.parametrize("name", ["ccf", "ipm"])
def test_nan_theta_returns_nonfinite(name):
    w = small(name)
    prob = gpu_problem(w, precision=2, n_slices=6)
    bad = w.theta.copy()
    bad[3] = np.nan
    rc, loss = prob.gn_residual(dev(bad), w.lam)
    assert rc == GN_ERR_NONFINITE and not np.isfinite(loss)
    for step in (prob.gn_step, prob.gn_step_graph):
        theta = dev(bad)
        before = host(theta).copy()
        rc, lam, gam, info = step(theta, w.lam, w.gamma)
        assert rc == GN_ERR_NONFINITE, (step.__name__, rc)
        assert info["chol_retries"] == 0
        np.testing.assert_array_equal(host(theta), before)
        assert lam == w.lam and gam == w.gamma
    # the handle stays usable: a finite theta steps normally afterwards
    theta = dev(w.theta)
    rc, lam, gam, info = prob.gn_step(theta, w.lam, w.gamma)
    assert rc in (0, 1) and np.isfinite(info["loss_before"])
    prob.close()


def test_nan_collocation_point_returns_nonfinite():
    w = small("burgers")
    y = w.y.copy()
    y[0, 7] = np.nan
    w.y = y
    prob = gpu_problem(w)
    rc, loss = prob.gn_residual(dev(w.theta), w.lam)
    assert rc == GN_ERR_NONFINITE
    theta = dev(w.theta)
    rc, lam, gam, info = prob.gn_step(theta, w.lam, w.gamma)
    assert rc == GN_ERR_NONFINITE
    np.testing.assert_array_equal(host(theta), w.theta)
    prob.close()


def test_bounded_waits_time_out_and_the_context_recovers():
    from paper_2509_14185_gb300 import gn
    L = gn.lib()
    w = small("ccf")
    prob = gpu_problem(w, precision=2, n_slices=6)
    Pp = prob.P + 1
    J = prob.jacobian(dev(w.theta), w.lam)
    r = torch.zeros(J.shape[0], dtype=torch.float64, device="cuda")
    G_ref = torch.zeros((Pp, Pp), dtype=torch.float64, device="cuda")
    g_ref = prob.new_vec(Pp)
    prob.gn_gram(J, J.shape[0], r, G_ref, g_ref, precision=1)   # also settles the split-K choice
    torch.cuda.synchronize()
    G = torch.full((Pp, Pp), 7.0, dtype=torch.float64, device="cuda")
    g = prob.new_vec(Pp)
    try:
        assert L.gn_test_bounded_waits(20_000_000, 1) == 0
        rc = L.gn_gram(prob.h, gn._ptr(J), J.stride(0), J.shape[0], gn._ptr(r), gn._ptr(G), gn._ptr(g), 1, 0)
        assert rc == GN_ERR_TIMEOUT
        delta = prob.new_vec(Pp)
        rc, gam, ret = prob.gn_damped_solve(G_ref, g_ref, 1e-6, delta)   # split factorisation's updates
        assert rc == GN_ERR_TIMEOUT
        theta = dev(w.theta)
        rc = L.gn_step(prob.h, gn._ptr(theta), ctypes.byref(ctypes.c_double(w.lam)),
                       ctypes.byref(ctypes.c_double(w.gamma)), None)
        assert rc == GN_ERR_TIMEOUT
        np.testing.assert_array_equal(host(theta), w.theta)
    finally:
        assert L.gn_test_bounded_waits(0, 0) == 0
    # same context, default bound, copies issued again: the Gram equals the undisturbed one
    torch.cuda.synchronize()
    prob.gn_gram(J, J.shape[0], r, G, g, precision=1)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(np.tril(host(G)), np.tril(host(G_ref)))
    prob.close()


def test_layered_passes_time_out_and_recover():
    """The passes over many points wait for tensor-core products in every precision.  With none issued:
    calls that synchronise return GN_ERR_TIMEOUT and leave theta alone; gn_jacobian and gn_gradient only launch,
    leave no entry unwritten, and the next call that synchronises reports them, once."""
    from paper_2509_14185_gb300 import gn
    from paper_2509_14185_gb300 import inputs as I
    L = gn.lib()
    n = 2100
    w = I.small_case(I.IPM, [2, 48, 48, 48, 2], n, n_bnd=30, seed=3)
    prob, ref = gpu_problem(w), gpu_problem(w)
    Pp, th = prob.P + 1, dev(w.theta)
    J0, g0 = ref.jacobian(th, w.lam), ref.gradient(th, w.lam)
    loss0 = ref.gn_residual(th, w.lam)[1]
    J = torch.full_like(J0, 7.0)
    g = prob.new_vec(Pp)
    A = torch.eye(Pp, dtype=torch.float64, device="cuda")
    delta, out = prob.new_vec(Pp), ctypes.c_double(0.0)

    def step(p, theta, call=L.gn_step):
        lam, gam = ctypes.c_double(w.lam), ctypes.c_double(1e-2)
        return call(p.h, gn._ptr(theta), ctypes.byref(lam), ctypes.byref(gam), None), lam.value, gam.value

    torch.cuda.synchronize()
    try:
        assert L.gn_test_bounded_waits(20_000_000, 1) == 0
        assert L.gn_residual(prob.h, gn._ptr(th), w.lam, None, ctypes.byref(out)) == GN_ERR_TIMEOUT
        assert L.gn_max_residual(prob.h, gn._ptr(th), w.lam, ctypes.byref(out)) == GN_ERR_TIMEOUT
        assert L.gn_jacobian(prob.h, gn._ptr(th), w.lam, gn._ptr(J), J.stride(0), 0, J.shape[0]) == 0
        assert L.gn_gradient(prob.h, gn._ptr(th), w.lam, None, gn._ptr(g)) == 0
    finally:
        assert L.gn_test_bounded_waits(0, 0) == 0
    torch.cuda.synchronize()
    off = 2 * 48 + 48
    for i, o in ((48, 48), (48, 48)):
        assert bool(torch.isnan(J[:2 * n, off:off + i * o]).all())
        off += i * o + o
    assert bool(torch.isnan(g).any())
    assert prob.gn_damped_solve(A, g0, 1.0, delta)[0] == GN_ERR_TIMEOUT     # reported
    assert prob.gn_damped_solve(A, g0, 1.0, delta)[0] == 0                  # and cleared
    theta, theta_ref = dev(w.theta), dev(w.theta)
    pg = gpu_problem(w)
    try:
        assert L.gn_test_bounded_waits(20_000_000, 1) == 0
        assert step(prob, theta)[0] == GN_ERR_TIMEOUT
        assert step(pg, theta, L.gn_step_graph) == (GN_ERR_TIMEOUT, w.lam, 1e-2)
    finally:
        assert L.gn_test_bounded_waits(0, 0) == 0
    np.testing.assert_array_equal(host(theta), w.theta)
    # undisturbed again
    assert prob.gn_residual(th, w.lam) == (0, loss0)
    assert torch.equal(prob.jacobian(th, w.lam), J0) and torch.equal(prob.gradient(th, w.lam), g0)
    assert step(prob, theta) == step(ref, theta_ref) and torch.equal(theta, theta_ref)
    for p in (prob, ref, pg):
        p.close()
