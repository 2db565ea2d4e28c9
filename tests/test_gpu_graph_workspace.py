"""Captured steps against calls in between that move a workspace whose address the graph holds: the
next captured step must be recorded again, and equal the step taken launch by launch."""
import numpy as np
import pytest
import torch

from paper_2509_14185_gb300 import gn
from paper_2509_14185_gb300 import inputs as I
from tests.gpu_cases import dev, gpu_problem, host, small

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


def _gram(handle, Pp, rows, precision=1):
    """A split Gram of `rows` rows on the handle; what its old workspace was is overwritten."""
    J = torch.randn(rows, Pp, dtype=torch.float64, device="cuda")
    G = torch.empty(Pp, Pp, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    rc = gn.lib().gn_gram(handle, gn._ptr(J), Pp, rows, None, gn._ptr(G), None, precision, 0)
    assert rc == 0
    torch.cuda.empty_cache()
    torch.full((1 << 27,), float("nan"), dtype=torch.float64, device="cuda")   # 1 GB


@pytest.mark.parametrize("name,between", [
    ("burgers", "more rows"), ("ccf", "more rows"), ("ccf", "tile"), ("ipm", "split"), ("ccf", "solve")])
def test_step_graph_after_a_moved_workspace(name, between):
    w = small(name)
    pe, pg = gpu_problem(w, precision=2, n_slices=6), gpu_problem(w, precision=2, n_slices=6)
    Pp = pg.P + 1
    if between in ("tile", "split"):
        for p in (pe, pg):
            p.gn_set_gram_tile(64)
    te, tg = dev(w.theta), dev(w.theta)
    a, b = pe.gn_step(te, w.lam, 1e-2), pg.gn_step_graph(tg, w.lam, 1e-2)
    assert a[:3] == b[:3] and torch.equal(te, tg)
    if between == "more rows":
        _gram(pg.h, Pp, 20 * w.n_pts)
    elif between == "solve":
        pg.gn_set_precision(1, 6)
        _gram(pg.h, Pp, 6000)
        pg.gn_set_precision(2, 6)
    else:
        for p in (pe, pg):
            p.gn_set_gram_tile(0)
            if between == "split":
                p.gn_set_gram_split(2)
        _gram(pg.h, Pp, pg.n_rows)
    for _ in range(2):
        a, b = pe.gn_step(te, a[1], a[2]), pg.gn_step_graph(tg, b[1], b[2])
        assert a[:3] == b[:3] and a[3]["loss_after"] == b[3]["loss_after"] and torch.equal(te, tg)
    pe.close()
    pg.close()


def test_batch_graph_after_a_moved_workspace():
    ws = [small("burgers"), small("ccf"), small("ipm")]
    be, bg = gn.GNBatch(ws, n_streams=2, precision=2), gn.GNBatch(ws, n_streams=2, precision=2)
    te, tg = [dev(w.theta) for w in ws], [dev(w.theta) for w in ws]
    lam, gam = [w.lam for w in ws], [1e-2] * len(ws)
    bg.gn_batch_capture_graph(tg)
    bg.gn_set_lambda_trainable(False)        # the graph keeps the setting that it was captured with
    le, ge = list(lam), list(gam)
    lg, gg = list(lam), list(gam)
    for k in range(3):
        if k:
            _gram(bg.handle(k), bg.P[k] + 1, 4000 * k)
        le, ge, _, se = be.gn_batch_step(te, le, ge)
        lg, gg, _, sg = bg.gn_batch_graph_step(lg, gg)
        assert (le, ge, se) == (lg, gg, sg)
        assert all(torch.equal(x, y) for x, y in zip(te, tg))
    assert all(np.all(np.isfinite(host(t))) for t in tg)


@pytest.mark.parametrize("precision", [1, 2])
def test_streamed_step_with_a_remainder(precision):
    """Row blocks of more rows than one product of residues takes, the last block shorter: the captured
    step equals the eager one, the Gram stays on the residues, and no row count up to the
    block's needs more memory than the step."""
    w = I.small_case(I.BURGERS, [1, 20, 20, 1], 63000)
    pe = gpu_problem(w, precision=precision, n_slices=6, row_block=33000)
    pg = gpu_problem(w, precision=precision, n_slices=6, row_block=33000)
    te, tg = dev(w.theta), dev(w.theta)
    a, b = pe.gn_step(te, w.lam, 1e-2), pg.gn_step_graph(tg, w.lam, 1e-2)
    assert a[:3] == b[:3] and torch.equal(te, tg)
    n = pg.P + 1
    J = torch.randn(33000, n, dtype=torch.float64, device="cuda")
    ref = torch.tril(J[:31000].T @ J[:31000])
    G = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for rows in (32768, 30001, 16512, 1000, 33000, 31000):
        pg.gn_gram(J, rows, None, G, None, precision=1)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    # slices would be off by their FP32 sums, near 1e-10
    assert float((torch.tril(G) - ref).abs().max() / ref.abs().max()) <= 1e-13
    a, b = pe.gn_step(te, a[1], a[2]), pg.gn_step_graph(tg, b[1], b[2])
    assert a[:3] == b[:3] and torch.equal(te, tg)
    pe.close()
    pg.close()
