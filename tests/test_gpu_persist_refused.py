"""Where the cooperative launch of the persistent PCG is refused (a context that may use only part of the
SMs), solves go on with another form instead of failing. The refusal is the launch's error code, faked on
the host (MHD_FAULT_COOP_LAUNCH): from the first solve on, when the form is chosen, and after a form was
chosen that then cannot be launched any more. Gates as for the split kernels in test_gpu_parity."""
import numpy as np
import pytest

import oracle as O
import paper_1811_02605_gb300 as P
from paper_1811_02605_gb300 import inputs as I
from tests.gpu_util import dev_state, fields, grid, oracle_iterate_at, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

D = I.GridDesc(23, 17, 46, 1.0, 10.0, 1.07)


def _solve(g, og, b, mixed):
    x = to_dev(np.zeros_like(b))
    prm = P.make_params(tol=1e-11, max_iter=5000, precision=P.PREC_MIXED if mixed else P.PREC_FP64, inner_tol=0.1, max_outer=60)
    st, it, _, rr = P.pcg_solve(g, 4.0, to_dev(b), x, prm)
    xr, itr, _, _ = og.pcg(4.0, b, tol=1e-11, max_iter=5000)
    assert st == P.MHD_OK and rr <= 1e-11
    if mixed:
        assert rel_l2(to_np(x), xr) < 1e-8
    else:
        assert abs(it - itr) <= 1 and rel_l2(to_np(x), oracle_iterate_at(og, 4.0, b, it, itr, xr)) < 1e-11


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("late", [0, 1])
@pytest.mark.parametrize("reserve", [0, 1])
def test_solve_goes_on_with_another_form(monkeypatch, mixed, late, reserve):
    og = O.Grid.from_desc(D)
    b = np.random.default_rng(3).normal(size=(3, D.nr, D.nt, D.np)) * og.volumes()[None, :, :, None]
    g = grid(D)
    if not late:
        monkeypatch.setenv("MHD_FAULT_COOP_LAUNCH", "1")
    if reserve:
        P.mhd_grid_reserve(g, P.RESERVE_MIXED if mixed else P.RESERVE_PC1)
    _solve(g, og, b, mixed)
    form = P.mhd_grid_kernel_forms(g)[mixed]
    persist = -9 if mixed else -3
    assert (form == persist) == bool(late) and form != 0
    monkeypatch.setenv("MHD_FAULT_COOP_LAUNCH", "1")
    _solve(g, og, b, mixed)
    assert P.mhd_grid_kernel_forms(g)[mixed] not in (0, persist)
    monkeypatch.delenv("MHD_FAULT_COOP_LAUNCH")
    _solve(g, og, b, mixed)


def test_step(monkeypatch):
    monkeypatch.setenv("MHD_FAULT_COOP_LAUNCH", "1")
    st = I.initial_state(D, 0, False)
    ds = dev_state(st)
    status, info = P.mhd_step(grid(D), P.make_params(nu=1e-3, cfl=0.4, tol=1e-10), fields(ds))
    assert status == P.MHD_OK
    ref, rinfo = O.Grid.from_desc(D).step(st, nu=1e-3, cfl=0.4, tol=1e-10)
    assert all(abs(a - c) <= 1 for a, c in zip(info["iters"], rinfo["iters"]))
    for k in ref:
        assert rel_l2(to_np(ds[k]), ref[k]) < 1e-10, k
