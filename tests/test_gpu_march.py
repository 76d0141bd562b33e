"""The FP32 single-reduction iteration as one plane-marching kernel (MHD_FORCE_SLAB=-10), at the sizes
where its tiling can go wrong: fewer phi groups or theta rows than a tile, tiles that end inside the
grid, one phi group (every phi neighbour is the cell's own group), two planes, more columns than
resident CTAs (whole columns first, the rest in slabs), one to three components.

It evaluates the expressions of the single-reduction pair (Sec. 2.2 PCG, PC1) and differs from it in the
order of the sums. Gates as for the other single-reduction forms: after k inner iterations within
1e-5 of the folded form (it forms alpha from another expression, so a few FP32 roundings per step), and
a solve that meets the FP64 tolerance on the true residual within 1e-6 of the oracle's solution."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1811_02605_gb300 as P
from paper_1811_02605_gb300 import inputs as I
from tests.gpu_util import grid, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

GRIDS = [I.GridDesc(2, 2, 8, 1.0, 2.0, 1.1), I.GridDesc(5, 6, 4, 1.0, 3.0, 1.1), I.GridDesc(12, 17, 72, 1.0, 5.0, 1.06),
         I.GridDesc(7, 35, 132, 1.0, 4.0, 1.06), I.GridDesc(40, 16, 64, 1.0, 10.0, 1.04)]


def _name(d):
    return f"{d.nr}x{d.nt}x{d.np}"


def _solve(monkeypatch, form, d, b, x0, **kw):
    monkeypatch.setenv("MHD_FORCE_SLAB", form)
    g = grid(d)
    x = to_dev(x0)
    st, it, ou, rr = P.pcg_solve(g, 3.0, to_dev(b), x, P.make_params(precision=P.PREC_MIXED, **kw))
    assert P.mhd_grid_kernel_forms(g) == (0, int(form))
    return st, it, ou, rr, to_np(x)


def _system(d, seed):
    rng = np.random.default_rng(seed)
    og = O.Grid.from_desc(d)
    return og, rng.normal(size=(3, d.nr, d.nt, d.np)) * og.volumes()[None, :, :, None], rng.normal(size=(3, d.nr, d.nt, d.np)) * 0.1


@pytest.mark.parametrize("d", GRIDS + [I.GridDesc(6, 130, 1024, 1.0, 2.0, 1.05)], ids=_name)
@pytest.mark.parametrize("k", [1, 2, 7])
def test_trajectory(monkeypatch, d, k):
    # k odd leaves an x update pending at the correction, k even does not
    _, b, x0 = _system(d, 51)
    for nc in (3, 1, 2):
        out = {}
        for form in ("-2", "-10"):
            st, it, ou, _, x = _solve(monkeypatch, form, d, b[:nc], x0[:nc], tol=1e-14, inner_tol=1e-12, max_outer=1, max_iter=k)
            out[form] = (it, x)
        assert out["-10"][0] == out["-2"][0]
        assert rel_l2(out["-10"][1], out["-2"][1]) < 1e-5, (nc, rel_l2(out["-10"][1], out["-2"][1]))


@pytest.mark.parametrize("d", GRIDS, ids=_name)
@pytest.mark.parametrize("restart,inner", [(0, 0.1), (1, 1e-5)])
def test_solve(monkeypatch, d, restart, inner):
    og, b, x0 = _system(d, 52)
    kw = dict(tol=1e-9, inner_tol=inner, mixed_restart=restart, max_outer=60, max_iter=5000)
    st, it, ou, rr, x = _solve(monkeypatch, "-10", d, b, x0, **kw)
    st7, it7, ou7, _, _ = _solve(monkeypatch, "-7", d, b, x0, **kw)
    assert st == P.MHD_OK and rr <= 1e-9
    assert np.linalg.norm(b - og.apply_M(3.0, x)) <= 1e-9 * np.linalg.norm(b) * 1.0000001
    xr = og.pcg(3.0, b, x0=x0, tol=1e-13)[0]
    assert rel_l2(x, xr) < 1e-6
    assert st7 == P.MHD_OK and abs(it - it7) <= max(2, 0.05 * it7), (it, it7)
