"""The stop norm of the marching kernel (MHD_FORCE_SLAB=-10), sum dg r~^2: its weights dg, scaled by a power
of two, stay below 1, so a product with r~^2 overflows no earlier than r~^2 itself. The solve is then
scale-invariant: a right-hand side times a power of two gives the same iterations and that multiple of the
solution, bit for bit, up to residuals whose square is near the largest float. The grid's diagonals spread
over a factor of 500, and the residual sits where they are largest; the pair it replaces (-7) sums in FP64
and is the same test's control."""
import numpy as np
import pytest

import oracle as O
import paper_1811_02605_gb300 as P
from paper_1811_02605_gb300 import inputs as I
from tests.gpu_util import grid, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

D = I.GridDesc(24, 8, 16, 1.0, 20.0, 1.4)


@pytest.mark.parametrize("form", ["-7", "-10"])
def test_solve_is_invariant_under_powers_of_two(monkeypatch, form):
    monkeypatch.setenv("MHD_FORCE_SLAB", form)
    og = O.Grid.from_desc(D)
    # the diagonal by rows, from the operator on unit vectors
    dg = np.zeros((D.nr, D.nt))
    for i in range(D.nr):
        for j in range(D.nt):
            e = np.zeros((1, D.nr, D.nt, D.np))
            e[0, i, j, 0] = 1.0
            dg[i, j] = og.apply_M(1.0, e)[0, i, j, 0]
    hot = dg > dg.max() / 4
    assert dg.max() / dg[-1, D.nt // 2] > 150
    b = np.zeros((1, D.nr, D.nt, D.np))
    b[0][hot] = np.random.default_rng(0).uniform(0.7, 1.4, size=(hot.sum(), D.np)) * np.sqrt(dg[hot])[:, None]
    out = {}
    for e in (0, -20, 60):   # 2^60: r~^2 about 1e36
        x = to_dev(np.zeros_like(b))
        st, it, ou, rr = P.pcg_solve(grid(D), 1.0, to_dev(np.ldexp(b, e)), x,
                                     P.make_params(precision=P.PREC_MIXED, tol=1e-9, inner_tol=0.1, max_outer=60, max_iter=5000))
        assert st == P.MHD_OK, (e, st)
        out[e] = (it, ou, rr, np.ldexp(to_np(x), -e))
    assert rel_l2(out[0][3], og.pcg(1.0, b, tol=1e-12)[0]) < 1e-6
    for e in (-20, 60):
        assert out[e][:3] == out[0][:3]
        assert np.array_equal(out[e][3], out[0][3])
