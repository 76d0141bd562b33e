"""The timed choice of the kernel forms (the first solve's, or mhd_grid_reserve's): the form it takes is
one that a real solve finds fast, whatever the alpha of the first solve. Above the sizes that fit the
CTAs' shared memory the persistent and the marching form compete; a trial that ends early (a breakdown
of inconsistent CG scalars, convergence at alpha = 0) must not count as a fast one.

Gate: an inner solve of 60 iterations with the chosen form takes at most 1.15 times what it takes with
the fastest of the candidates, each forced in turn (MHD_FORCE_SLAB). The forms are 30% apart or more at
these sizes, and repeated times differ by a few per cent."""
import numpy as np
import pytest
import torch

import paper_1811_02605_gb300 as P
from paper_1811_02605_gb300 import inputs as I
from tests.gpu_util import grid, to_dev

pytestmark = pytest.mark.gpu

FORMS32 = ("-9", "-10", "-7", "-4", "-2")
FORMS64 = ("-65", "-1", "-64")
CODE64 = {"-65": -3, "-1": -1, "-64": -2}


def _ms(d, b, mixed):
    g = grid(d)
    prm = (P.make_params(tol=1e-30, inner_tol=1e-30, precision=P.PREC_MIXED, max_outer=1, max_iter=60) if mixed
           else P.make_params(tol=1e-30, max_iter=60))
    best = 1e30
    for rep in range(6):
        x = torch.zeros_like(b)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        st, it, _, _ = P.pcg_solve(g, 50.0, b, x, prm)
        e1.record()
        torch.cuda.synchronize()
        assert st == P.MHD_ERR_NOCONV and it == 60
        if rep:
            best = min(best, e0.elapsed_time(e1))
    return best


def _rhs(d):
    return to_dev(np.random.default_rng(4).normal(size=(3, d.nr, d.nt, d.np)))


@pytest.mark.parametrize("first", ["reserve", "alpha 0", "alpha 50"])
@pytest.mark.parametrize("d,mixed", [(I.GridDesc(100, 100, 104, 1.0, 10.0, 1.02), 1), (I.GridDesc(96, 96, 192, 1.0, 10.0, 1.02), 1),
                                     (I.GridDesc(80, 80, 82, 1.0, 10.0, 1.02), 0)],
                         ids=["100x100x104 mixed", "96x96x192 mixed", "80x80x82 fp64"])
def test_chosen_form_is_near_the_fastest(monkeypatch, d, mixed, first):
    b = _rhs(d)
    ms = {}
    for form in FORMS32 if mixed else FORMS64:
        monkeypatch.setenv("MHD_FORCE_SLAB", form)
        ms[int(form) if mixed else CODE64[form]] = _ms(d, b, mixed)
    monkeypatch.delenv("MHD_FORCE_SLAB")
    g = grid(d)
    if first == "reserve":
        P.mhd_grid_reserve(g, P.RESERVE_MIXED if mixed else P.RESERVE_PC1)
    else:
        prm = P.make_params(tol=1e-9, inner_tol=0.1, precision=P.PREC_MIXED if mixed else P.PREC_FP64, max_outer=60)
        assert P.pcg_solve(g, float(first.split()[1]), b, torch.zeros_like(b), prm)[0] == P.MHD_OK
    form = P.mhd_grid_kernel_forms(g)[1 if mixed else 0]
    assert ms[form] <= 1.15 * min(ms.values()), (form, ms)


@pytest.mark.parametrize("d,mixed", [(I.GridDesc(45, 61, 128, 1.0, 10.0, 1.02), 0), (I.GridDesc(78, 70, 128, 1.0, 10.0, 1.02), 1)],
                         ids=["45x61x128 fp64", "78x70x128 mixed"])
def test_persistent_form_by_rule_up_to_shared_memory(d, mixed):
    # the largest grids with np = 128, but a row or two, whose vectors fit 152 CTAs with 220 KB of shared memory
    # each (351,360 cells in FP64, 701,952 in FP32)
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("sizes for 152 SMs")
    g = grid(d)
    P.mhd_grid_reserve(g, P.RESERVE_MIXED if mixed else P.RESERVE_PC1)
    assert P.mhd_grid_kernel_forms(g)[1 if mixed else 0] == (-9 if mixed else -3)
