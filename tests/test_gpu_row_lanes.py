"""The explicit kernels give a row (i, j) to 2 to 32 lanes and cut it into parts, by a rule on its length and the
number of rows; the operator call takes ranges of phi pairs across rows. Results at the grids where either can go wrong
(fewer elements than lanes, one more than a whole number of passes, parts that end inside a pass, ranges that touch many
rows) against the oracle, with the gates of the parity tests; and the time: cells in short, ragged or few long rows take no more
than twice (with the few polar sums of a 4x4x8192 grid, four times) what as many cells in rows of one warp's
width take."""
import pytest
import torch

import paper_1811_02605_gb300 as P
from paper_1811_02605_gb300 import inputs as I
from tests import test_gpu_parity as parity
from tests.gpu_util import grid

pytestmark = pytest.mark.gpu

GRIDS = [I.GridDesc(40, 30, 2, 1.0, 3.0, 1.03), I.GridDesc(33, 21, 6, 1.0, 3.0, 1.04), I.GridDesc(30, 40, 10, 1.0, 3.0, 1.04),
         I.GridDesc(50, 41, 18, 1.0, 4.0, 1.03), I.GridDesc(60, 50, 34, 1.0, 4.0, 1.03), I.GridDesc(41, 37, 66, 1.0, 4.0, 1.03),
         I.GridDesc(2, 3, 1026, 1.0, 2.0, 1.1), I.GridDesc(3, 4, 2050, 1.0, 2.0, 1.1), I.GridDesc(6, 5, 300, 1.0, 3.0, 1.1)]


@pytest.mark.parametrize("d", GRIDS, ids=lambda d: f"{d.nr}x{d.nt}x{d.np}")
def test_results(d):
    parity.test_operator_matches_oracle(d)
    parity.test_coeffs_match_oracle(d)
    parity.test_force_matches_oracle(d)
    for eta in (0.0, 2e-3):
        parity.test_induction_matches_oracle(d, eta)
    parity.test_diagnostics_match_oracle(d)


def _us(nr, nt, np_):
    """Device time of the force, an induction with resistivity and the operator of three components."""
    gen = torch.Generator("cuda").manual_seed(3)

    def field(*shape):
        return 0.01 * torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)
    bt = field(nr, nt + 1, np_)
    bt[:, 0] = bt[:, -1] = 0.0
    f = P.make_fields(field(nr + 1, nt, np_), bt, field(nr, nt, np_), field(nr, nt, np_), field(nr, nt, np_), field(nr, nt, np_))
    g = grid(I.GridDesc(nr, nt, np_, 1.0, 10.0, 1.0 + 1.0 / nr))
    b, vb = field(3, nr, nt, np_), field(3, nr, nt, np_)
    q = torch.empty_like(b)
    times = []
    for call in (lambda: P.mhd_force(g, f, 1e-3, q), lambda: P.mhd_induction(g, vb, 1e-9, 1e-9, f),
                 lambda: P.mhd_apply_operator(g, 1.0, b, q)):
        best = 1e30
        for rep in range(12):
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            call()
            e1.record()
            torch.cuda.synchronize()
            if rep > 1:
                best = min(best, 1e3 * e0.elapsed_time(e1))
        times.append(best)
    return times


@pytest.mark.parametrize("shape,like,factor", [((512, 512, 4), (128, 128, 64), 2.0), ((300, 200, 34), (300, 212, 32), 1.5),
                                               ((16, 16, 4096), (128, 128, 64), 2.0), ((4, 4, 8192), (64, 64, 32), 4.0)])
def test_time(shape, like, factor):
    a, b = _us(*shape), _us(*like)
    assert all(x <= factor * y for x, y in zip(a, b)), (a, b)
