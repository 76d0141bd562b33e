"""The explicit kernels and the operator call hand rows (i, j) to warps: the grids where that can go wrong (rows shorter
than a warp, just over one and over several, a last element alone, three rows per shell with both polar rules, row
counts that are not a multiple of a CTA's) against the oracle (Sec. 2.1, 2.2), with the gates of the parity tests."""
import pytest

from paper_1811_02605_gb300 import inputs as I
from tests import test_gpu_parity as parity

pytestmark = pytest.mark.gpu

GRIDS = [I.GridDesc(2, 3, 4, 1.0, 2.0, 1.1), I.GridDesc(3, 3, 34, 1.0, 3.0, 1.1), I.GridDesc(5, 3, 62, 1.0, 3.0, 1.1),
         I.GridDesc(2, 9, 96, 1.0, 4.0, 1.1), I.GridDesc(7, 5, 130, 1.0, 5.0, 1.06)]


@pytest.mark.parametrize("d", GRIDS, ids=lambda d: f"{d.nr}x{d.nt}x{d.np}")
def test_rows(d):
    parity.test_operator_matches_oracle(d)
    parity.test_coeffs_match_oracle(d)
    parity.test_force_matches_oracle(d)
    for eta in (0.0, 2e-3):
        parity.test_induction_matches_oracle(d, eta)
    parity.test_diagnostics_match_oracle(d)
