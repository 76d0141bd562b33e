"""PC2's line kernel (Sec. 2.2 block-Jacobi ILU(0), phi lines) at the line lengths where its split into lanes and segments
can go wrong: one segment, lengths on and beside the borders between the lane counts and segment lengths, lengths that
are not a multiple of four (8-byte copies in FP32), a number of lines that does not fill the last warp, and the
first length beyond the register kernel. FP64 iterates after a fixed number of iterations against the oracle's, gate
1e-12 as for the other line lengths; mixed solves on the true residual."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1811_02605_gb300 as P
from paper_1811_02605_gb300 import inputs as I
from tests.gpu_util import grid, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

LENGTHS = [2, 4, 30, 32, 34, 64, 96, 98, 126, 128, 130, 190, 192, 256, 258, 382, 384, 510, 514, 640, 642, 768, 770]


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("nr,nt", [(3, 5), (2, 2)])
def test_line_lengths(n, nr, nt):
    d = I.GridDesc(nr, nt, n, 1.0, 2.0, 1.1)
    g, og = grid(d), O.Grid.from_desc(d)
    b = np.random.default_rng(n).normal(size=(3, nr, nt, n)) * og.volumes()[None, :, :, None]
    for nc, k in ((3, 3), (2, 1), (1, 4)):
        x = torch.zeros((nc, nr, nt, n), dtype=torch.float64, device="cuda")
        st, it, _, _ = P.pcg_solve(g, 0.5, to_dev(b[:nc]), x, P.make_params(tol=1e-30, max_iter=k, preconditioner=1))
        assert st == P.MHD_ERR_NOCONV and it == k
        xr, _, _, _ = og.pcg(0.5, b[:nc], fixed_iters=k, pc2="lines")
        assert rel_l2(to_np(x), xr) < 1e-12, (nc, k)
    for restart, inner in ((0, 0.1), (1, 1e-4)):
        x = torch.zeros((3, nr, nt, n), dtype=torch.float64, device="cuda")
        prm = P.make_params(tol=1e-10, precision=P.PREC_MIXED, inner_tol=inner, mixed_restart=restart, max_outer=60, preconditioner=1)
        st, _, _, _ = P.pcg_solve(g, 0.5, to_dev(b), x, prm)
        assert st == P.MHD_OK
        assert np.linalg.norm(b - og.apply_M(0.5, to_np(x))) <= 1e-10 * np.linalg.norm(b) * 1.0000001
