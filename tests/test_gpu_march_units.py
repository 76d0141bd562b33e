"""The marching kernel (MHD_FORCE_SLAB=-10) where a CTA marches more than one unit of work after another, in
the same shared memory: units that are slabs of a column with an odd and with an even number of steps, and
whole columns first with the rest in slabs. A mirror of the host's tiling rule says which shape a grid takes,
so that the cases cannot stop covering these. Gates as for the kernel's other trajectories
(test_gpu_march.py): within 1e-5 of the folded form after k iterations."""
import numpy as np
import pytest
import torch

import paper_1811_02605_gb300 as P
from paper_1811_02605_gb300 import inputs as I
from tests.gpu_util import grid, rel_l2, to_dev, to_np

ROWS, GROUPS, CTAS = 20, 14, 3   # most theta rows and phi groups a CTA writes, CTAs per SM


def tiling(nr, nt, np_, nc, sms=152):
    """(cost, columns, whole columns, slabs, units, planes of a slab) as the launch chooses them."""
    npg, ctas, best = np_ // 4, CTAS * sms, None
    nj0, nk0 = -(-nt // ROWS), -(-npg // GROUPS)
    for nk in range(nk0, nk0 + 4):
        for nj in range(nj0, nj0 + 4):
            tg = min(GROUPS, (-(-npg // nk) + 1) & ~1)
            tj = -(-nt // nj)
            cols = nc * -(-nt // tj) * -(-npg // tg)
            whole = cols // ctas * ctas
            for s in range(1, min(nr, 64) + 1):
                for full in {0, whole if whole < cols else 0}:
                    rest = cols - full
                    plen = -(-nr // s)
                    slabs = -(-nr // plen)
                    rounds = -(-rest * slabs // ctas)
                    cost = 2 * (full // ctas * (nr + 6) + rounds * (plen + 6)) + (tg % 4 != 0)
                    if best is None or cost < best[0]:
                        best = (cost, cols, full, slabs, full + rest * slabs, -(-nr // slabs))
    return best


# grid, whole columns first, steps of a slab (planes + 4) odd
CASES = [(I.GridDesc(24, 160, 512, 1.0, 3.0, 1.03), False, 0), (I.GridDesc(21, 160, 512, 1.0, 3.0, 1.03), False, 1),
         (I.GridDesc(9, 180, 1024, 1.0, 2.0, 1.05), True, 0), (I.GridDesc(6, 130, 1400, 1.0, 2.0, 1.05), True, 1)]


def test_cases_cover_the_shapes():
    for d, whole, odd in CASES:
        _, cols, full, slabs, units, plen = tiling(d.nr, d.nt, d.np, 3)
        assert units > CTAS * 152, (d, units)
        assert (0 < full < cols) == whole and (plen + 4) % 2 == odd, (d, full, plen)


@pytest.mark.gpu
@pytest.mark.parametrize("d", [c[0] for c in CASES], ids=lambda d: f"{d.nr}x{d.nt}x{d.np}")
@pytest.mark.parametrize("k", [1, 6])
def test_trajectory(monkeypatch, d, k):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("shapes for 152 SMs")
    rng = np.random.default_rng(17)
    b, x0 = to_dev(rng.normal(size=(3, d.nr, d.nt, d.np))), rng.normal(size=(3, d.nr, d.nt, d.np))
    out = {}
    for form in ("-2", "-10"):
        monkeypatch.setenv("MHD_FORCE_SLAB", form)
        g, x = grid(d), to_dev(x0)
        st, it, _, _ = P.pcg_solve(g, 3.0, b, x, P.make_params(precision=P.PREC_MIXED, tol=1e-14, inner_tol=1e-12, max_outer=1,
                                                               max_iter=k))
        assert st == P.MHD_ERR_NOCONV and it == k and P.mhd_grid_kernel_forms(g) == (0, int(form))
        out[form] = to_np(x)
    assert rel_l2(out["-10"], out["-2"]) < 1e-5
