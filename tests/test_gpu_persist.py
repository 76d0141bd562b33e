"""The point-Jacobi PCG whose iterations all run inside one cooperative launch (MHD_FORCE_SLAB=-65 for
the FP64 solve, -9 for the FP32 inner solve), at the sizes where its partition can go wrong: fewer
groups of phi-neighbours than CTAs, chunks that end inside a row, odd row counts, np not a multiple of
4, vectors that fit shared memory and vectors that do not (more than 368 thousand cells in FP64).

It evaluates the same expressions as the split kernels (Sec. 2.2 PCG, PC1) and differs from them only
in the order in which the dot products are summed. Gates: a fixed number of iterations agrees with the
split kernels to 1e-12 relative L2 in FP64 (the gate of the fixed trajectories against the oracle) and
to 1e-6 in FP32 (a few FP32 roundings), and a converged solve with the oracle as in test_gpu_parity."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1811_02605_gb300 as P
from paper_1811_02605_gb300 import inputs as I
from tests.gpu_util import grid, oracle_iterate_at, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

SMALL = [I.GridDesc(2, 2, 2, 1.0, 2.0, 1.1), I.GridDesc(5, 6, 8, 1.0, 3.0, 1.1), I.GridDesc(23, 17, 46, 1.0, 10.0, 1.07),
         I.GridDesc(32, 32, 64, 1.0, 20.0, 1.05)]
LARGE = [I.GridDesc(61, 47, 118, 1.0, 10.0, 1.03), I.GridDesc(65, 63, 130, 1.0, 10.0, 1.02)]


def _name(d):
    return f"{d.nr}x{d.nt}x{d.np}"


def _system(d, seed):
    rng = np.random.default_rng(seed)
    V = O.Grid.from_desc(d).volumes()[None, :, :, None]
    return rng.normal(size=(3, d.nr, d.nt, d.np)) * V, rng.normal(size=(3, d.nr, d.nt, d.np)) * 0.1


@pytest.mark.parametrize("d", SMALL + LARGE, ids=_name)
@pytest.mark.parametrize("k", [1, 2, 25])
def test_fp64_trajectory_equals_split_kernels(monkeypatch, d, k):
    b, x0 = _system(d, 5)
    for nc in (3, 1, 2):
        out = {}
        for form in ("-1", "-65"):
            monkeypatch.setenv("MHD_FORCE_SLAB", form)
            g = grid(d)
            x = to_dev(x0[:nc])
            # a 2x2x2 grid has 8 unknowns a component: CG may meet any tolerance within k iterations
            st, it, _, rr = P.pcg_solve(g, 2.5, to_dev(b[:nc]), x, P.make_params(tol=1e-13, max_iter=k))
            assert st in (P.MHD_OK, P.MHD_ERR_NOCONV)
            out[form] = (to_np(x), it, rr)
            if nc == 3:
                assert P.mhd_grid_kernel_forms(g)[0] == (-3 if form == "-65" else -1)
        assert out["-65"][1] == out["-1"][1]
        assert rel_l2(out["-65"][0], out["-1"][0]) < 1e-12, (nc, rel_l2(out["-65"][0], out["-1"][0]))


@pytest.mark.parametrize("d", SMALL[1:], ids=_name)
def test_fp64_solve_matches_oracle(monkeypatch, d):
    monkeypatch.setenv("MHD_FORCE_SLAB", "-65")
    g, og = grid(d), O.Grid.from_desc(d)
    b, x0 = _system(d, 3)
    for alpha in (0.05, 4.0):
        x = to_dev(x0)
        st, it, _, rr = P.pcg_solve(g, alpha, to_dev(b), x, P.make_params(tol=1e-11, max_iter=5000))
        xr, itr, _, _ = og.pcg(alpha, b, x0=x0, tol=1e-11, max_iter=5000)
        assert st == P.MHD_OK and rr <= 1e-11 and abs(it - itr) <= 1, (it, itr)
        assert rel_l2(to_np(x), oracle_iterate_at(og, alpha, b, it, itr, xr, x0=x0)) < 1e-11, (it, itr)


@pytest.mark.parametrize("d", SMALL[1:] + LARGE + [I.GridDesc(96, 90, 192, 1.0, 10.0, 1.02)], ids=_name)
@pytest.mark.parametrize("restart,inner", [(0, 0.1), (1, 1e-5)])
def test_fp32_inner_solve(monkeypatch, d, restart, inner):
    b, x0 = _system(d, 7)
    out = {}
    for form in ("-2", "-9"):
        monkeypatch.setenv("MHD_FORCE_SLAB", form)
        g = grid(d)
        x = to_dev(x0)
        st, it, ou, _ = P.pcg_solve(g, 3.0, to_dev(b), x, P.make_params(tol=1e-14, inner_tol=1e-12, precision=P.PREC_MIXED,
                                                                       max_outer=1, max_iter=5))
        assert st == P.MHD_ERR_NOCONV and it == 5 and ou == 1
        y = to_dev(x0)
        st, it, ou, rr = P.pcg_solve(g, 3.0, to_dev(b), y, P.make_params(tol=1e-11, inner_tol=inner, precision=P.PREC_MIXED,
                                                                       max_outer=60, max_iter=5000, mixed_restart=restart))
        assert st == P.MHD_OK and rr <= 1e-11
        out[form] = (to_np(x), to_np(y), it, ou)
        assert P.mhd_grid_kernel_forms(g) == (0, int(form))
    assert rel_l2(out["-9"][0], out["-2"][0]) < 1e-6
    # both stop on the true FP64 residual at 1e-11; well conditioned, so the solutions agree far below 1e-6
    assert rel_l2(out["-9"][1], out["-2"][1]) < 1e-8
    assert abs(out["-9"][2] - out["-2"][2]) <= max(2, 0.02 * out["-2"][2])


def test_edge_cases(monkeypatch):
    monkeypatch.setenv("MHD_FORCE_SLAB", "-65")
    d = SMALL[1]
    g = grid(d)
    z = torch.zeros((3, d.nr, d.nt, d.np), dtype=torch.float64, device="cuda")
    x = torch.ones_like(z)
    assert P.pcg_solve(g, 1.0, z, x, P.make_params())[:2] == (P.MHD_OK, 0) and torch.all(x == 0)
    b = torch.randn(z.shape, dtype=torch.float64, device="cuda")
    x = torch.zeros_like(b)
    assert P.pcg_solve(g, 0.0, b, x, P.make_params(tol=1e-12))[:2] == (P.MHD_OK, 1)
    x.zero_()
    assert P.pcg_solve(g, 1.0, b, x, P.make_params(tol=1e-14, max_iter=0))[:2] == (P.MHD_ERR_NOCONV, 0)
    b[0, 0, 0, 0] = float("nan")
    x.zero_()
    assert P.pcg_solve(g, 1.0, b, x, P.make_params())[0] == P.MHD_ERR_NONFINITE


@pytest.mark.parametrize("mixed", [0, 1])
def test_wait_that_runs_out_returns_a_status(monkeypatch, mixed):
    # the exchange waits for one arrival that never comes, with a short limit; the context stays usable
    d = SMALL[2]
    b, _ = _system(d, 9)
    monkeypatch.setenv("MHD_FORCE_SLAB", "-9" if mixed else "-65")
    g = grid(d)
    prm = P.make_params(tol=1e-9, precision=mixed, inner_tol=0.1)
    x = torch.zeros(b.shape, dtype=torch.float64, device="cuda")
    monkeypatch.setenv("MHD_FAULT_BARRIER_MS", "100")
    with pytest.raises(P.MhdError) as e:
        P.pcg_solve(g, 1.0, to_dev(b), x, prm)
    assert e.value.status == P.MHD_ERR_TIMEOUT
    monkeypatch.delenv("MHD_FAULT_BARRIER_MS")
    x.zero_()
    assert P.pcg_solve(g, 1.0, to_dev(b), x, prm)[0] == P.MHD_OK
