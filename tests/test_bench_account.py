"""bench.py's accounting of a profiled run over the kernel forms a grid may have chosen: every form has a
bandwidth that the part can have (no more than its HBM, or for the flops its FP64 pipe), a form that is
one launch a solve is not divided by launches that it does not make, and no form is left out. On a GPU,
the whole bench line of a grid whose solves take the persistent kernel."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
import paper_1811_02605_gb300 as P  # noqa: E402

HBM = 6790.7
BIG = 256 * 256 * 512


def _prof(**kw):
    return {k: kw.get(k, (0.0, 0)) for k in P.KERNELS}


@pytest.mark.parametrize("prof,ms_iter,name", [
    # 1000 inner iterations in 10 inner solves
    (_prof(march32=(374.0, 1040), cgr32=(1.3, 10)), 0.3753, "one plane-marching kernel"),
    (_prof(cgr32=(120.0, 1040), cgu32=(420.0, 1040)), 0.540, "single-reduction pair"),
    (_prof(pfold32=(200.0, 1040), rupd32=(400.0, 1040)), 0.600, "recompute pair"),
    (_prof(pspmv32=(420.0, 1040), update32=(200.0, 1040)), 0.620, "p update folded"),
    (_prof(pupdate32=(300.0, 1040), spmv32=(180.0, 1040), update32=(190.0, 1040)), 0.670, "split"),
    (_prof(spmv32=(500.0, 1040), update32=(520.0, 1040)), 1.02, "plane-marching pair"),
], ids=["march", "single-reduction", "recompute", "folded", "split", "tiled"])
def test_fp32_forms_of_a_large_grid(prof, ms_iter, name):
    gbs, kernels, form = bench.pcg32_account(prof, 1000, BIG, HBM)
    assert abs(gbs - 72 * BIG / (ms_iter * 1e-3) / 1e9) < 1e-6 * gbs
    assert form.startswith(name)
    assert set(kernels) == {k for k, v in prof.items() if v[1]}
    assert all(0.0 < v["frac_of_hbm"] < 1.0 for v in kernels.values()), kernels


def test_fp32_persistent_form_of_a_small_grid():
    N = 48 * 48 * 96
    gbs, kernels, form = bench.pcg32_account(_prof(persist32=(11.8, 10)), 1000, N, HBM)
    assert abs(gbs - 72 * N / 11.8e-6 / 1e9) < 1e-6 * gbs and gbs < HBM
    assert form.startswith("one persistent launch") and set(kernels) == {"persist32"}
    assert kernels["persist32"]["avg_launch_ms"] == 1.18 and kernels["persist32"]["ms_per_iteration"] == 0.0118


@pytest.mark.parametrize("form,prof,N,ms_iter", [
    (-3, _prof(persist64=(39.3, 9)), 32 * 32 * 64, 0.0131),
    (-1, _prof(pupdate64=(1860.0, 3060), spmv64=(3750.0, 3060), update64=(1260.0, 3060)), BIG, 2.29),
    (-2, _prof(pupdate64=(2900.0, 9180), spmv64=(4140.0, 9180), update64=(1260.0, 3060)), BIG, 2.12),
    (16, _prof(spmv64=(5000.0, 3060), update64=(1200.0, 3060)), BIG, 2.07),
], ids=["persistent", "split", "overlapped", "tiled"])
def test_fp64_forms(form, prof, N, ms_iter):
    ms, gbs, kernels, roof = bench.pcg64_account(prof, 3000, N, HBM, form, ms_iter, 200)
    assert abs(ms - sum(v[0] for v in prof.values())) < 1e-9 and ms > 0
    assert 0.0 < gbs < HBM and set(kernels) == {k for k, v in prof.items() if v[1]}
    assert 0.0 < roof["frac"] <= 1.0 and 0.0 < roof["iteration"]["fp64_pipe_frac"] <= 1.0, roof
    assert ("k_persist" in roof["kernel"]) == (form == -3)


@pytest.mark.gpu
def test_bench_line_where_solves_are_persistent():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--grid", "16x16x32", "--steps", "1", "--warmup",
                          "3", "--no-cpu-baseline", "--no-sts", "--no-res"], capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert out.returncode == 0, out.stderr[-2000:]
    line = json.loads(out.stdout.strip().splitlines()[-1])
    assert "persist64" in line["pcg_gbs"]["kernels"] and 0.0 < line["roofline"]["frac"] < 1.0
    for entry in (line["mixed"], line["mixed_reliable"]):
        assert "persist32" in entry["kernels"] and 0.0 < entry["pcg_frac_of_hbm"] < 1.0
    assert line["gpu_launches"] > 0 and line["value"] > 0
