"""Host-side arithmetic of bench.py (CPU): the energy-norm weights the
benchmark uses to state the FP32 error equal -diag(M) of the oracle."""
import os

import numpy as np

import bench
import oracle as ora
from paper_2509_19061_gb300 import inputs


def test_energy_weights_are_minus_diag_m():
    for nx, ny, lx, ly in ((37, 23, 1.3, 0.9), (16, 16, 1.0, 1.0), (5, 9, 0.5, 2.0)):
        prob = inputs.sinker_problem(nx, ny, eta_in=1e3, lx=lx, ly=ly)
        prob.eta_c, prob.eta_n = inputs.random_viscosity(nx, ny, nx + ny, (-2.0, 2.0))
        wx, wy = bench.energy_weights(prob)
        dx, dy = ora.diag_M(ora.Grid(nx, ny, prob.hx, prob.hy, prob.eta_c, prob.eta_n))
        assert wx.shape == dx.shape and wy.shape == dy.shape
        assert np.allclose(wx, -dx, rtol=1e-14, atol=0.0)
        assert np.allclose(wy, -dy, rtol=1e-14, atol=0.0)


def test_the_named_kernel_is_the_one_that_runs():
    """The kernel a benchmark row names is what the library's plan says, over
    sizes, precisions, variants and sweep counts, and its profile is tied to that
    kernel's own sources."""
    from paper_2509_19061_gb300 import api, build
    build.build()

    def name(n, dt, **kw):
        return bench.sweep_kernel_name(api, n, dt, max_cluster=16, **kw)

    exact = dict(variant="ras", tile=(32, 32), k=4, overlap=3)
    assert name(8192, "f32", sweeps=100, **exact) == "k_ras_stream"
    assert name(1024, "f64", sweeps=100, **exact) == "k_stream64"
    assert name(64, "f64", sweeps=10, **exact) == name(128, "f32", sweeps=10, **exact) == "k_jacobi_cluster"
    assert name(2000, "f32", variant="rbgs", sweeps=20) == "k_rbgs_stream"
    assert name(2000, "f64", variant="rbgs", sweeps=20) is None
    for kernel, paths in bench.KERNEL_SOURCES.items():
        text = "".join(open(os.path.join(bench.ROOT, p)).read() for p in paths)
        assert kernel + "(" in text, kernel


def test_the_printed_line_is_short():
    """The line keeps every figure of the run itself; the extra legs' tables stay
    out of it, so that it fits the last few KB of the output."""
    import json
    run = dict(metric="m", value=1110.123456789012, unit="u", n_gpus=1, steps=20, warmup=5, ms_per_step=6.123456789,
               higher_is_better=True, scaling="weak", vs_baseline=None, dtype="f32", data="synthetic",
               config={"workload": "w" * 60, "tile": [48, 64], "step": "s" * 60, "l2": "l" * 80}, gpu_launches=1,
               clocks={"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}, step_ms={"median": 6.1, "ci95": [6, 7]},
               energy_residual_after_step=0.5, e2e={"value": 700.0, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2})
    line = dict(run, roofline=dict({k: 1.0 for k in bench.ROOFLINE}, traffic_note="n" * 300))
    line.update({k: {"row %d" % i: {"ms_per_call": 1.0} for i in range(60)} for k in bench.TABLES})
    line["time_to_1e-8"].update(workload="w", f32_inner={"seconds": 0.05}, f64_inner={"seconds": 0.4})
    line["cpu_baseline"].update(value=0.02, unit="u", cores=1, kind="oracle")
    out = bench.short_line(line, "tables.json")
    assert all(out[k] == v for k, v in run.items())
    assert out["roofline"] == {k: 1.0 for k in bench.ROOFLINE}
    assert out["time_to_1e-8"]["f32_inner"] == 0.05 and out["cpu_baseline"]["value"] == 0.02
    assert len(json.dumps(line)) > 20000 and len(json.dumps(out)) < 2500
