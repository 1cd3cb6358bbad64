"""The reverse sweep's chi2 and d chi2 / d p0 keep their bits, whichever kernels its passes run in.

A track whose covariance is nearly singular turns the last bit of one step into 1e-5 to 1e-3 of its
derivative, which no comparison with FP64 can tell from the FP32 rounding that is there anyway: the
values recorded in golden/fit_derivative.npz are compared for equality.  (They hold for the CUDA 13.0
compiler: another one may round a step otherwise.)"""
import os

import numpy as np
import pytest

from paper_2312_11728_gb300 import build as B
from paper_2312_11728_gb300 import mkgb, pipeline, synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group, geometry", [("endcap", S.geometry_phase2), ("modular", S.geometry_phase2_modular_disks)])
def test_derivative_keeps_its_bits(group, geometry):
    B.build()
    mkgb.load_library()
    with np.load(os.path.join(os.path.dirname(__file__), "golden", "fit_derivative.npz")) as f:
        d = {k[len(group) + 1:]: f[k] for k in f.files if k.startswith(group + "_")}
    ctx = pipeline.make_context(geometry(), S.default_params())
    ctx.load_hits(1, d["off"], d["xyz"], d["cov"], hit_module=d.get("mod"))
    n, L = d["layers"].shape[0], d["xscale"].shape[0]
    f32 = lambda *s: np.zeros(s, np.float32)
    chi2, dp0, dal, dxs, status = f32(n), f32(n, 6), f32(L, 6), f32(L), np.zeros(n, np.int32)
    ctx.fit_grad(d["layers"].astype(np.int32), d["hits"].astype(np.int32), d["p0"], d["c0"], d["align"], d["xscale"],
                 chi2, dp0, dal, dxs, status)
    assert not status.any()
    np.testing.assert_array_equal(chi2, d["chi2"])
    np.testing.assert_array_equal(dp0, d["dp0"])
