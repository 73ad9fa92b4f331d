"""Diagnostics of rows on either side of the size that picks the kernel (160
points), of rows shorter than a warp and longer than a block, against the FP64
oracle, for every gravity axis.  Bounds: sums 1e-13 relative, speed and Mach
number 1e-12 relative (test_diagnostics_match_oracle); the disturbance pressure,
a difference of values near (gamma - 1) E, 16 ulps of the largest of these."""
import numpy as np
import pytest

import nopcs_synth as S
import oracle
from gpu_util import binding, stream_ptr, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,ga", [((5, 61, 43), 2), ((31, 47, 60), 1), ((32, 40, 41), 0), ((160, 19, 22), 0),
                                  ((161, 19, 22), 0), ((161, 20, 61), 2), ((257, 13, 100), 1), ((700, 5, 6), 2)])
def test_diagnostics_of_row_lengths(n, ga, prec):
    N = binding()
    p = S.box_params(n, sub_n=(0, 0, 0), perturb_amp=1e-3, gravity_axis=ga, base_subtract=prec)
    orc = oracle.Solver(p)
    Q = orc.initial_state()
    rng = np.random.default_rng(7)
    Q[0] *= 1 + 1e-4 * rng.standard_normal(Q[0].shape)
    Q[4] *= 1 + 1e-4 * rng.standard_normal(Q[4].shape)
    ctx = N.nopcs_init([p], prec=prec, stream=stream_ptr())
    try:
        N.nopcs_set_state(ctx, 0, to_dev(Q).data_ptr())
        d = N.nopcs_diagnostics(ctx, 0)
        assert N.nopcs_diagnostics(ctx, 0) == d
    finally:
        N.nopcs_destroy(ctx)
    r = orc.diagnostics(Q)
    for k in ("mass", "energy_total"):
        assert abs(d[k] - r[k]) <= 1e-13 * abs(r[k]), (k, d[k], r[k])
    for k in ("max_speed", "max_mach"):
        assert abs(d[k] - r[k]) <= 1e-12 * abs(r[k]), (k, d[k], r[k])
    ulp = np.finfo(float).eps * (p["gamma"] - 1) * np.abs(Q[4]).max()
    assert abs(d["max_dp"] - r["max_dp"]) <= 16 * ulp, (d["max_dp"], r["max_dp"])
