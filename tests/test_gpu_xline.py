"""FP64 flux sweep along long x lines on either side of the rule that picks
sub-domain tiles or whole lines (columns per 32-lane warp, sub-domain length),
against the FP64 oracle, with the gate of test_rhs_matches_oracle: 1e-12 of the
field's maximum, for the momentum plus 30 ulps of the pressure-gradient terms."""
import numpy as np
import pytest

import nopcs_synth as S
import oracle
from gpu_util import binding, stream_ptr, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,sub", [(640, 64), (768, 64), (767, 64), (832, 64), (416, 32), (384, 32), (512, 32)])
@pytest.mark.parametrize("ga", [0, 2])
def test_rhs_of_long_lines(nx, sub, ga):
    import torch
    N = binding()
    p = S.box_params((nx, 9, 11), sub_n=(sub, 0, 0), gravity_axis=ga, perturb_amp=1e-3, seed=9)
    orc = oracle.Solver(p)
    Q = orc.initial_state()
    rng = np.random.default_rng(1)
    Q[4] *= 1 + 1e-4 * rng.standard_normal(Q[4].shape)
    Q[0] *= 1 + 1e-4 * rng.standard_normal(Q[0].shape)
    ref = orc.rhs(Q)
    ref[1:4][:, [0, -1]] = 0
    ref[1:4][:, :, [0, -1]] = 0
    ref[1:4][:, :, :, [0, -1]] = 0
    ctx = N.nopcs_init([p], prec=N.NOPCS_FP64, stream=stream_ptr())
    try:
        r = torch.empty(Q.shape, dtype=torch.float64, device="cuda")
        N.nopcs_rhs(ctx, 0, to_dev(Q).data_ptr(), r.data_ptr())
        got = r.cpu().numpy()
        pr = (p["gamma"] - 1) * (Q[4] - 0.5 * (Q[1] ** 2 + Q[2] ** 2 + Q[3] ** 2) / Q[0])
        h = min(p["len"][a] / (p["n"][a] - 1) for a in range(3))
        floor = 30 * np.finfo(float).eps * np.abs(pr).max() / h
        d = np.abs(got - ref).reshape(5, -1).max(axis=1)
        s_ = np.abs(ref).reshape(5, -1).max(axis=1)
        assert np.all(d[[0, 4]] <= 1e-12 * s_[[0, 4]]), (d, s_)
        assert np.all(d[1:4] <= 1e-12 * s_[1:4] + floor), (d, s_, floor)
    finally:
        N.nopcs_destroy(ctx)
